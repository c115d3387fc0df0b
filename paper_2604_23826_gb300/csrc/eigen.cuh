// eigen.cuh -- symmetric eigen-decomposition pieces shared by the one-block solvers of the finalize
// kernels and the grid-wide solver: cyclic Jacobi with the parallel round-robin ordering (Brent and
// Luk), in FP64 and in FP32.
//
// GB300 runs FP64 at 2 operations per clock and SM: 64 cycles for any FP64 warp instruction,
// ~570 for a division or a square root.  So the FP64 rotations take their angle from FP32 (t to
// ~20 bits; the rotation itself is orthonormal to FP64 rounding, it only misses the exact zero by
// 2^-20 of the entry, which the next sweep removes), and everything that can be exact without the
// FP64 unit -- exponents, comparisons, conversions -- runs on the integer pipe.
#pragma once

#include <utility>

#include "common.cuh"

namespace ss {
namespace eig {

// Pair i of round r on the even order m: pair 0 is (r, m - 1), pair i > 0 ((r + i) mod (m - 1),
// (r - i) mod (m - 1)).  Every index occurs in exactly one pair of a round, so a round's rotations
// commute and act on independent 2 x 2 blocks.
__device__ __forceinline__ void pair_of(int r, int i, int m, int& p, int& q) {
  p = r + i;
  q = r - i;
  if (p >= m - 1) p -= m - 1;
  if (q < 0) q += m - 1;
  if (i == 0) q = m - 1;
}

__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }

// x * 2^-(E - 1023) to 23 bits, 0 below 2^-126 (E >= x's exponent field)
__device__ __forceinline__ float scaled32(double x, int E) {
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)), lo = static_cast<uint32_t>(__double2loint(x));
  const int ef = static_cast<int>((hi >> 20) & 0x7FFu), e = ef - E + 127;
  return ef > 0 && e > 0 ? __uint_as_float((hi & 0x80000000u) | (static_cast<uint32_t>(e) << 23) |
                                           ((hi & 0xFFFFFu) << 3) | (lo >> 29))
                         : 0.f;
}

__device__ __forceinline__ float rsqrt32(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// tan of the Jacobi angle, |t| <= 1, of [[p, a], [a, q]] with d = q - p (a not zero, of a magnitude
// whose square FP32 holds, or d is)
__device__ __forceinline__ float tan32(float d, float a) {
  const float x = fmaf(d, d, 4.f * a * a);
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fmaf(x, rsqrt32(x), fabsf(d))));
  return (d >= 0.f ? 2.f * a : -2.f * a) * r;
}

// The rotation (c, s) that (nearly) annihilates apq, orthonormal to FP64 rounding.  null: what is
// left of apq lies below 2^-56 of sqrt(|app aqq|) and may be set to zero, as the classical
// rotation sets it (without it, equal eigenvalues would keep rounding noise there).
__device__ __forceinline__ void rotation64(double app, double aqq, double apq, double& c, double& s, bool& null) {
  c = 1.0;
  s = 0.0;
  null = true;
  const int ea = exp_field(apq);
  if (((__double2hiint(apq) << 1) | __double2loint(apq)) == 0) return;
  const double d = aqq - app;
  const int ed = exp_field(d), E = max(ea, ed);
  if (E == 0x7FF) {  // infinite or NaN: the result is undefined, as it always was
    c = s = __longlong_as_double(0x7ff8000000000000ll);
    null = false;
    return;
  }
  null = 2 * ea + 72 <= exp_field(app) + exp_field(aqq);
  const float a = scaled32(apq, E);
  if (a == 0.f) return;
  const float t = tan32(scaled32(d, E), a);
  // c = 1 / sqrt(1 + t^2) from the FP32 value by one third-order step
  const double T = f32_to_f64(t), x = f32_to_f64(rsqrt32(fmaf(t, t, 1.f)));
  const double u = fma(T, T, 1.0);
  const double e = fma(-(u * x), x, 1.0);
  c = fma(x * e, fma(0.375, e, 0.5), x);
  s = T * c;
}

// bits of a double as an unsigned key in the values' order (no NaN), and of its magnitude
__device__ __forceinline__ unsigned long long order_key(double x) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  return (b >> 63) ? ~b : b | (1ull << 63);
}
__device__ __forceinline__ unsigned long long magnitude_key(double x) {
  return static_cast<unsigned long long>(__double_as_longlong(x)) & ~(1ull << 63);
}

constexpr int kThreads = 256;  // of every block that runs these

// fixed-order sum over the block, in every thread
template <typename T>
__device__ __forceinline__ T block_total(T v, T* s_red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
  __syncthreads();
  T t = s_red[threadIdx.x & 7];
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  __syncthreads();
  return t;
}
template <typename T>
__device__ __forceinline__ T block_max(T v, T* s_red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
  __syncthreads();
  T t = s_red[threadIdx.x & 7];
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) t = max(t, __shfl_xor_sync(0xffffffffu, t, o));
  __syncthreads();
  return t;
}

// ------------------------------- FP64 -------------------------------
struct Scratch64 {
  double c[128], s[128], red[8];
  int p[128], q[128], null[128];
};

// Cyclic Jacobi on A (order n, at most 256; shared or global memory), its rotations applied to V's
// columns, which hold the basis on entry.  Returns the sweeps taken.
__device__ inline int jacobi64(double* A, int lda, double* V, int ldv, int n, Scratch64& S) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, m = n + (n & 1), h = m / 2;
  double fro2 = 0.0;
  int sweep = 0;
  for (; sweep < 60; ++sweep) {
    double off = 0.0, dia = 0.0;
    for (int r = warp; r < n; r += kThreads / 32)
      for (int c = lane; c < n; c += 32) {
        const double x = A[r * lda + c];
        if (r != c)
          off = fma(x, x, off);
        else
          dia = fma(x, x, dia);
      }
    off = block_total(off, S.red);
    if (sweep == 0) fro2 = block_total(dia, S.red) + off;
    if (off == 0.0 || off <= 1e-34 * fro2) break;
    for (int round = 0; round < m - 1; ++round) {
      if (tid < h) {
        int p, q;
        pair_of(round, tid, m, p, q);
        double c = 1.0, s = 0.0;
        bool null = true;
        if (q < n) rotation64(A[p * lda + p], A[q * lda + q], A[p * lda + q], c, s, null);
        S.c[tid] = c;
        S.s[tid] = s;
        S.p[tid] = p;
        S.q[tid] = q;
        S.null[tid] = null;
      }
      __syncthreads();
      // rows p, q, then columns p, q (and of V): pairs over the warps, lanes along the row or column
      for (int i = warp; i < h; i += kThreads / 32) {
        const int p = S.p[i], q = S.q[i];
        const double c = S.c[i], s = S.s[i];
        if (q >= n || s == 0.0) continue;
        for (int k = lane; k < n; k += 32) {
          const double x = A[p * lda + k], y = A[q * lda + k];
          A[p * lda + k] = fma(c, x, -(s * y));
          A[q * lda + k] = fma(s, x, c * y);
        }
      }
      __syncthreads();
      for (int i = warp; i < h; i += kThreads / 32) {
        const int p = S.p[i], q = S.q[i];
        const double c = S.c[i], s = S.s[i];
        if (q >= n || s == 0.0) continue;
        for (int k = lane; k < n; k += 32) {
          const double x = A[k * lda + p], y = A[k * lda + q];
          A[k * lda + p] = fma(c, x, -(s * y));
          A[k * lda + q] = fma(s, x, c * y);
          const double v = V[k * ldv + p], w = V[k * ldv + q];
          V[k * ldv + p] = fma(c, v, -(s * w));
          V[k * ldv + q] = fma(s, v, c * w);
        }
      }
      __syncthreads();
      if (tid < h && S.q[tid] < n && S.s[tid] != 0.0) {
        const int p = S.p[tid], q = S.q[tid];
        const double x = S.null[tid] ? 0.0 : A[p * lda + q];
        A[p * lda + q] = x;
        A[q * lda + p] = x;
      }
      __syncthreads();
    }
  }
  return sweep;
}

// ------------------------------- FP32, shared memory -------------------------------
// Cyclic Jacobi on a matrix of even order M.  Instead of moving the pairs over a fixed matrix, every
// round rotates the same pairs of positions (i, h + i), i < h = M / 2, and writes its result to where
// the next round wants it: position 0 stays, the others move one place around the ring
// 1, 2, .. h - 1, 2h - 1, .. h + 1, h.  After M - 1 rounds every two indices have met and all are back.
// So with M known at compile time a thread's addresses are a few registers and immediate offsets for
// the whole solve (rows over the warps, lanes along the pairs: all accesses conflict-free): a rotated
// row pair costs 28 instructions, a row of V eight.  The rounds are bound by instruction issue:
// finding pairs and addresses anew in each, order 64 took 3100 cycles a round.
constexpr int k32Max = 96;  // largest order
struct Scratch32 {
  float2 rot[2][k32Max / 2];  // (c, s) of every pair of a round
  float red[8];
};
// floats of the work area of order m: two copies of the matrix, then two of the vectors
__host__ __device__ constexpr int jacobi32_floats(int m) { return 4 * m * m; }

template <int OFF>
__device__ __forceinline__ float lds32(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(a), "n"(OFF) : "memory");
  return v;
}
template <int OFF>
__device__ __forceinline__ float2 lds64(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2+%3];" : "=f"(v.x), "=f"(v.y) : "r"(a), "n"(OFF) : "memory");
  return v;
}
template <int OFF>
__device__ __forceinline__ void sts32(uint32_t a, float v) {
  asm volatile("st.shared.f32 [%0+%1], %2;" ::"r"(a), "n"(OFF), "f"(v) : "memory");
}

template <int M>
struct Jacobi32 {
  static constexpr int h = M / 2;
  static constexpr int HP = h <= 8 ? 8 : h <= 16 ? 16 : 32;  // lanes along the pairs
  static constexpr int NSUB = 32 / HP;                       // rows a warp takes at once
  static constexpr int NG = (h + 31) / 32;                   // pairs of a lane
  static constexpr int WA = (h + 31) / 32, NW = kThreads / 32 - WA;  // WA warps find the angles, NW rotate V
  static constexpr int SA = kThreads / 32 * NSUB, SV = NW * NSUB;    // row steps
  static constexpr int UA = (h + SA - 1) / SA, UV = (M + SV - 1) / SV;
  static constexpr int kCopy = 4 * M * M;                    // bytes from one copy to the other
  static_assert(M % 2 == 0 && M <= k32Max, "order");

  static __device__ __forceinline__ int next_place(int t) {
    if (t == 0) return 0;
    if (t < h) return t == h - 1 ? 2 * h - 1 : t + 1;
    return t == h ? 1 : t - 1;
  }

  uint32_t rot, ang;            // rotations; the angle thread's diagonal block
  uint32_t rj[NG], ri;          // this lane's and this row pair's rotations
  uint32_t a;                   // A at this thread's first row pair and pair of columns
  uint32_t dt[NG], db[NG];      // where row i + 1 of the next copy takes the two columns
  uint32_t v, vt[NG], vb[NG];   // the same for a row of V
  uint32_t first_t, first_b, last_t;  // rows' byte offsets from those of i + 1 and h + i - 1 at the ring's ends
  int i0, j0, r0, tid;

  __device__ __forceinline__ Jacobi32(const float* A, const float* V, Scratch32& S) {
    tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5, sub = lane / HP;
    j0 = lane % HP;
    i0 = warp * NSUB + sub;
    r0 = (warp - WA) * NSUB + sub;
    rot = smem_u32(S.rot);
    ri = rot + 8 * i0;
    ang = smem_u32(A) + 4 * (tid * M + tid);
    a = smem_u32(A) + 4 * (i0 * M + j0);
    v = smem_u32(V) + 4 * (r0 * M + j0);
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      const int j = j0 + 32 * g, t = j < h ? next_place(j) : 0, b = j < h ? next_place(h + j) : 0;
      rj[g] = rot + 8 * j;
      dt[g] = smem_u32(A) + 4 * ((i0 + 1) * M + t);
      db[g] = smem_u32(A) + 4 * ((i0 + 1) * M + b);
      vt[g] = smem_u32(V) + 4 * (r0 * M + t);
      vb[g] = smem_u32(V) + 4 * (r0 * M + b);
    }
    // row pair i goes to rows i + 1 and h + i - 1, pair 0 to 0 and 1, and pair h - 1's first row to 2h - 1
    first_t = i0 == 0 ? static_cast<uint32_t>(-4 * M) : 0u;
    first_b = i0 == 0 ? static_cast<uint32_t>(4 * M * (1 - (h - 1))) : 0u;
    last_t = i0 + (UA - 1) * SA == h - 1 ? static_cast<uint32_t>(4 * M * (h - 1)) : 0u;
  }

  __device__ __forceinline__ bool lane_has(int g) const { return j0 + 32 * g < h; }

  // V's columns by the rotations in rot[1 - B], from copy 1 - B to copy B (warps WA on)
  template <int B>
  __device__ __forceinline__ void rotate_V() const {
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      if (!lane_has(g)) continue;
      const float2 r = B ? lds64<0>(rj[g]) : lds64<8 * (k32Max / 2)>(rj[g]);
      rows_of_V<B>(g, r, std::make_integer_sequence<int, UV>{});
    }
  }
  template <int B, int... U>
  __device__ __forceinline__ void rows_of_V(int g, const float2& r, std::integer_sequence<int, U...>) const {
    float x[UV], y[UV];
    (load_V<B, U>(g, x[U], y[U]), ...);
    (store_V<B, U>(g, r, x[U], y[U]), ...);
  }
  template <int B, int U>
  __device__ __forceinline__ void load_V(int g, float& x, float& y) const {
    if (r0 + U * SV >= M) return;
    constexpr int o = (1 - B) * kCopy + 4 * U * SV * M;
    x = g ? lds32<o + 128>(v) : lds32<o>(v);
    y = g ? lds32<o + 4 * h + 128>(v) : lds32<o + 4 * h>(v);
  }
  template <int B, int U>
  __device__ __forceinline__ void store_V(int g, const float2& r, float x, float y) const {
    if (r0 + U * SV >= M) return;
    constexpr int o = B * kCopy + 4 * U * SV * M;
    sts32<o>(vt[g], fmaf(r.x, x, -(r.y * y)));
    sts32<o>(vb[g], fmaf(r.y, x, r.x * y));
  }

  // row pairs of A by the rotations in rot[B] from both sides, from copy B to copy 1 - B
  template <int B>
  __device__ __forceinline__ void rotate_A() const {
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      if (!lane_has(g)) continue;
      const float2 r = B ? lds64<8 * (k32Max / 2)>(rj[g]) : lds64<0>(rj[g]);
      pairs_of_A<B>(g, r, std::make_integer_sequence<int, UA>{});
    }
  }
  template <int B, int... U>
  __device__ __forceinline__ void pairs_of_A(int g, const float2& r, std::integer_sequence<int, U...>) const {
    float x[UA][4];
    float2 q[UA];
    (load_A<B, U>(g, x[U], q[U]), ...);
    (store_A<B, U>(g, r, x[U], q[U]), ...);
  }
  template <int B, int U>
  __device__ __forceinline__ void load_A(int g, float (&x)[4], float2& q) const {
    if ((U + 1) * SA > h && i0 + U * SA >= h) return;
    constexpr int o = B * kCopy + 4 * U * SA * M;
    q = lds64<8 * U * SA + B * 8 * (k32Max / 2)>(ri);
    x[0] = g ? lds32<o + 128>(a) : lds32<o>(a);
    x[1] = g ? lds32<o + 4 * h + 128>(a) : lds32<o + 4 * h>(a);
    x[2] = g ? lds32<o + 4 * h * M + 128>(a) : lds32<o + 4 * h * M>(a);
    x[3] = g ? lds32<o + 4 * h * M + 4 * h + 128>(a) : lds32<o + 4 * h * M + 4 * h>(a);
  }
  template <int B, int U>
  __device__ __forceinline__ void store_A(int g, const float2& rj_, const float (&x)[4], const float2& q) const {
    if ((U + 1) * SA > h && i0 + U * SA >= h) return;
    constexpr int o = (1 - B) * kCopy + 4 * U * SA * M, ob = o + 4 * M * (h - 2);  // rows i + 1 and h + i - 1
    const float u00 = fmaf(rj_.x, x[0], -(rj_.y * x[1])), u01 = fmaf(rj_.y, x[0], rj_.x * x[1]);
    const float u10 = fmaf(rj_.x, x[2], -(rj_.y * x[3])), u11 = fmaf(rj_.y, x[2], rj_.x * x[3]);
    const bool diag = i0 + U * SA == j0 + 32 * g;  // the rotated pair's own entry is zero by construction
    const float y00 = fmaf(q.x, u00, -(q.y * u10)), y11 = fmaf(q.y, u01, q.x * u11);
    const float y01 = diag ? 0.f : fmaf(q.x, u01, -(q.y * u11)), y10 = diag ? 0.f : fmaf(q.y, u00, q.x * u10);
    uint32_t tt = dt[g], tb = db[g], bt = dt[g], bb = db[g];
    if (U == 0) {
      tt += first_t;
      tb += first_t;
      bt += first_b;
      bb += first_b;
    }
    if (U == UA - 1) {
      tt += last_t;
      tb += last_t;
    }
    sts32<o>(tt, y00);
    sts32<o>(tb, y01);
    sts32<ob>(bt, y10);
    sts32<ob>(bb, y11);
  }

  // one round on copy B of A; the last round's rotations of V if there are any
  template <int B>
  __device__ __forceinline__ void round(bool pending) const {
    if (tid < 32 * WA) {
      if (tid < h) {
        const float x = lds32<B * kCopy + 4 * h>(ang);
        const float d = lds32<B * kCopy + 4 * h * M + 4 * h>(ang) - lds32<B * kCopy>(ang);
        const float t = fabsf(x) > 1e-18f ? tan32(d, x) : 0.f;  // the matrix is scaled to order one
        const float c = rsqrt32(fmaf(t, t, 1.f));
        sts32<B * 8 * (k32Max / 2)>(rot + 8 * tid, c);
        sts32<B * 8 * (k32Max / 2) + 4>(rot + 8 * tid, t * c);
      }
    } else if (pending) {
      rotate_V<B>();
    }
    __syncthreads();
    rotate_A<B>();
    __syncthreads();
  }
  // (by value: the copy lives in registers)
  template <int B>
  static __device__ __noinline__ void sweep(Jacobi32 J, bool pending) {
#pragma unroll 1
    for (int r = 0; r < h - 1; ++r) {
      J.template round<B>(pending);
      J.template round<1 - B>(true);
      pending = true;
    }
    J.template round<B>(pending);
  }
};

// Cyclic Jacobi in FP32 on A (M x M floats, followed by its next copy), its rotations applied to V's
// columns (the same).  At most max_sweeps; stops once the off-diagonal part is at the level of FP32
// rounding.  Returns the sweeps taken; `copy`: which copies hold the results.
template <int M>
__device__ __forceinline__ int jacobi32(const float* A, const float* V, int max_sweeps, Scratch32& S, int& copy) {
  const int tid = threadIdx.x;
  const Jacobi32<M> J(A, V, S);
  float prev = 0.f, fro2 = 0.f;
  int sweep = 0;
  copy = 0;
  for (; sweep < max_sweeps; ++sweep) {
    if (max_sweeps > 1) {
      const float* X = A + copy * M * M;
      float off = 0.f, dia = 0.f;
      for (int i = tid; i < M * M; i += kThreads) {
        const float x = X[i];
        if (i / M != i % M)
          off = fmaf(x, x, off);
        else
          dia = fmaf(x, x, dia);
      }
      off = block_total(off, S.red);
      if (sweep == 0) fro2 = block_total(dia, S.red) + off;
      if (!(off > 1e-14f * fro2) || (sweep > 0 && off <= 1e-9f * fro2 && off > 0.25f * prev)) break;
      prev = off;
    }
    if (copy == 0)
      Jacobi32<M>::template sweep<0>(J, sweep > 0);
    else
      Jacobi32<M>::template sweep<1>(J, sweep > 0);
    copy ^= 1;
  }
  if (sweep > 0 && tid >= 32 * Jacobi32<M>::WA) {
    if (copy == 0)
      J.template rotate_V<0>();
    else
      J.template rotate_V<1>();
  }
  __syncthreads();
  return sweep;
}
// the order FP32 rotations take n columns at: a multiple of eight up to 32, of sixteen above
__host__ __device__ constexpr int jacobi32_order(int n) { return n <= 32 ? (n + 7) / 8 * 8 : (n + 15) / 16 * 16; }

// ------------------------------- refinement -------------------------------
// One entry of the correction of approximate eigenvectors X of A (Ogita and Aishima, "Iterative
// refinement for symmetric eigenvalue decomposition", 2018): with S = X^T A X, G = X^T X and
// lambda_i = S_ii / G_ii, X (I + E) is better by a square.  A pair whose eigenvalues are too close
// for the first-order step (unresolved; its off-diagonal above `noise`) is counted in bad, and only
// made orthogonal.
__device__ __forceinline__ double correction(int i, int j, double S, double G, double li, double lj, double noise,
                                             int& bad) {
  const double num = i == j ? 1.0 - G : fma(-lj, G, S), an = fabs(num);
  if (!(an <= 1e300)) {  // not finite
    bad = 2;
    return 0.0;
  }
  if (i == j) return 0.5 * num;
  const double gap = lj - li, ag = fabs(gap);
  const bool small = an <= noise;
  if (ag > 0.0 && an <= (small ? 1e-9 : 0.125) * ag) return num / gap;
  if (!small) bad = max(bad, 1);
  return -0.5 * G;
}
// E - 1023 for a matrix whose squared Frobenius norm is fro2 (normal): every |entry| < 2^(E - 1023)
__device__ __forceinline__ int scale_exponent(double fro2) { return 1023 + (exp_field(fro2) - 1023 + 2 + 2048) / 2 - 1024; }
// corrections below this need no further step: what it leaves behind is their square times sqrt(m)
constexpr double kRefined = 5e-9;

}  // namespace eig
}  // namespace ss
