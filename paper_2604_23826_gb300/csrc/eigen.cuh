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

// About a^2 / |p q| of an entry a between the diagonal's p and q, from the exponents alone (a power of
// two, at most 1; 0 for a = 0): sums of these tell how far a matrix is from diagonal in each pair's own
// units.  Columns of very different units have eigenvalues far below the rounding of the largest, and an
// off-diagonal that is nothing beside the norm may be everything to two of those.  fp, fq: exponents that
// the diagonal's count as at least, of what its own rounding comes from.
__device__ __forceinline__ float square_ratio(int ea, int ep, int eq, int fp, int fq) {
  const int d = 2 * ea - max(ep, fp) - max(eq, fq);
  return ea == 0 || d < -126 ? 0.f : __int_as_float((127 + min(d, 0)) << 23);
}
__device__ __forceinline__ int exp_field32(float x) { return (__float_as_int(x) >> 23) & 0xFF; }

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
__device__ __forceinline__ int block_or(int v, int* s_red) {
  v = __reduce_or_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
  __syncthreads();
  const int t = __reduce_or_sync(0xffffffffu, s_red[threadIdx.x & 7]);
  __syncthreads();
  return t;
}

// A matrix's diagonal (at most 256), by the block: the exponent field of its smallest that is not zero, and the
// diagonal itself in FP32 over 2^(E - 1023), E - 1023 even and every |entry| below that.
struct Variances {
  int least, E;
};
__device__ __forceinline__ Variances variances(const double* A, int ld, int n, float* diag, int* s_red) {
  const int t = threadIdx.x;
  const double a = t < n ? A[static_cast<size_t>(t) * (ld + 1)] : 0.0;
  const int e = exp_field(a);
  Variances v{-block_max(e ? -e : -0x7FF, s_red), block_max(e, s_red) + 1};
  v.E += (v.E + 1) & 1;
  if (t < n) diag[t] = fabsf(scaled32(a, v.E));
  __syncthreads();
  return v;
}
// A column's weight sum_l a_ll x_lj^2, from the scaled diagonal, as an exponent field: products with it round to
// about eps of that.
__device__ __forceinline__ int weight_exponent(float w, int E) { return exp_field32(w) ? exp_field32(w) - 127 + E : 0; }

// ------------------------------- FP64 -------------------------------
struct Scratch64 {
  double c[128], s[128], red[8];
  int p[128], q[128], null[128], weight[256];
};

// FP64 rotations are at an end when the off-diagonal is negligible (`norm`, by the caller) and so are the
// sum of its ratios in the pairs' own units: below 1e-28, or at the level of rounding (2e-15 an entry) and
// falling no further, or falling no further for four sweeps.  (Rotations from the refined basis of a
// cluster of close eigenvalues may reduce little in their first sweeps.)
struct Ratios64 {
  float prev = 0.f;
  int stalled = 0;
  bool settled = false;
  __device__ __forceinline__ bool done(bool norm, float rel, int n) {
    stalled = settled && rel > 0.0625f * prev ? stalled + 1 : 0;
    settled |= norm;
    prev = rel;
    return settled && (rel <= 1e-28f || (stalled >= 1 && rel <= 4e-30f * n * n) || stalled >= 4);
  }
};

// Cyclic Jacobi on A (order n, at most 256; shared or global memory), its rotations applied to V's
// columns, which hold the basis on entry; diag, E: of the matrix in its own basis.  Returns the sweeps taken.
__device__ inline int jacobi64(double* A, int lda, double* V, int ldv, int n, const float* diag, int E, Scratch64& S) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, m = n + (n & 1), h = m / 2;
  double fro2 = 0.0;
  Ratios64 ratios;
  int sweep = 0;
  for (; sweep < 60; ++sweep) {
    double off = 0.0, dia = 0.0;
    float rel = 0.f;
    if (tid < n) {
      float w = 0.f;
      for (int l = 0; l < n; ++l) {
        const float x = scaled32(V[l * ldv + tid], 1023);
        w = fmaf(diag[l] * x, x, w);
      }
      S.weight[tid] = weight_exponent(w, E);
    }
    __syncthreads();
    for (int r = warp; r < n; r += kThreads / 32)
      for (int c = lane; c < n; c += 32) {
        const double x = A[r * lda + c];
        if (r != c) {
          off = fma(x, x, off);
          rel += square_ratio(exp_field(x), exp_field(A[r * lda + r]), exp_field(A[c * lda + c]), S.weight[r],
                              S.weight[c]);
        } else {
          dia = fma(x, x, dia);
        }
      }
    off = block_total(off, S.red);
    rel = block_total(rel, reinterpret_cast<float*>(S.red));
    if (sweep == 0) fro2 = block_total(dia, S.red) + off;
    if (off == 0.0 || ratios.done(off <= 1e-34 * fro2, rel, n)) break;
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
// row pair costs 28 instructions, a row of V eight.  V follows A one round behind, and its rotation
// fills the time the angles take.  Up to order 32 every warp finds all the angles itself, a pair a
// lane, and takes those of its row pairs by shuffles: a round has one barrier.  Above, shared memory is
// the bound (order 64: 512 of a round's 1000 cycles) and that costs more than it saves (324 us against
// 337 for 64 columns): one warp finds the angles while the others rotate V, then all rotate A.
// kCross: only the h^2 pairs of an index below h and one above, in h rounds: the lower positions stay,
// the upper ones move one place around their own ring.
// Runs on NT threads (numbered tid), the whole block or warps that meet at barrier `bar`.
constexpr int k32Max = 64;  // largest order
struct Scratch32 {
  float2 rot[k32Max / 2];  // (c, s) of every pair of a round
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
__device__ __forceinline__ float2 lds_rot(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts_rot(uint32_t a, float2 v) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
template <int OFF>
__device__ __forceinline__ void sts32(uint32_t a, float v) {
  asm volatile("st.shared.f32 [%0+%1], %2;" ::"r"(a), "n"(OFF), "f"(v) : "memory");
}

template <int M, int NT = kThreads, bool kCross = false>
struct Jacobi32 {
  static constexpr int h = M / 2;
  static constexpr int HP = h <= 8 ? 8 : h <= 16 ? 16 : 32;  // lanes along the pairs
  static constexpr int SA = NT / HP;                         // rows the warps take at once
  static constexpr bool kSelf = h <= 16;                     // every warp finds the angles
  static constexpr int SV = kSelf ? SA : SA - 1;             // rows of V: all warps, or all but the first
  static constexpr int UA = (h + SA - 1) / SA, UV = (M + SV - 1) / SV;
  static constexpr int kCopy = 4 * M * M;                    // bytes from one copy to the other
  static constexpr int kRounds = kCross ? h : M - 1;
  // row pair i goes to rows i + kTop and h + i + kBot, but for the ends of the ring
  static constexpr int kTop = kCross ? 0 : 1, kBot = kCross ? 1 : -1;
  static_assert(M % 2 == 0 && M <= k32Max && (!kCross || h % 2 == 0) && (kSelf || HP == 32), "order");

  static __device__ __forceinline__ int next_place(int t) {
    if (kCross) return t < h ? t : t == M - 1 ? h : t + 1;
    if (t == 0) return 0;
    if (t < h) return t == h - 1 ? M - 1 : t + 1;
    return t == h ? 1 : t - 1;
  }

  uint32_t ang;     // the diagonal block of this lane's pair
  uint32_t a, v;    // A at this thread's first row pair and pair of columns, V at its first row
  uint32_t dt, db;  // where row i0 + kTop of the next copy takes the two columns
  uint32_t vt, vb;  // the same for a row of V
  uint32_t first_t, first_b, last_t, last_b;  // what the ends of the ring add to the rows' byte offsets
  uint32_t rot;     // the rotations
  int i0, r0, j0, bar;

  __device__ __forceinline__ Jacobi32(const float* A, const float* V, Scratch32& S, int tid, int barrier) {
    i0 = tid / HP;
    r0 = kSelf ? i0 : i0 - 1;
    rot = smem_u32(S.rot);
    j0 = tid % HP;
    bar = barrier;
    const int j = min(j0, h - 1), t = next_place(j), b = next_place(h + j);
    ang = smem_u32(A) + 4 * (j * M + j);
    a = smem_u32(A) + 4 * (i0 * M + j);
    v = smem_u32(V) + 4 * (r0 * M + j);
    dt = smem_u32(A) + 4 * ((i0 + kTop) * M + t);
    db = smem_u32(A) + 4 * ((i0 + kTop) * M + b);
    vt = smem_u32(V) + 4 * (r0 * M + t);
    vb = smem_u32(V) + 4 * (r0 * M + b);
    const int i1 = i0 + (UA - 1) * SA;  // this thread's last row pair
    first_t = i0 == 0 ? 4 * M * (next_place(0) - kTop) : 0;
    first_b = i0 == 0 ? 4 * M * (next_place(h) - (h + kBot)) : 0;
    last_t = i1 == h - 1 ? 4 * M * (next_place(h - 1) - (h - 1 + kTop)) : 0;
    last_b = i1 == h - 1 ? 4 * M * (next_place(M - 1) - (M - 1 + kBot)) : 0;
  }

  template <int B, int U>
  __device__ __forceinline__ void load_A(float (&x)[4]) const {
    if ((U + 1) * SA > h && i0 + U * SA >= h) return;
    constexpr int o = B * kCopy + 4 * U * SA * M;
    x[0] = lds32<o>(a);
    x[1] = lds32<o + 4 * h>(a);
    x[2] = lds32<o + 4 * h * M>(a);
    x[3] = lds32<o + 4 * h * M + 4 * h>(a);
  }
  template <int B, int U>
  __device__ __forceinline__ void store_A(float c, float s, const float (&x)[4], float ci, float si) const {
    if (((U + 1) * SA > h && i0 + U * SA >= h) || (HP > h && j0 >= h)) return;
    constexpr int o = (1 - B) * kCopy + 4 * U * SA * M, ob = o + 4 * M * (h + kBot - kTop);
    const float u00 = fmaf(c, x[0], -(s * x[1])), u01 = fmaf(s, x[0], c * x[1]);
    const float u10 = fmaf(c, x[2], -(s * x[3])), u11 = fmaf(s, x[2], c * x[3]);
    const bool diag = i0 + U * SA == j0;  // the rotated pair's own entry is zero by construction
    const float y00 = fmaf(ci, u00, -(si * u10)), y11 = fmaf(si, u01, ci * u11);
    const float y01 = diag ? 0.f : fmaf(ci, u01, -(si * u11)), y10 = diag ? 0.f : fmaf(si, u00, ci * u10);
    const uint32_t top = (U == 0 ? first_t : 0u) + (U == UA - 1 ? last_t : 0u);
    const uint32_t bot = (U == 0 ? first_b : 0u) + (U == UA - 1 ? last_b : 0u);
    sts32<o>(dt + top, y00);
    sts32<o>(db + top, y01);
    sts32<ob>(dt + bot, y10);
    sts32<ob>(db + bot, y11);
  }
  template <int B, int U>
  __device__ __forceinline__ void load_V(float (&x)[2]) const {
    if ((U + 1) * SV > M && r0 + U * SV >= M) return;
    constexpr int o = B * kCopy + 4 * U * SV * M;
    x[0] = lds32<o>(v);
    x[1] = lds32<o + 4 * h>(v);
  }
  template <int B, int U>
  __device__ __forceinline__ void store_V(float c, float s, const float (&x)[2]) const {
    if (((U + 1) * SV > M && r0 + U * SV >= M) || (HP > h && j0 >= h)) return;
    constexpr int o = (1 - B) * kCopy + 4 * U * SV * M;
    sts32<o>(vt, fmaf(c, x[0], -(s * x[1])));
    sts32<o>(vb, fmaf(s, x[0], c * x[1]));
  }

  // V's rows by the rotations of the round before, from copy B to copy 1 - B
  template <int B, int... W>
  __device__ __forceinline__ void rotate_V(float2 rot, std::integer_sequence<int, W...>) const {
    float y[UV][2];
    (load_V<B, W>(y[W]), ...);
    (store_V<B, W>(rot.x, rot.y, y[W]), ...);
  }
  __device__ __forceinline__ void meet() const {
    if (NT == kThreads)
      __syncthreads();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(NT) : "memory");
  }
  // The rotation (c, s) that annihilates apq, |angle| <= pi / 4: cos(2 angle) = |d| / sqrt(d^2 + 4 apq^2),
  // d = aqq - app, then c and s from the half-angle formulas, and c once more from c^2 + s^2 = 1 (the
  // roots' last bits would change the vectors' lengths, round after round): a chain of two reciprocal
  // roots, where the tangent's had four special functions.
  __device__ __forceinline__ static float2 angle(float apq, float app, float aqq) {
    const float d = aqq - app;
    const float r = rsqrt32(fmaf(d, d, 4.f * apq * apq));
    const float c2 = fmaf(0.5f * fabsf(d), r, 0.5f);
    const float y = rsqrt32(c2), c = c2 * y, s = (d >= 0.f ? apq : -apq) * r * y;
    const float e = fmaf(c, c, fmaf(s, s, -1.f));
    const bool turn = fabsf(apq) > 1e-18f;  // 30 decades below the matrix's norm (kUp32)
    return make_float2(turn ? fmaf(-0.5f * e, y, c) : 1.f, turn ? s : 0.f);
  }
  // one round of A, from copy B to copy 1 - B, and (kV) of V the round before (now: the last round's
  // rotation of this lane's pair, then this one's)
  template <int B, bool kV, int... U, class SeqV>
  __device__ __forceinline__ void round(float2& now, std::integer_sequence<int, U...>, SeqV uv) const {
    float x[UA][4];
    float2 q[UA];
    if (kSelf) {
      const float apq = lds32<B * kCopy + 4 * h>(ang), app = lds32<B * kCopy>(ang);
      const float aqq = lds32<B * kCopy + 4 * h * M + 4 * h>(ang);
      (load_A<B, U>(x[U]), ...);
      const float2 r = angle(apq, app, aqq);
      if (kV) rotate_V<1 - B>(now, uv);
      now = r;
      ((q[U].x = __shfl_sync(0xffffffffu, r.x, min(i0 + U * SA, h - 1)),
        q[U].y = __shfl_sync(0xffffffffu, r.y, min(i0 + U * SA, h - 1))),
       ...);
    } else {
      if (i0 == 0) {
        const float apq = lds32<B * kCopy + 4 * h>(ang), app = lds32<B * kCopy>(ang);
        const float aqq = lds32<B * kCopy + 4 * h * M + 4 * h>(ang);
        const float2 r = angle(apq, app, aqq);
        if (j0 < h) sts_rot(rot + 8 * j0, r);
      } else if (kV) {
        rotate_V<1 - B>(now, uv);
      }
      meet();
      now = lds_rot(rot + 8 * min(j0, h - 1));
      ((q[U] = lds_rot(rot + 8 * min(i0 + U * SA, h - 1))), ...);
      (load_A<B, U>(x[U]), ...);
    }
    (store_A<B, U>(now.x, now.y, x[U], q[U].x, q[U].y), ...);
    meet();
  }
  // (by value: the copy lives in registers)
  template <int B>
  static __device__ __noinline__ void sweep(Jacobi32 J) {
    constexpr auto ua = std::make_integer_sequence<int, UA>{};
    constexpr auto uv = std::make_integer_sequence<int, UV>{};
    float2 now = make_float2(1.f, 0.f);
    J.template round<B, false>(now, ua, uv);
#pragma unroll 1
    for (int r = 0; r < (kRounds - 1) / 2; ++r) {
      J.template round<1 - B, true>(now, ua, uv);
      J.template round<B, true>(now, ua, uv);
    }
    if (kRounds % 2 == 0) J.template round<1 - B, true>(now, ua, uv);
    if (kSelf || J.i0 > 0) J.template rotate_V<kRounds % 2 ? B : 1 - B>(now, uv);
    J.meet();
  }
};

// FP32 rotations are at an end when the off-diagonal is at the level of FP32's rounding (or falls no
// further near it), and in the pairs' own units too: the small eigenvalues of columns of different units
// (or of a nearly diagonal seeded matrix) are rotated as far as the large ones.
template <typename T>
__device__ __forceinline__ bool rotated32(int sweep, T off, T prev, T fro2, T done, float rel, float prev_rel) {
  const bool norm = !(off > done * fro2) || (sweep > 0 && off <= T(1e-9) * fro2 && off > T(0.25) * prev);
  return norm && (rel <= 1e-6f || (sweep > 0 && rel > 0.25f * prev_rel));
}

// Cyclic Jacobi in FP32 on A (M x M floats, followed by its next copy), its rotations applied to V's
// columns (the same), by the whole block.  At most max_sweeps; stops once the off-diagonal part is at
// the level of FP32 rounding.  floor: of the smallest variance.  Returns the sweeps taken; `copy`: which copies hold
// the results.
template <int M>
__device__ __forceinline__ int jacobi32(const float* A, const float* V, int max_sweeps, int floor, Scratch32& S, int& copy) {
  const int tid = threadIdx.x;
  const Jacobi32<M> J(A, V, S, tid, 0);
  float prev = 0.f, prev_rel = 0.f, fro2 = 0.f;
  int sweep = 0;
  copy = 0;
  for (; sweep < max_sweeps; ++sweep) {
    const float* X = A + copy * M * M;
    float off = 0.f, dia = 0.f, rel = 0.f;
    for (int i = tid; i < M * M; i += kThreads) {
      const float x = X[i];
      const int r = i / M, c = i % M;
      if (r != c) {
        off = fmaf(x, x, off);
        rel += square_ratio(exp_field32(x), exp_field32(X[r * M + r]), exp_field32(X[c * M + c]), floor, floor);
      } else {
        dia = fmaf(x, x, dia);
      }
    }
    off = block_total(off, S.red);
    rel = block_total(rel, S.red);
    if (sweep == 0) fro2 = block_total(dia, S.red) + off;
    if (rotated32(sweep, off, prev, fro2, M <= 24 ? 1e-14f : 1e-12f, rel, prev_rel)) break;
    prev = off;
    prev_rel = rel;
    if (copy == 0)
      Jacobi32<M>::template sweep<0>(J);
    else
      Jacobi32<M>::template sweep<1>(J);
    copy ^= 1;
  }
  return sweep;
}
// ------------------------------- refinement -------------------------------
// What rounding leaves in an entry of X^T A X that should be zero depends on its two columns: a
// covariance's |a_kl| <= sqrt(a_kk a_ll), so products of the columns i and j of X leave about eps b_i b_j,
// b_j^2 = sum_l a_ll x_lj^2, which is far below the norm's rounding where both columns are combinations of
// table columns of small units (and near it where a rank-deficient matrix has its zero eigenvalues).
// A column's share of that, and of the rounding of its eigenvalue, is kept as its noise: an entry's is
// the product of two.  (A bound from the norm took FP32's leavings among small eigenvalues for rounding:
// 40 columns of units over four decades, vectors wrong by 3e-7, over eight by 4e-3; now to 1e-14.)
struct Noise {
  double unit;  // 2^((E - 1023) / 2)
  int E;        // of variances()
  float root;   // 4 sqrt(columns)
  // of a column: `weight` = sum_l a_ll x_lj^2, scaled; `f` and `inverse` for the ratios of two columns
  __device__ __forceinline__ double column(double lambda, float weight, float& f, float& inverse) const {
    f = 1.0536712e-8f * sqrtf(fmaxf(16.f * fabsf(scaled32(lambda, E)), root * weight));  // sqrt(2^-53) times
    inverse = f > 0.f ? 1.f / f : 0.f;
    return f32_to_f64(f) * unit;
  }
};
// an exponent E with every |entry| < 2^(E - 1023), for a matrix whose squared Frobenius norm is fro2 (normal)
__device__ __forceinline__ int scale_exponent(double fro2) { return 1023 + (exp_field(fro2) - 1023 + 2 + 2048) / 2 - 1024; }
__device__ __forceinline__ Noise noise_of(int E, int n) {
  return Noise{__hiloint2double((1023 + (E - 1023) / 2) << 20, 0), E, 4.f * sqrtf(static_cast<float>(n))};
}
// FP32 rotations take the matrix at 2^40 times its scale, so that what they leave alone (1e-18, whose square
// FP32 still holds) lies 30 decades below the norm
constexpr int kUp32 = 40;
// the smallest variance's exponent in the matrix those work on (E: scale_exponent)
__device__ __forceinline__ int floor32(int least, int E) { return max(0, min(254, least - E + kUp32 + 127)); }

// corrections below this need no further step: what it leaves behind is their square times sqrt(m)
constexpr float kRefined = 5e-9f;
// of an entry's noise: off-diagonals below this may, in the first step, be the squares of FP32's errors
constexpr double kCoarse = 5000.0;
constexpr int kSteps = 8;
constexpr int kPolish = 3;  // the step to go on from after FP64 rotations: small corrections, then none but tiny ones
// what a step found
constexpr int kMore = 1;    // some correction is too large to be the last
constexpr int kClose = 2;   // some eigenvalues are too close for the refinement
constexpr int kFailed = 4;  // not a refinement any more

// the largest correction that a step takes
__device__ __forceinline__ double reach(int step) {
  return step < 2 ? 0.125 : step == 2 ? 0.03 : step == 3 ? 2e-3 : kRefined;
}

// One entry of the correction of approximate eigenvectors X of A (Ogita and Aishima, "Iterative
// refinement for symmetric eigenvalue decomposition", 2018): with S = X^T A X, G = X^T X and
// lambda_i = S_ii / G_ii, X (I + E) is better by a square.  A pair whose eigenvalues are too close for the
// first-order step is only made orthogonal, and reported unless its off-diagonal is no more than
// rounding leaves.  What the two entries of a pair get is decided alike: E_ij + E_ji = -G_ij.
// Off-diagonals at the level of rounding (`noise`) are corrected like others in the first two steps,
// but for eigenvalues that rounding cannot tell apart; from then on they are rounding and stay.
// coarse (the first step): off-diagonals this small are still the squares of FP32's errors, and within a
// cluster of equal eigenvalues hundreds of corrections of a tenth would add up (matrices of rank p / 2
// went to the FP64 rotations: 256 columns 26 ms, 2.3 so); above 1e-3 they wait for the next step.
// Later steps take only what converges at least as fast as squares do, the last two only corrections that
// need no further step: the rest, clusters of close eigenvalues, ends as an orthonormal basis that FP64
// rotations start from (they started from the identity: 12 columns in clusters of 1e-6, seeded, 395 us, 285 so;
// 256 columns, four such clusters, 18.4 ms, 9.8 so).
// up, down: column i's noise over j's, and j's over i's.  A correction puts X_i's eigenvalue times its
// square into lambda_j, so it counts that much more where i's eigenvalue is the larger.
__device__ __forceinline__ double correction(int i, int j, double S, double G, double li, double lj, double noise,
                                             float up, float down, int step, bool coarse, int& found) {
  const double num = i == j ? 1.0 - G : fma(-lj, G, S), an = i == j ? fabs(num) : fmax(fabs(num), fabs(fma(-li, G, S)));
  if (!(fabs(num) <= 1e300) || !(an <= 1e300)) {  // not finite
    found |= kFailed;
    return 0.0;
  }
  double e = i == j ? 0.5 * num : -0.5 * G;
  float weight = 1.f;
  if (i != j) {
    const double gap = lj - li, ag = fabs(gap);
    bool turn = ag > 0.0;
    if (an <= noise) {
      if (turn && an * f32_to_f64(fmaxf(1.f, fmaxf(up, down))) <= 1e-9 * ag) return num / gap;
      turn = step < 2 && ag > 64.0 * noise;
    } else if (coarse && an <= kCoarse * noise && an > 1e-3 * ag) {
      found |= kMore;
      turn = false;
    } else if (!turn || !(an <= reach(step) * ag)) {
      found |= kClose;
      turn = false;
    }
    if (turn) {
      e = num / gap;
      weight = fmaxf(1.f, up);
    }
  }
  if (!(fabs(e) <= 0.5))
    found |= kFailed;
  else if (weight * fabsf(scaled32(e, 1023)) > kRefined)
    found |= kMore;
  return e;
}

}  // namespace eig
}  // namespace ss
