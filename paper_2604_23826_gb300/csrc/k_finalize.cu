// k_finalize.cu -- from the sufficient statistics (n, s, S) to mean, covariance, correlation and, up
// to 23 analysis columns or for many contexts at once, the PCA eigenpairs (arxiv 2604.23826: "Data
// Representation and Sufficient Statistics" -- mean, covariance and correlation from the aggregated
// matrices only; "Numerical Considerations" -- cancellation between X^T X and N mu mu^T, and the
// identifier dropped from the analysis; "Principal Component Analysis Results" -- eigenpairs of the
// p x p matrix).
//
// STATS_EXACT: the digit Gram G is recombined into exact integers
//   r_j = sum_a 256^a G[0][(j,a)],  R_jk = sum_{a,b} 256^(a+b) G[(j,a)][(k,b)]
// (values scaled by 2^-shift for real columns) and centred exactly: C_jk = n R_jk - r_j r_k, so no
// cancellation can occur; cov_jk = C_jk 2^-(shift_j + shift_k) / (n (n - 1)) is then rounded.  The
// digit products of one weight are added first, so an entry takes 15 wide additions and not 49.
// FP64 modes: the paper's raw-moment formula (S_jk - s_j s_k / n) / (n - 1) in FP64.
//
// Bound: latency, and FP64 at 2 operations per clock and SM (a division or square root ~570 cycles a
// warp).  Tables of more than 23 columns spread their entries over blocks, one entry per thread; each
// block finds all standard deviations for itself, so no block waits for another.
//
// Eigenpairs: up to 23 columns in this kernel; a single wider context goes to the grid-wide solver
// (k_eigen.cu).  In a batch, contexts of 24..64 columns take a cluster of 1 to 4 blocks each.  Either way FP32 Jacobi in
// shared memory, then the Ogita-Aishima refinement in FP64, with FP64 Jacobi from the refined basis
// where eigenvalues are too close for it (a round of FP64 rotations alone takes 2800 cycles: chains of
// 64-cycle operations); wider ones of a batch FP64 Jacobi.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "eigen.cuh"
#include "kernels.h"

namespace ss {

namespace {

using namespace eig;

constexpr double kNaN = __builtin_nan("");
constexpr int kEigBlockMax = 64;                // eigen-problems one block takes in shared memory
constexpr int kSmallMax = 23, kSmallLd = 25;    // ... within the finalize kernel
static_assert(jacobi32_floats(24) <= 2 * 2 * 24 * kSmallLd, "the FP32 work area lies in two FP64 buffers");

// ------------------------------- 256-bit integers -------------------------------
struct i256 {
  uint64_t w[4];  // two's complement, w[0] least significant
};

__device__ __forceinline__ i256 i256_from(int64_t v) {
  const uint64_t ext = v < 0 ? ~0ull : 0ull;
  return i256{{static_cast<uint64_t>(v), ext, ext, ext}};
}
__device__ __forceinline__ bool i256_neg(const i256& a) { return static_cast<int64_t>(a.w[3]) < 0; }
__device__ __forceinline__ bool i256_zero(const i256& a) { return !(a.w[0] | a.w[1] | a.w[2] | a.w[3]); }

__device__ __forceinline__ i256 i256_add(const i256& a, const i256& b) {
  i256 r;
  uint64_t c = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint64_t s = a.w[i] + b.w[i];
    const uint64_t c1 = s < a.w[i];
    r.w[i] = s + c;
    const uint64_t c2 = r.w[i] < s;
    c = c1 | c2;
  }
  return r;
}
__device__ __forceinline__ i256 i256_negate(const i256& a) {
  i256 r;
#pragma unroll
  for (int i = 0; i < 4; ++i) r.w[i] = ~a.w[i];
  return i256_add(r, i256_from(1));
}
__device__ __forceinline__ i256 i256_sub(const i256& a, const i256& b) { return i256_add(a, i256_negate(b)); }
__device__ __forceinline__ i256 i256_abs(const i256& a) { return i256_neg(a) ? i256_negate(a) : a; }

// a << bits, 0 <= bits < 256
__device__ __forceinline__ i256 i256_shl(const i256& a, int bits) {
  i256 r{{0, 0, 0, 0}};
  const int lw = bits >> 6, b = bits & 63;
  for (int i = 3; i >= 0; --i) {
    const int src = i - lw;
    if (src < 0) continue;
    uint64_t v = a.w[src] << b;
    if (b && src > 0) v |= a.w[src - 1] >> (64 - b);
    r.w[i] = v;
  }
  return r;
}

// |a| * |b| modulo 2^256, unsigned limbs
__device__ __forceinline__ i256 u256_mul(const i256& a, const i256& b) {
  i256 r{{0, 0, 0, 0}};
  for (int i = 0; i < 4; ++i) {
    uint64_t carry = 0;
    for (int j = 0; i + j < 4; ++j) {
      const uint64_t lo = a.w[i] * b.w[j];
      const uint64_t hi = __umul64hi(a.w[i], b.w[j]);
      uint64_t s = r.w[i + j] + lo;
      uint64_t c = s < lo;
      s += carry;
      c += s < carry;
      r.w[i + j] = s;
      carry = hi + c;
    }
  }
  return r;
}
__device__ __forceinline__ i256 i256_mul(const i256& a, const i256& b) {
  const bool neg = i256_neg(a) != i256_neg(b);
  const i256 m = u256_mul(i256_abs(a), i256_abs(b));
  return neg ? i256_negate(m) : m;
}

// Correctly rounded conversion to double (round to nearest even): the top 64
// significant bits with a sticky bit for everything below them.
__device__ double i256_to_double(const i256& a) {
  if (i256_zero(a)) return 0.0;
  const bool neg = i256_neg(a);
  const i256 m = i256_abs(a);
  int top = 3;
  while (top > 0 && m.w[top] == 0) --top;
  const int lz = __clzll(static_cast<long long>(m.w[top]));
  const int msb = top * 64 + 63 - lz;  // index of the highest set bit
  double d;
  if (msb < 64) {
    d = __ull2double_rn(m.w[0]);
  } else {
    const int sh = msb - 63;  // drop sh low bits
    const i256 t = i256{{0, 0, 0, 0}};
    (void)t;
    const int lw = sh >> 6, b = sh & 63;
    uint64_t hi64 = m.w[lw] >> b;
    if (b && lw + 1 < 4) hi64 |= m.w[lw + 1] << (64 - b);
    uint64_t sticky = 0;
    for (int i = 0; i < lw; ++i) sticky |= m.w[i];
    if (b) sticky |= m.w[lw] & ((1ull << b) - 1);
    d = ldexp(__ull2double_rn(hi64 | (sticky ? 1ull : 0ull)), sh);
  }
  return neg ? -d : d;
}

__device__ bool i256_fits_i128(const i256& a, int64_t& lo, int64_t& hi) {
  lo = static_cast<int64_t>(a.w[0]);
  hi = static_cast<int64_t>(a.w[1]);
  const uint64_t ext = hi < 0 ? ~0ull : 0ull;
  return a.w[2] == ext && a.w[3] == ext;
}

// ------------------------------- entries of the results -------------------------------
typedef __int128 i128;

__device__ __forceinline__ i256 widen(i128 v) {
  const uint64_t ext = v < 0 ? ~0ull : 0ull;
  return i256{{static_cast<uint64_t>(v), static_cast<uint64_t>(v >> 64), ext, ext}};
}

// R_jk: |G| < 2^62 (2^46 rows of products below 2^16), eight of them to a weight, weights 256^0 ..
// 256^14: the lower eight weights and the upper seven each fit 128 bits
__device__ i256 cross_product(const long long* G, const FinalPlanCol& cj, const FinalPlanCol& ck) {
  i128 lo = 0, hi = 0;
  for (int c = 0; c <= cj.k + ck.k - 2; ++c) {
    i128 d = 0;
    for (int a = max(0, c - ck.k + 1); a <= min(cj.k - 1, c); ++a) d += G[(cj.off + a) * kDigits + ck.off + c - a];
    if (c < 8)
      lo += d * (static_cast<i128>(1) << (8 * c));
    else
      hi += d * (static_cast<i128>(1) << (8 * (c - 8)));
  }
  return i256_add(widen(lo), i256_shl(widen(hi), 64));
}

// FP64 modes: the column sum, S and covariance entries as returned (shifted sums mapped back:
// s = s' + n c, S = S' + c s'^T + s' c^T + n c c^T)
__device__ __forceinline__ double shifted_sum(const FinalParams& P, int j) { return P.fs[j] + P.fs_lo[j]; }
__device__ __forceinline__ double raw_sum(const FinalParams& P, int j, double n) {
  const double v = shifted_sum(P, j);
  return P.shift ? fma(n, P.shift[j], v) : v;
}
__device__ __forceinline__ double raw_S(const FinalParams& P, int t, int j, int k, double n) {
  const double v = P.fS[t] + P.fS_lo[t];
  if (!P.shift) return v;
  const double cj = P.shift[j], ck = P.shift[k];
  return __dadd_rn(v, fma(n * cj, ck, fma(cj, shifted_sum(P, k), shifted_sum(P, j) * ck)));
}
__device__ __forceinline__ double raw_cov(const FinalParams& P, int t, int j, int k, double n) {
  const double q = __ddiv_rn(__dmul_rn(shifted_sum(P, j), shifted_sum(P, k)), n);
  return __ddiv_rn(__dsub_rn(P.fS[t] + P.fS_lo[t], q), n - 1.0);
}
// cov_jk / (sqrt(cov_jj) sqrt(cov_kk)) from the standard deviations; NaN (given as a negative
// deviation) where a variance is not positive
__device__ __forceinline__ double correlation(double cov, double sa, double sb, bool diagonal) {
  if (sa < 0.0 || sb < 0.0) return kNaN;
  return diagonal ? 1.0 : __ddiv_rn(cov, __dmul_rn(sa, sb));
}
__device__ __forceinline__ double deviation(double var) { return var > 0.0 ? sqrt(var) : -1.0; }

__device__ __forceinline__ int packed_row(int p, int j) { return j * p - j * (j - 1) / 2; }
// (j, k) of packed upper entry t
__device__ __forceinline__ void packed_entry(int t, int p, int& j, int& k) {
  const float b = 2.f * p + 1.f;
  j = max(0, min(p - 1, static_cast<int>((b - sqrtf(b * b - 8.f * t)) * 0.5f)));
  while (packed_row(p, j + 1) <= t) ++j;
  while (packed_row(p, j) > t) --j;
  k = j + t - packed_row(p, j);
}

// analysis index of each table column (-1: identifier); returns the number of analysis columns
__device__ int analysis_index(const FinalParams& P, short* idx) {
  __shared__ int s_cnt[8];
  const int tid = threadIdx.x, lane = tid & 31;
  const bool in = tid < P.p && !P.col[tid].is_ident;
  const unsigned b = __ballot_sync(0xffffffffu, in);
  if (lane == 0) s_cnt[tid >> 5] = __popc(b);
  __syncthreads();
  int before = 0, total = 0;
  for (int w = 0; w < kThreads / 32; ++w) {
    before += w < (tid >> 5) ? s_cnt[w] : 0;
    total += s_cnt[w];
  }
  if (tid < P.p) idx[tid] = in ? static_cast<short>(before + __popc(b & ((1u << lane) - 1))) : -1;
  __syncthreads();
  return total;
}

// eigenvalues lambda, eigenvectors = columns of V (n x n, leading dimension ld), to the results:
// descending (ties by index), the largest-magnitude component of each vector positive
__device__ void put_eigenpairs(const double* lambda, const double* V, int ld, int n, int* order, double* evals,
                               double* evecs) {
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid < n) order[tid] = tid;
  __syncthreads();
  if (tid < n) {
    const unsigned long long k = order_key(lambda[tid]);
    int rank = 0;
    for (int d = 0; d < n; ++d) {
      const unsigned long long o = order_key(lambda[d]);
      rank += (o > k || (o == k && d < tid)) ? 1 : 0;
    }
    order[rank] = tid;
  }
  __syncthreads();
  for (int k = tid >> 5; k < n; k += kThreads / 32) {
    const int col = order[k];
    unsigned long long best = 0;
    int bi = 1 << 20;
    for (int i = lane; i < n; i += 32) {
      const unsigned long long key = magnitude_key(V[i * ld + col]);
      if (bi == 1 << 20 || key > best) {
        best = key;
        bi = i;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ob > best || (ob == best && oi < bi)) {
        best = ob;
        bi = oi;
      }
    }
    const long long flip = __double_as_longlong(V[bi * ld + col]) & (1ll << 63);  // the sign bit
    for (int i = lane; i < n; i += 32)
      evecs[k * n + i] = __longlong_as_double(__double_as_longlong(V[i * ld + col]) ^ flip);
    if (lane == 0) evals[k] = lambda[col];
  }
  __syncthreads();
}

// The blocks that work on one decomposition together: a cluster, or one block alone.  Each holds all
// matrices in its own shared memory; a product's entries are dealt to all of them and put into every
// copy.
struct Team {
  int rank, size;
  __device__ __forceinline__ void put(double* p, double v) const {
    *p = v;
    for (int d = 1; d < size; ++d) {
      uint32_t a;
      const int to = rank + d < size ? rank + d : rank + d - size;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(to));
      asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
    }
  }
  // all of the team's threads, with what they have put
  __device__ __forceinline__ void meet() const {
    if (size > 1)
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else
      __syncthreads();
  }
};
constexpr int kTeamMax = 4;

// Z(i, j) = sum_k X(k, i) Y(k, j) for 2 x 2 tiles shared out over the team's threads (FP64-bound: a
// tile's four multiply-adds take 256 cycles a warp, its loads hide behind them), or, up to kOneByOne
// columns, whose tiles would not fill the SM's four FP64 units, an entry a thread (11 columns:
// 2816 cycles in tiles, 704 so).
constexpr int kOneByOne = 16;
template <class FX, class FY, class Put>
__device__ __forceinline__ void team_product(const Team& team, int n, FX&& X, FY&& Y, Put&& put) {
  if (n <= kOneByOne) {
    const int t = threadIdx.x, i = t / n, j = t % n;
    if (i < n) {
      double z = 0.0;
      for (int k = 0; k < n; ++k) z = fma(X(k, i), Y(k, j), z);
      put(i, j, z);
    }
    return;
  }
  const int nt = (n + 1) / 2;
  for (int t = threadIdx.x + team.rank * kThreads; t < nt * nt; t += team.size * kThreads) {
    const int i0 = 2 * (t / nt), j0 = 2 * (t % nt), i1 = min(i0 + 1, n - 1), j1 = min(j0 + 1, n - 1);
    double z00 = 0.0, z01 = 0.0, z10 = 0.0, z11 = 0.0;
    for (int k = 0; k < n; ++k) {
      const double x0 = X(k, i0), x1 = X(k, i1), y0 = Y(k, j0), y1 = Y(k, j1);
      z00 = fma(x0, y0, z00);
      z01 = fma(x0, y1, z01);
      z10 = fma(x1, y0, z10);
      z11 = fma(x1, y1, z11);
    }
    put(i0, j0, z00);
    if (j1 > j0) put(i0, j1, z01);
    if (i1 > i0) put(i1, j0, z10);
    if (i1 > i0 && j1 > j0) put(i1, j1, z11);
  }
}

struct MixedScratch {
  union {
    Scratch32 s32;
    Scratch64 s64;
  };
  double lambda[kEigBlockMax], noise[kEigBlockMax], gd[kEigBlockMax], red[8];
  float diag[kEigBlockMax], nf[kEigBlockMax], ni[kEigBlockMax];
  double found[kTeamMax];  // what each block found
};

// The order eigen_mixed's FP32 rotations take n columns at: the matrices are laid out by it and the
// rotations compiled for it.
template <bool kSmall>
__host__ __device__ constexpr int mixed_order(int n) {
  return kSmall ? (n + 7) / 8 * 8 : n <= 32 ? 32 : (n + 15) / 16 * 16;
}
constexpr bool orders_exist() {
  for (int n = 1; n <= kEigBlockMax; ++n) {
    const bool small = n <= kSmallMax;
    const int m = small ? mixed_order<true>(n) : mixed_order<false>(n);
    if (m < n || !(small ? m == 8 || m == 16 || m == 24 : m == 32 || m == 48 || m == 64)) return false;
  }
  return true;
}
static_assert(orders_exist(), "eigen_mixed has the rotations of every order");

// Eigenpairs of A (n x n, 1 <= n <= 64, anywhere) in one block: FP32 Jacobi, FP64 refinement, and FP64
// Jacobi from the refined basis where eigenvalues are too close for it (or from A as it is), refined once more.  X, W, S:
// shared memory of leading dimension ld (odd, above n), S right behind W.  The eigenvalues are left in M.lambda, the
// vectors in the columns of X (which may become the buffer S or W was).  Returns the sweeps taken.
// A team shares the refinement (not kSmall); the rotations, and everything decided, all its blocks do
// alike.
// kSmall: at most 23 columns; else at least 24.
template <bool kSmall>
__device__ int eigen_mixed(const double* A, int n, double*& X, double* W, double* S, int ld, MixedScratch& M,
                           const Team& team) {
  const int tid = threadIdx.x, first = tid + team.rank * kThreads, step = team.size * kThreads;
  const Team alone{0, 1};
  double f = 0.0;
  for (int i = tid; i < n * n; i += kThreads) f = fma(A[i], A[i], f);
  const double fro2 = block_total(f, M.red);
  const Variances var = variances(A, n, n, M.diag, reinterpret_cast<int*>(M.red));
  const Noise noise = noise_of(var.E, n);
  int sweeps = 0;
  const bool in_range = fro2 > 1e-280 && fro2 < 1e280;
  if (in_range) {
    const int E = scale_exponent(fro2);
    const int m = mixed_order<kSmall>(n);
    float* fA = reinterpret_cast<float*>(W);  // W and S, one behind the other
    float* fV = fA + 2 * m * m;
    for (int i = tid; i < m * m; i += kThreads) {
      const int r = i / m, c = i % m;
      fA[i] = r < n && c < n ? scaled32(A[r * n + c], E - kUp32) : 0.f;
      fV[i] = r == c ? 1.f : 0.f;
    }
    __syncthreads();
    int copy = 0;
    if constexpr (kSmall) {
      switch (m) {
        case 8: sweeps = jacobi32<8>(fA, fV, 20, floor32(var.least, E), M.s32, copy); break;
        case 16: sweeps = jacobi32<16>(fA, fV, 20, floor32(var.least, E), M.s32, copy); break;
        case 24: sweeps = jacobi32<24>(fA, fV, 20, floor32(var.least, E), M.s32, copy); break;
      }
    } else {
      switch (m) {
        case 32: sweeps = jacobi32<32>(fA, fV, 20, floor32(var.least, E), M.s32, copy); break;
        case 48: sweeps = jacobi32<48>(fA, fV, 20, floor32(var.least, E), M.s32, copy); break;
        case 64: sweeps = jacobi32<64>(fA, fV, 20, floor32(var.least, E), M.s32, copy); break;
      }
    }
    fV += copy * m * m;
    for (int i = tid; i < n * n; i += kThreads) X[(i / n) * ld + i % n] = f32_to_f64(fV[(i / n) * m + i % n]);
  }
  // the refinement; if need be FP64 rotations, and its late steps for what they leave
  int it = 0;
  for (bool rotated = false;; rotated = true) {
    team.meet();  // the others may put into W and S now
    bool refined = false, warm = false;
    for (; in_range && it < kSteps; ++it) {
      team_product(
          team, n, [&](int k, int i) { return A[k * n + i]; }, [&](int k, int j) { return X[k * ld + j]; },
          [&](int i, int j, double v) { team.put(W + i * ld + j, v); });
      team.meet();
      // X^T W on and above the diagonal of S, X^T X below it (its diagonal in gd)
      const bool single = kSmall && n <= kOneByOne;
      const int nt = single ? n : (n + 1) / 2, half = nt * (nt + 1) / 2;
      for (int t = first; t < 2 * half; t += step) {
        const bool gram = t >= half;
        if (single) {
          int i, j;
          packed_entry(gram ? t - half : t, n, i, j);
          const double* Y = gram ? X : W;
          double z = 0.0;
          for (int k = 0; k < n; ++k) z = fma(X[k * ld + i], Y[k * ld + j], z);
          if (!gram)
            S[i * ld + j] = z;
          else if (i == j)
            M.gd[i] = z;
          else
            S[j * ld + i] = z;
          continue;
        }
        int I, Jt;
        packed_entry(gram ? t - half : t, nt, I, Jt);
        const double* Y = gram ? X : W;
        const int i0 = 2 * I, j0 = 2 * Jt, i1 = min(i0 + 1, n - 1), j1 = min(j0 + 1, n - 1);
        double z00 = 0.0, z01 = 0.0, z10 = 0.0, z11 = 0.0;
        for (int k = 0; k < n; ++k) {
          const double x0 = X[k * ld + i0], x1 = X[k * ld + i1], y0 = Y[k * ld + j0], y1 = Y[k * ld + j1];
          z00 = fma(x0, y0, z00);
          z01 = fma(x0, y1, z01);
          z10 = fma(x1, y0, z10);
          z11 = fma(x1, y1, z11);
        }
        auto put = [&](int i, int j, double v) {
          if (i > j) return;
          team.put(!gram ? S + i * ld + j : i == j ? M.gd + i : S + j * ld + i, v);
        };
        put(i0, j0, z00);
        put(i0, j1, z01);
        if (i1 > i0) {
          put(i1, j0, z10);
          put(i1, j1, z11);
        }
      }
      team.meet();
      if (tid < n) {
        const double l = S[tid * ld + tid] / M.gd[tid];
        float w = 0.f;
        for (int k = 0; k < n; ++k) {
          const float x = scaled32(X[k * ld + tid], 1023);
          w = fmaf(M.diag[k] * x, x, w);
        }
        M.lambda[tid] = l;
        M.noise[tid] = noise.column(l, w, M.nf[tid], M.ni[tid]);
      }
      __syncthreads();
      int found = 0;
      for (int i = first; i < n * n; i += step) {
        const int r = i / n, c = i % n, lo = min(r, c), hi = max(r, c);
        const double e = correction(r, c, S[lo * ld + hi], r == c ? M.gd[r] : S[hi * ld + lo], M.lambda[r], M.lambda[c],
                                    M.noise[r] * M.noise[c], M.nf[r] * M.ni[c], M.nf[c] * M.ni[r], it, !kSmall && it == 0,
                                    found);
        team.put(W + r * ld + c, e);
      }
      found = block_or(found, reinterpret_cast<int*>(M.red));
      if (team.size > 1) {
        if (tid == 0) team.put(&M.found[team.rank], __longlong_as_double(found));
        team.meet();
        for (int r = 0; r < team.size; ++r) found |= static_cast<int>(__double_as_longlong(M.found[r]));
      }
      if (found & kFailed) break;
      team_product(
          team, n, [&](int k, int i) { return X[i * ld + k]; }, [&](int k, int j) { return W[k * ld + j]; },
          [&](int i, int j, double v) { team.put(S + i * ld + j, X[i * ld + j] + v); });
      team.meet();
      double* t = X;
      X = S;
      S = t;
      if (!(found & kMore)) {
        refined = !(found & kClose);
        warm = !refined;
        break;
      }
    }
    if (refined || rotated) break;
    if (warm) {  // FP64 Jacobi on X^T A X, from the refined basis
      team_product(
          alone, n, [&](int k, int i) { return A[k * n + i]; }, [&](int k, int j) { return X[k * ld + j]; },
          [&](int i, int j, double v) { W[i * ld + j] = v; });
      __syncthreads();
      team_product(
          alone, n, [&](int k, int i) { return X[k * ld + i]; }, [&](int k, int j) { return W[k * ld + j]; },
          [&](int i, int j, double v) {
            if (i <= j) S[i * ld + j] = S[j * ld + i] = v;
          });
    } else {
      for (int i = tid; i < n * n; i += kThreads) {
        S[(i / n) * ld + i % n] = A[i];
        X[(i / n) * ld + i % n] = i / n == i % n ? 1.0 : 0.0;
      }
    }
    __syncthreads();
    sweeps += jacobi64(S, ld, X, ld, n, M.diag, var.E, M.s64);
    if (tid < n) M.lambda[tid] = S[tid * ld + tid];
    it = kPolish;
  }
  __syncthreads();
  return sweeps;
}

// One context in one block.
__device__ void finalize_body(const FinalParams& P) {
  __shared__ union {
    struct {
      long long G[kDigits * kDigits];
      i128 r[kMaxCols];
    } exact;
    struct {
      double X[24 * kSmallLd], W[24 * kSmallLd], S[24 * kSmallLd];
      MixedScratch scratch;
    } small;
    Scratch64 any;
  } U;
  __shared__ short s_idx[256];
  __shared__ double s_sd[256], s_lambda[256];
  __shared__ float s_diag[256];
  __shared__ int s_order[256];
  __shared__ double s_den;
  __shared__ int s_over;
  const int tid = threadIdx.x, p = P.p, T = p * (p + 1) / 2;
  if (tid == 0) s_over = 0;
  const int pa = analysis_index(P, s_idx);
  const FinalLayout L = final_layout(p, pa);
  double* out = P.out;
  double* flags = out + L.flags;
  double* cov = out + L.cov;
  double* corr = out + L.corr;
  const bool raw = !P.analysis_only;
  long long rows = 0;
  double n_d = 0.0;
  bool nonpositive = false;  // a variance of zero (EXACT) or not above zero

  if (P.mode == 0) {
    for (int i = tid; i < kDigits * kDigits; i += kThreads) {
      const int r = i / kDigits, c = i % kDigits;
      U.exact.G[i] = (r <= c) ? P.g[r * kDigits + c] : P.g[c * kDigits + r];
    }
    __syncthreads();
    const long long* G = U.exact.G;
    const long long n = G[0];
    rows = n;
    n_d = static_cast<double>(n);
    if (tid == 0) {
      if (raw) reinterpret_cast<long long*>(out)[L.n] = n;
      s_den = i256_to_double(i256_mul(i256_from(n), i256_from(n - 1)));
    }
    // exact column sums r_j (scaled by 2^-shift_j)
    if (tid < p) {
      const FinalPlanCol cj = P.col[tid];
      i128 r = 0;
      for (int a = cj.k - 1; a >= 0; --a) r = r * 256 + G[cj.off + a];
      U.exact.r[tid] = r;
      const double s = ldexp(i256_to_double(widen(r)), -cj.shift);
      if (raw) {
        out[L.s + tid] = s;
        reinterpret_cast<int64_t*>(out)[L.s_ex + 2 * tid] = cj.is_real ? 0 : static_cast<int64_t>(r);
        reinterpret_cast<int64_t*>(out)[L.s_ex + 2 * tid + 1] = cj.is_real ? 0 : static_cast<int64_t>(r >> 64);
      }
      if (s_idx[tid] >= 0) out[L.mean + s_idx[tid]] = s / n_d;
    }
    __syncthreads();
    // exact cross products R_jk and, for analysis pairs, the exact centred numerator
    for (int t = tid; t < T; t += kThreads) {
      int j, k;
      packed_entry(t, p, j, k);
      const FinalPlanCol cj = P.col[j], ck = P.col[k];
      const i256 R = cross_product(G, cj, ck);
      int64_t lo = 0, hi = 0;
      if (!cj.is_real && !ck.is_real) {
        if (!i256_fits_i128(R, lo, hi)) atomicOr(&s_over, 1);
      }
      if (raw) {
        out[L.S + t] = ldexp(i256_to_double(R), -(cj.shift + ck.shift));
        reinterpret_cast<int64_t*>(out)[L.S_ex + 2 * t] = lo;
        reinterpret_cast<int64_t*>(out)[L.S_ex + 2 * t + 1] = hi;
      }
      const int aj = s_idx[j], ak = s_idx[k];
      if (aj >= 0 && ak >= 0 && n >= 2) {
        const i256 C = i256_sub(i256_mul(i256_from(n), R), i256_mul(widen(U.exact.r[j]), widen(U.exact.r[k])));
        const double v = ldexp(i256_to_double(C) / s_den, -(cj.shift + ck.shift));
        cov[aj * pa + ak] = v;
        cov[ak * pa + aj] = v;
        if (j == k) {
          s_sd[aj] = deviation(v);
          nonpositive |= v == 0.0;
        }
      }
    }
  } else {
    const long long n = *P.fn;
    rows = n;
    n_d = static_cast<double>(n);
    if (tid == 0 && raw) reinterpret_cast<long long*>(out)[L.n] = n;
    if (tid < p) {
      const double s = raw_sum(P, tid, n_d);
      if (raw) {
        out[L.s + tid] = s;
        reinterpret_cast<int64_t*>(out)[L.s_ex + 2 * tid] = 0;
        reinterpret_cast<int64_t*>(out)[L.s_ex + 2 * tid + 1] = 0;
      }
      if (s_idx[tid] >= 0) out[L.mean + s_idx[tid]] = s / n_d;
    }
    for (int t = tid; t < T; t += kThreads) {
      int j, k;
      packed_entry(t, p, j, k);
      if (raw) {
        out[L.S + t] = raw_S(P, t, j, k, n_d);
        reinterpret_cast<int64_t*>(out)[L.S_ex + 2 * t] = 0;
        reinterpret_cast<int64_t*>(out)[L.S_ex + 2 * t + 1] = 0;
      }
      const int aj = s_idx[j], ak = s_idx[k];
      if (aj >= 0 && ak >= 0 && n >= 2) {
        const double v = raw_cov(P, t, j, k, n_d);
        cov[aj * pa + ak] = v;
        cov[ak * pa + aj] = v;
        if (j == k) {
          s_sd[aj] = deviation(v);
          nonpositive |= !(v > 0.0);
        }
      }
    }
  }
  const int zeros = __syncthreads_count(nonpositive);
  for (int i = tid; n_d >= 2.0 && i < pa * pa; i += kThreads)
    corr[i] = correlation(cov[i], s_sd[i / pa], s_sd[i % pa], i / pa == i % pa);
  const bool pca_ok = P.want_pca && pa > 0 && n_d >= 2.0 && !(P.pca_on == 1 && zeros > 0);
  if (tid == 0) {
    flags[0] = s_over ? 1.0 : 0.0;
    flags[1] = zeros;
    flags[2] = 0.0;
    flags[3] = 0.0;
    flags[5] = 0.0;
    flags[6] = 0.0;
    if (P.status) reinterpret_cast<unsigned long long*>(flags)[4] = *P.status;
    if (P.defer_m < 0) flags[7] = pca_ok ? 1.0 : 0.0;
    if (P.analysis_only) reinterpret_cast<long long*>(flags)[8] = rows;
    if (P.defer_ctl) *P.defer_ctl = pca_ok ? 1 : 0;
  }
  __syncthreads();
  const double* src = P.pca_on ? corr : cov;
  if (!pca_ok) {
    for (int i = tid; i < pa; i += kThreads) out[L.evals + i] = kNaN;
    for (int i = tid; i < pa * pa; i += kThreads) out[L.evecs + i] = kNaN;
  } else if (P.defer_A) {
    // the grid-wide solver takes over: the matrix, zero-padded to order defer_m
    const int m = P.defer_m;
    for (int i = tid; i < m * m; i += kThreads) {
      const int r = i / m, c = i % m;
      P.defer_A[i] = (r < pa && c < pa) ? src[r * pa + c] : 0.0;
    }
  } else if (P.defer_m < 0) {
    // the batched eigen-solver takes over
  } else if (pa <= kSmallMax) {
    double* X = U.small.X;
    const int sweeps = eigen_mixed<true>(src, pa, X, U.small.W, U.small.S, kSmallLd, U.small.scratch,
                                        Team{0, 1});
    put_eigenpairs(U.small.scratch.lambda, X, kSmallLd, pa, s_order, out + L.evals, out + L.evecs);
    if (tid == 0) {
      flags[2] = sweeps;
      flags[3] = 1.0;
    }
  } else {
    double* A = P.work;
    double* V = P.work + static_cast<size_t>(pa) * pa;
    for (int i = tid; i < pa * pa; i += kThreads) {
      A[i] = src[i];
      V[i] = i / pa == i % pa ? 1.0 : 0.0;
    }
    __syncthreads();
    const Variances var = variances(A, pa, pa, s_diag, reinterpret_cast<int*>(U.any.red));
    const int sweeps = jacobi64(A, pa, V, pa, pa, s_diag, var.E, U.any);
    if (tid < pa) s_lambda[tid] = A[tid * pa + tid];
    __syncthreads();
    put_eigenpairs(s_lambda, V, pa, pa, s_order, out + L.evals, out + L.evecs);
    if (tid == 0) {
      flags[2] = sweeps;
      flags[3] = 1.0;
    }
  }
}

}  // namespace

__global__ void __launch_bounds__(kThreads, 1) finalize_kernel(const __grid_constant__ FinalParams P) {
  finalize_body(P);
}

// many contexts at once: block b finalizes Ps[b] (each with its own scratch and output)
__global__ void __launch_bounds__(kThreads, 1) finalize_batched_kernel(const FinalParams* __restrict__ Ps) {
  finalize_body(Ps[blockIdx.x]);
}

// One context of the FP64 modes over a grid, an entry per thread: no eigenpairs, but the matrix
// prepared for the grid-wide solver.
__global__ void __launch_bounds__(kThreads) finalize_wide_kernel(const __grid_constant__ FinalParams P) {
  __shared__ short s_idx[256];
  __shared__ double s_sd[256];
  const int tid = threadIdx.x, p = P.p, T = p * (p + 1) / 2;
  const int pa = analysis_index(P, s_idx);
  const FinalLayout L = final_layout(p, pa);
  double* out = P.out;
  const long long n = *P.fn;
  const double n_d = static_cast<double>(n);
  bool nonpositive = false;
  if (tid < p) {
    const int a = s_idx[tid];
    if (a >= 0 && n >= 2) {
      const double v = raw_cov(P, packed_row(p, tid), tid, tid, n_d);
      s_sd[a] = deviation(v);
      nonpositive = !(v > 0.0);
    }
    if (blockIdx.x == 0) {
      const double s = raw_sum(P, tid, n_d);
      out[L.s + tid] = s;
      reinterpret_cast<int64_t*>(out)[L.s_ex + 2 * tid] = 0;
      reinterpret_cast<int64_t*>(out)[L.s_ex + 2 * tid + 1] = 0;
      if (a >= 0) out[L.mean + a] = s / n_d;
    }
  }
  const int zeros = __syncthreads_count(nonpositive);
  const bool pca_ok = P.want_pca && pa > 0 && n >= 2 && !(P.pca_on == 1 && zeros > 0);
  if (blockIdx.x == 0 && tid == 0) {
    reinterpret_cast<long long*>(out)[L.n] = n;
    double* flags = out + L.flags;
    flags[0] = 0.0;
    flags[1] = zeros;
    flags[2] = 0.0;
    flags[3] = 0.0;
    flags[5] = 0.0;
    flags[6] = 0.0;
    if (P.status) reinterpret_cast<unsigned long long*>(flags)[4] = *P.status;
    if (P.defer_ctl) *P.defer_ctl = pca_ok ? 1 : 0;
  }
  const int gtid = blockIdx.x * kThreads + tid, nthreads = gridDim.x * kThreads, m = P.defer_m;
  for (int t = gtid; t < T; t += nthreads) {
    int j, k;
    packed_entry(t, p, j, k);
    out[L.S + t] = raw_S(P, t, j, k, n_d);
    reinterpret_cast<int64_t*>(out)[L.S_ex + 2 * t] = 0;
    reinterpret_cast<int64_t*>(out)[L.S_ex + 2 * t + 1] = 0;
    const int a = s_idx[j], b = s_idx[k];
    if (a >= 0 && b >= 0 && n >= 2) {
      const double v = raw_cov(P, t, j, k, n_d), r = correlation(v, s_sd[a], s_sd[b], a == b);
      out[L.cov + a * pa + b] = v;
      out[L.cov + b * pa + a] = v;
      out[L.corr + a * pa + b] = r;
      out[L.corr + b * pa + a] = r;
      if (pca_ok && P.defer_A) {
        const double x = P.pca_on ? r : v;
        P.defer_A[a * m + b] = x;
        P.defer_A[b * m + a] = x;
      }
    }
  }
  if (pca_ok && P.defer_A) {
    for (int i = gtid; i < m * m; i += nthreads)
      if (i / m >= pa || i % m >= pa) P.defer_A[i] = 0.0;
  }
  if (!pca_ok) {
    for (int i = gtid; i < pa; i += nthreads) out[L.evals + i] = kNaN;
    for (int i = gtid; i < pa * pa; i += nthreads) out[L.evecs + i] = kNaN;
  }
}

// ------------------------------- eigenpairs of a batch, 24..64 columns -------------------------------
namespace {

constexpr int kBatchMax = kEigBlockMax;
constexpr int kBatchLd = kBatchMax + 1;
constexpr size_t kBatchBytes = 3 * sizeof(double) * kBatchMax * kBatchLd;
static_assert(jacobi32_floats(kBatchMax) <= 2 * 2 * kBatchMax * kBatchLd, "the FP32 work area lies in two FP64 buffers");

}  // namespace

// A job a cluster of 1, 2 or 4 blocks.  Bound: the refinement's FP64 products, 68 us each for 64 columns
// on one SM (two steps of three such), next to 200 us of rotations, which every block of a cluster does
// alike.  126 matrices of 24 to 64 columns: one block each 838 us, two 551; 63 matrices 804 and, four
// each, 447.  (Past two blocks an SM the repeated rotations would cost more than the shared products
// save.)
__global__ void __launch_bounds__(kThreads, 2) eig_batched_kernel(const EigJob* __restrict__ jobs) {
  extern __shared__ __align__(16) double dynd[];
  __shared__ MixedScratch M;
  __shared__ int s_order[256];
  Team team;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(team.rank));
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(team.size));
  const EigJob job = jobs[blockIdx.x / team.size];
  if (job.flags[7] == 0.0) return;  // the finalize kernel found the eigenpairs undefined
  double* X = dynd;
  const int sweeps = eigen_mixed<false>(job.matrix, job.n, X, dynd + kBatchMax * kBatchLd, dynd + 2 * kBatchMax * kBatchLd,
                                        kBatchLd, M, team);
  if (team.rank != 0) return;
  put_eigenpairs(M.lambda, X, kBatchLd, job.n, s_order, job.evals, job.evecs);
  if (threadIdx.x == 0) {
    job.flags[2] = sweeps;
    job.flags[3] = 1.0;
  }
}

bool batched_eigen_deferred(int pa) { return pa > kSmallMax && pa <= kBatchMax; }

cudaError_t launch_finalize_batched(const FinalParams* d_params, int count, const EigJob* d_jobs, int njobs,
                                    cudaStream_t stream) {
  if (count <= 0) return cudaSuccess;
  finalize_batched_kernel<<<count, kThreads, 0, stream>>>(d_params);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || njobs <= 0) return e;
  e = cudaFuncSetAttribute(eig_batched_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kBatchBytes));
  if (e != cudaSuccess) return e;
  // as many blocks a job as still run side by side, two on an SM
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int size = 4 * njobs <= 2 * sms ? 4 : 2 * njobs <= 2 * sms ? 2 : 1;
  cudaLaunchAttribute cluster{};
  cluster.id = cudaLaunchAttributeClusterDimension;
  cluster.val.clusterDim.x = size;
  cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(njobs * size);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kBatchBytes;
  cfg.stream = stream;
  cfg.attrs = &cluster;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, eig_batched_kernel, d_jobs);
}

cudaError_t launch_finalize(const FinalParams& P, cudaStream_t stream) {
  // one block holds a wider table's entries too, but takes up to a millisecond over them
  if (P.mode != 0 && P.p > kSmallMax && (P.defer_A || !P.want_pca)) {
    const int blocks = (P.p * (P.p + 1) / 2 + kThreads - 1) / kThreads;  // 129 at most
    finalize_wide_kernel<<<blocks, kThreads, 0, stream>>>(P);
  } else {
    finalize_kernel<<<1, kThreads, 0, stream>>>(P);
  }
  return cudaGetLastError();
}

}  // namespace ss
