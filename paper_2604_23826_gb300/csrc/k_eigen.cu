// k_eigen.cu -- the eigen-solver spread over the GPU (arxiv 2604.23826, "Principal Component
// Analysis Results"), for 24 or more analysis columns or with a seed: a cooperative grid, one
// 256-thread block per SM at most, whose blocks meet at bounded grid-wide barriers.
//
//   1. (seed) accepted only if its columns are orthonormal to 1e-9; T = V^T A V.  Cold: T = A, V = I.
//   2. FP32 Jacobi on T scaled to order one: up to 64 columns in one block's shared memory, above
//      that block-cyclic over the grid: pairs of 16-column blocks, a 32 x 32 problem each, and every
//      32 x 32 block of T and V multiplied by the pairs' rotations: one grid barrier a block round.
//   3. X = V Q, then the Ogita-Aishima refinement in FP64: W = A X, S = X^T W, G = X^T X, the
//      correction E from S, G and X <- X + X E, until E is below 5e-9 (its square is left): two or
//      three steps of four products, each spread over the grid in 16 x 16 tiles.  What is rounding is
//      told from each pair's own columns, so the eigenpairs of columns of very different units are
//      as good as those of like ones.
//   4. If eigenvalues are too close for the refinement (or it fails), block-cyclic Jacobi in FP64,
//      from the refined basis (or from the matrix as it came), and the refinement's late steps.
// Bound: latency.  A block round of step 2 takes 18,000 cycles: 17 dependent rounds of its 32 x 32
// problems 10,400, their loads, the product, and the stores and barrier the rest.  Step 3 is FP64 at 2
// operations per clock and SM: 256 columns, 0.13 ms a step.  (FP64 rotations alone, chains of divisions
// and square roots of one warp: 256 columns, 11 sweeps, 14.7 ms; all of this 1.65.)
#include <math.h>

#include "common.cuh"
#include "eigen.cuh"
#include "kernels.h"

namespace ss {

namespace {

using namespace eig;

constexpr int kJW = 8;         // FP64 block Jacobi: indices per block
constexpr int kJP = 2 * kJW;   // order of a block pair's diagonal problem
static_assert(kJP * kJP == kThreads, "one thread per entry of a block-pair tile");
constexpr int kFW = 16, kFP = 2 * kFW;  // the same for the FP32 block Jacobi
constexpr unsigned long long kGridWaitNs = 2000000000ull;  // a grid-wide wait gives up after 2 s
constexpr unsigned int kDead = 0x80000000u;

__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int* a) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

struct Grid {
  unsigned int* bar;  // arrivals since the launch; bit 31: a wait has run out
  unsigned int target;
  unsigned long long wait_ns;
  int* s_ok;

  // Grid-wide barrier of a cooperative launch.  Thread 0 of each block publishes the block's writes
  // (fence) and arrives on a count that only grows; the others' arrivals are polled for.  A wait that
  // outlasts wait_ns marks the count; every block that sees the mark leaves (false).
  __device__ bool sync() {
    __syncthreads();
    if (threadIdx.x == 0) {
      target += gridDim.x;
      __threadfence();
      unsigned int v = atomicAdd(bar, 1u) + 1u;
      if (v < target) {
        const unsigned long long t0 = global_ns();
        for (unsigned int n = 1;; ++n) {
          v = ld_acquire_u32(bar);
          if (v >= target) break;  // everyone is here, or the mark is set
          if ((n & 63u) == 0 && global_ns() - t0 > wait_ns) {
            v = atomicOr(bar, kDead) | kDead;
            break;
          }
        }
      }
      __threadfence();
      *s_ok = (v & kDead) == 0;
    }
    __syncthreads();
    return *s_ok != 0;
  }
};

struct Shared {
  Scratch32 s32;
  double x[16][17], y[16][17], z[16][17], t[16][17];
  double qa[kJP][kJP + 1], qb[kJP][kJP + 1];
  double c[8], s[8];
  int null[8];
  double lambda[256], noise[256];
  float nf[256], ni[256], diag[256];
  int weight[256];
  double red[8];
  unsigned long long key[256];
  int order[256];
  unsigned long long best[8];
  int best_i[8];
  double val;
  int ok;
};
constexpr size_t kDynFloats32 = jacobi32_floats(k32Max);  // step 2 in one block
constexpr size_t kDynFloatsF = 2 * jacobi32_floats(kFP) + 2 * kFP * kFP;  // step 2 over the grid
constexpr size_t kDynBytes = sizeof(float) * (kDynFloats32 > kDynFloatsF ? kDynFloats32 : kDynFloatsF);

// Z(i, j) = sum_k X(i, k) Y(k, j) for 16 x 16 tiles shared out over the grid; X, Y: element
// functions, put(i, j, value)
template <class FX, class FY, class Put>
__device__ void grid_product(int m, Shared& S, FX&& X, FY&& Y, Put&& put) {
  const int nt = m / 16, r = threadIdx.x / 16, c = threadIdx.x % 16;
  for (int t = blockIdx.x; t < nt * nt; t += gridDim.x) {
    const int i0 = (t / nt) * 16, j0 = (t % nt) * 16;
    double acc = 0.0;
    double nx = X(i0 + r, c), ny = Y(r, j0 + c);
    for (int k0 = 0; k0 < m; k0 += 16) {
      S.x[r][c] = nx;
      S.y[r][c] = ny;
      __syncthreads();
      if (k0 + 16 < m) {
        nx = X(i0 + r, k0 + 16 + c);
        ny = Y(k0 + 16 + r, j0 + c);
      }
#pragma unroll
      for (int k = 0; k < 16; ++k) acc = fma(S.x[r][k], S.y[k][c], acc);
      __syncthreads();
    }
    put(i0 + r, j0 + c, acc);
  }
}

// S = X^T W and G = X^T X (both symmetric): the tiles on or above the diagonal of each, shared out
// over the grid; and the columns' weights sum_l a_ll x_lj^2 (FP32, beside G's diagonal tiles)
__device__ void grid_grams(int m, Shared& S, const double* X, const double* W, double* SO, double* GO, const double* A,
                           int E, float* weights) {
  const int nt = m / 16, r = threadIdx.x / 16, c = threadIdx.x % 16, half = nt * (nt + 1) / 2;
  for (int t = blockIdx.x; t < 2 * half; t += gridDim.x) {
    int I = 0, J = t % half;
    while (J >= nt - I) {
      J -= nt - I;
      ++I;
    }
    J += I;
    const double* Y = t < half ? W : X;
    double* O = t < half ? SO : GO;
    const bool weigh = t >= half && I == J;
    double acc = 0.0;
    float b = 0.f;
    double nx = __ldcg(X + static_cast<size_t>(r) * m + I * 16 + c), ny = __ldcg(Y + static_cast<size_t>(r) * m + J * 16 + c);
    double nd = weigh ? __ldcg(A + static_cast<size_t>(r) * (m + 1)) : 0.0;
    for (int k0 = 0; k0 < m; k0 += 16) {
      S.x[r][c] = nx;
      S.y[r][c] = ny;
      if (weigh) {  // this thread's row of column c
        const float x = scaled32(nx, 1023);
        b = fmaf(fabsf(scaled32(nd, E)) * x, x, b);
      }
      __syncthreads();
      if (k0 + 16 < m) {
        nx = __ldcg(X + static_cast<size_t>(k0 + 16 + r) * m + I * 16 + c);
        ny = __ldcg(Y + static_cast<size_t>(k0 + 16 + r) * m + J * 16 + c);
        if (weigh) nd = __ldcg(A + static_cast<size_t>(k0 + 16 + r) * (m + 1));
      }
#pragma unroll
      for (int k = 0; k < 16; ++k) acc = fma(S.x[k][r], S.y[k][c], acc);
      __syncthreads();
    }
    if (weigh) {
      S.t[r][c] = b;
      __syncthreads();
      if (threadIdx.x < 16) {
        float w = 0.f;
        for (int k = 0; k < 16; ++k) w += static_cast<float>(S.t[k][threadIdx.x]);
        __stcg(weights + I * 16 + threadIdx.x, w);
      }
    }
    // both halves hold the same value
    if (I == J) {
      S.z[r][c] = acc;
      __syncthreads();
      acc = r <= c ? acc : S.z[c][r];
      __stcg(O + static_cast<size_t>(I * 16 + r) * m + J * 16 + c, acc);
      __syncthreads();
    } else {
      __stcg(O + static_cast<size_t>(I * 16 + r) * m + J * 16 + c, acc);
      __stcg(O + static_cast<size_t>(J * 16 + c) * m + I * 16 + r, acc);
    }
  }
}

// the blocks' slots[0 .. grid) added (or their maximum taken) in a fixed order, in every thread
template <typename T>
__device__ T slots_total(const T* slots, Shared& S) {
  T v = 0;
  for (int b = threadIdx.x; b < static_cast<int>(gridDim.x); b += kThreads) v += __ldcg(slots + b);
  return block_total(v, reinterpret_cast<T*>(S.red));
}
__device__ double slots_max(const double* slots, Shared& S) {
  double v = 0.0;
  for (int b = threadIdx.x; b < static_cast<int>(gridDim.x); b += kThreads) v = fmax(v, __ldcg(slots + b));
  return block_max(v, S.red);
}
__device__ int slots_or(const double* slots, Shared& S) {
  int v = 0;
  for (int b = threadIdx.x; b < static_cast<int>(gridDim.x); b += kThreads) v |= __ldcg(reinterpret_cast<const int*>(slots + b));
  return block_or(v, reinterpret_cast<int*>(S.red));
}

// FP32 block-cyclic Jacobi over the grid (m a multiple of 32): A and its next copy B, V = I on entry.
// A sweep meets every two indices once: those of a block in its first round, with the rest of the
// pair's 32 x 32 problem, the two blocks' with one another in every round.
// An item of a round is one 32 x 32 block of A off the pairs' diagonal (and its transpose) or one of V.
// Its block of threads solves the two pairs' problems itself, half a block each: the same bits
// everywhere, and a grid barrier and a trip through memory less than solving them once.  (256 columns,
// all of the solver: 2.44 ms with full sweeps of problems solved once and two barriers a round, 1.64 so.)
// Returns the sweeps, -1 after a wait that ran out.
__device__ int grid_jacobi32(const JacobiParams& J, Grid& grid, Shared& S, float* dyn, float* A, float* B, float* V,
                             int floor) {
  const int m = J.m, nb = m / kFW, np = nb / 2, tid = threadIdx.x;
  constexpr int kE = kFP * kFP;
  float* sX = dyn + 2 * jacobi32_floats(kFP);
  float* sT = sX + kE;
  auto row_of = [](int bi, int bj, int l) { return l < kFW ? bi * kFW + l : bj * kFW + l - kFW; };
  const int nthreads = gridDim.x * kThreads, gtid = blockIdx.x * kThreads + tid;
  const int half = tid / (kThreads / 2), ht = tid % (kThreads / 2);
  float* pA = dyn + half * jacobi32_floats(kFP);  // this half's problem: two copies, then the rotations' two
  float* pV = pA + 2 * kE;
  double fro2 = 0.0, prev = 0.0;
  float prev_rel = 0.f;
  int sweep = 0;
  for (; sweep < 20; ++sweep) {
    float o = 0.f, d = 0.f, q = 0.f;
    for (int i = gtid; i < m * m; i += nthreads) {
      const float x = __ldcg(A + i);
      const int r = i / m, c = i % m;
      if (r != c) {
        o = fmaf(x, x, o);
        q += square_ratio(exp_field32(x), exp_field32(__ldcg(A + r * (m + 1))), exp_field32(__ldcg(A + c * (m + 1))), floor,
                          floor);
      } else {
        d = fmaf(x, x, d);
      }
    }
    const double bo = block_total(static_cast<double>(o), S.red), bd = block_total(static_cast<double>(d), S.red);
    const float bq = block_total(q, reinterpret_cast<float*>(S.red));
    if (tid == 0) {
      __stcg(J.slots + blockIdx.x, bo);
      __stcg(reinterpret_cast<float*>(J.slots + 256) + blockIdx.x, bq);
      __stcg(J.slots + 512 + blockIdx.x, bd);
    }
    if (!grid.sync()) return -1;
    const double off = slots_total(J.slots, S);
    const float rel = slots_total(reinterpret_cast<const float*>(J.slots + 256), S);
    if (sweep == 0) fro2 = off + slots_total(J.slots + 512, S);
    if (rotated32(sweep, off, prev, fro2, 1e-12, rel, prev_rel)) break;
    prev = off;
    prev_rel = rel;
    for (int br = 0; br < nb - 1; ++br) {
      const int copy = br == 0 ? 1 : 0;  // where the problems' results lie: 31 rounds, then 16 each
      const int nA = np * (np - 1) / 2, nItems = nA + np * np;
      for (int it = blockIdx.x; it < nItems; it += gridDim.x) {
        const bool isA = it < nA;
        int P1 = 0, P2, bi = 0, bj = 0, ci, cj;
        if (isA) {
          P2 = it;
          while (P2 >= np - 1 - P1) {
            P2 -= np - 1 - P1;
            ++P1;
          }
          P2 += P1 + 1;
          pair_of(br, P1, nb, bi, bj);
        } else {
          P1 = (it - nA) / np;  // strip of V
          P2 = (it - nA) % np;
        }
        pair_of(br, P2, nb, ci, cj);
        const bool solves = isA || half == 1;
        if (solves) {
          const int di = half ? ci : bi, dj = half ? cj : bj;
          float x[kE / (kThreads / 2)];
#pragma unroll
          for (int u = 0; u < kE / (kThreads / 2); ++u) {
            const int e = ht + u * (kThreads / 2), r = e / kFP, c = e % kFP;
            x[u] = __ldcg(A + static_cast<size_t>(row_of(di, dj, r)) * m + row_of(di, dj, c));
          }
#pragma unroll
          for (int u = 0; u < kE / (kThreads / 2); ++u) {
            const int e = ht + u * (kThreads / 2);
            pA[e] = x[u];
            pV[e] = e / kFP == e % kFP ? 1.f : 0.f;
          }
        }
        {
          float x[kE / kThreads];
#pragma unroll
          for (int u = 0; u < kE / kThreads; ++u) {
            const int e = tid + u * kThreads, r = e / kFP, c = e % kFP;
            const int gr = isA ? row_of(bi, bj, r) : P1 * kFP + r;
            x[u] = __ldcg((isA ? A : V) + static_cast<size_t>(gr) * m + row_of(ci, cj, c));
          }
#pragma unroll
          for (int u = 0; u < kE / kThreads; ++u) sX[tid + u * kThreads] = x[u];
        }
        __syncthreads();
        if (solves) {  // (the halves are whole warps, and meet at barriers of their own)
          if (br == 0) {
            const Jacobi32<kFP, kThreads / 2, false> K(pA, pV, S.s32, ht, 1 + half);
            K.template sweep<0>(K);
          } else {
            const Jacobi32<kFP, kThreads / 2, true> K(pA, pV, S.s32, ht, 1 + half);
            K.template sweep<0>(K);
          }
        }
        __syncthreads();
        const float* Q1 = dyn + 2 * kE + copy * kE;
        const float* Q2 = Q1 + jacobi32_floats(kFP);
        if (!isA && P1 == 0) {  // the pair's own problem, once
          const float* D = dyn + jacobi32_floats(kFP) + copy * kE;
#pragma unroll
          for (int u = 0; u < kE / kThreads; ++u) {
            const int e = tid + u * kThreads, r = e / kFP, c = e % kFP;
            __stcg(B + static_cast<size_t>(row_of(ci, cj, r)) * m + row_of(ci, cj, c), D[e]);
          }
        }
        const int tr = (tid / 16) * 2, tc = (tid % 16) * 2;
        const float* L = sX;
        if (isA) {  // T = Q1^T X
          float t00 = 0.f, t01 = 0.f, t10 = 0.f, t11 = 0.f;
#pragma unroll 8
          for (int k = 0; k < kFP; ++k) {
            const float2 x = *reinterpret_cast<const float2*>(Q1 + k * kFP + tr);
            const float2 y = *reinterpret_cast<const float2*>(sX + k * kFP + tc);
            t00 = fmaf(x.x, y.x, t00);
            t01 = fmaf(x.x, y.y, t01);
            t10 = fmaf(x.y, y.x, t10);
            t11 = fmaf(x.y, y.y, t11);
          }
          *reinterpret_cast<float2*>(sT + tr * kFP + tc) = make_float2(t00, t01);
          *reinterpret_cast<float2*>(sT + (tr + 1) * kFP + tc) = make_float2(t10, t11);
          __syncthreads();
          L = sT;
        }
        float y[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll 2
        for (int k = 0; k < kFP; k += 4) {
          const float4 a = *reinterpret_cast<const float4*>(L + tr * kFP + k);
          const float4 b = *reinterpret_cast<const float4*>(L + (tr + 1) * kFP + k);
          const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float2 q = *reinterpret_cast<const float2*>(Q2 + (k + u) * kFP + tc);
            y[0][0] = fmaf(av[u], q.x, y[0][0]);
            y[0][1] = fmaf(av[u], q.y, y[0][1]);
            y[1][0] = fmaf(bv[u], q.x, y[1][0]);
            y[1][1] = fmaf(bv[u], q.y, y[1][1]);
          }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            const int gc = row_of(ci, cj, tc + v);
            if (isA) {
              const int gr = row_of(bi, bj, tr + u);
              __stcg(B + static_cast<size_t>(gr) * m + gc, y[u][v]);
              __stcg(B + static_cast<size_t>(gc) * m + gr, y[u][v]);
            } else {
              __stcg(V + static_cast<size_t>(P1 * kFP + tr + u) * m + gc, y[u][v]);
            }
          }
        __syncthreads();
      }
      float* t = A;
      A = B;
      B = t;
      if (!grid.sync()) return -1;
    }
  }
  return sweep;
}

// FP64 block-cyclic Jacobi over the grid: diagonalises A (B: its next copy), rotating V's columns.
// Only the first n rows and columns take part, the matrix's own rounded up to a pair of blocks.
// Returns the sweeps (A then points to the diagonal form), -1 after a wait that ran out.
// Bound: the chains of the local rounds.  Angles from FP32 (rotation64) instead of an FP64 division and
// two roots, and 112 rows instead of 128 for 100 columns: a matrix of 100 columns in four clusters of
// eigenvalues 8.3 ms from the identity, 5.4 so (and 3.1 from the refined basis).
// E: of variances(), whose diagonal is in S.
__device__ int grid_jacobi64(const JacobiParams& J, Grid& grid, Shared& S, double*& A, double* B, double* V, int E) {
  const int tid = threadIdx.x, m = J.m, n = (J.pa + kJP - 1) / kJP * kJP, nb = n / kJW, np = nb / 2;
  const int lr_ = tid / kJP, lc_ = tid % kJP;
  const int nthreads = gridDim.x * kThreads, gtid = blockIdx.x * kThreads + tid;
  double fro2 = 0.0, prev = 0.0;
  Ratios64 ratios;
  int sweep = 0, stalled = 0;
  auto at = [m](int r, int c) { return static_cast<size_t>(r) * m + c; };
  float* weights = reinterpret_cast<float*>(J.slots + 384);
  auto weigh = [&] {  // V's columns, shared out over the grid
    for (int j = blockIdx.x; j < n; j += gridDim.x) {
      const float x = tid < J.pa ? scaled32(__ldcg(V + at(tid, j)), 1023) : 0.f;
      const float w = block_total(tid < J.pa ? S.diag[tid] * x * x : 0.f, reinterpret_cast<float*>(S.red));
      if (tid == 0) __stcg(weights + j, w);
    }
  };
  weigh();
  if (!grid.sync()) return -1;
  for (; sweep < 60; ++sweep) {
    if (tid < n) S.weight[tid] = weight_exponent(__ldcg(weights + tid), E);
    __syncthreads();
    double o = 0.0, d = 0.0;
    float q = 0.f;
    for (int i = gtid; i < n * n; i += nthreads) {
      const int r = i / n, c = i % n;
      const double x = __ldcg(A + at(r, c));
      if (r != c) {
        o = fma(x, x, o);
        q += square_ratio(exp_field(x), exp_field(__ldcg(A + at(r, r))), exp_field(__ldcg(A + at(c, c))), S.weight[r],
                          S.weight[c]);
      } else {
        d = fma(x, x, d);
      }
    }
    const double bo = block_total(o, S.red), bd = block_total(d, S.red);
    const float bq = block_total(q, reinterpret_cast<float*>(S.red));
    if (tid == 0) {
      __stcg(J.slots + blockIdx.x, bo);
      __stcg(reinterpret_cast<float*>(J.slots + 256) + blockIdx.x, bq);
      __stcg(J.slots + 512 + blockIdx.x, bd);
    }
    if (!grid.sync()) return -1;
    const double off = slots_total(J.slots, S);
    const float rel = slots_total(reinterpret_cast<const float*>(J.slots + 256), S);
    if (sweep == 0) fro2 = off + slots_total(J.slots + 512, S);
    // converged: off-diagonal mass negligible, or (block updates leave rounding noise in every
    // off-diagonal entry) no longer falling quadratically, at once at the level of rounding (2e-15 an
    // entry), in four sweeps below 1e-26 of ||A||^2; and the same in the pairs' own units
    stalled = sweep > 0 && off > 0.0625 * prev ? stalled + 1 : 0;
    const bool norm = off <= 1e-34 * fro2 || (stalled >= 1 && off <= 4e-30 * n * fro2) || (stalled >= 4 && off <= 1e-26 * fro2);
    if (off == 0.0 || ratios.done(norm, rel, n)) break;
    prev = off;
    weigh();  // for the next sweep's test, whose barriers are to come
    for (int br = 0; br < nb - 1; ++br) {
      // (1) every block pair's kJP x kJP diagonal problem: one cyclic Jacobi sweep in shared
      //     memory, its rotations accumulated in Q (to J.q), its result written to B
      for (int P = blockIdx.x; P < np; P += gridDim.x) {
        int bi, bj;
        pair_of(br, P, nb, bi, bj);
        const int gr = lr_ < kJW ? bi * kJW + lr_ : bj * kJW + lr_ - kJW;
        const int gc = lc_ < kJW ? bi * kJW + lc_ : bj * kJW + lc_ - kJW;
        // both halves alike: what rounding makes of their difference no rotation would take away
        S.x[lr_][lc_] = 0.5 * (__ldcg(A + at(gr, gc)) + __ldcg(A + at(gc, gr)));
        S.y[lr_][lc_] = lr_ == lc_ ? 1.0 : 0.0;
        __syncthreads();
        for (int lr = 0; lr < kJP - 1; ++lr) {
          if (tid < kJP / 2) {
            int p, q;
            pair_of(lr, tid, kJP, p, q);
            double c, sn;
            bool null;
            rotation64(S.x[p][p], S.x[q][q], S.x[p][q], c, sn, null);
            S.c[tid] = c;
            S.s[tid] = sn;
            S.null[tid] = null;
          }
          __syncthreads();
          if (tid < (kJP / 2) * kJP) {  // rows p, q
            const int i = tid / kJP, k = tid % kJP;
            int p, q;
            pair_of(lr, i, kJP, p, q);
            const double c = S.c[i], sn = S.s[i];
            if (sn != 0.0) {
              const double apk = S.x[p][k], aqk = S.x[q][k];
              S.x[p][k] = c * apk - sn * aqk;
              S.x[q][k] = sn * apk + c * aqk;
            }
          }
          __syncthreads();
          {  // columns p, q of the problem (first half of the threads) and of Q (second half)
            const int u = tid % ((kJP / 2) * kJP);
            const int i = u / kJP, k = u % kJP;
            int p, q;
            pair_of(lr, i, kJP, p, q);
            const double c = S.c[i], sn = S.s[i];
            const bool onS = tid < (kJP / 2) * kJP;
            double(*X)[kJP + 1] = onS ? S.x : S.y;
            if (sn != 0.0) {
              const double xkp = X[k][p], xkq = X[k][q];
              // what is left of the rotated pair's off-diagonal entries may be zero
              const bool zero = onS && S.null[i];
              X[k][p] = (zero && k == q) ? 0.0 : c * xkp - sn * xkq;
              X[k][q] = (zero && k == p) ? 0.0 : sn * xkp + c * xkq;
            }
          }
          __syncthreads();
        }
        __stcg(J.q + static_cast<size_t>(P) * kJP * kJP + tid, S.y[lr_][lc_]);
        __stcg(B + static_cast<size_t>(gr) * m + gc, S.x[lr_][lc_]);
        __syncthreads();
      }
      if (!grid.sync()) return -1;
      // (2) the other blocks of A, Q_P^T A[P rows][P' cols] Q_P' (into B), and V's columns,
      //     V[rows][P' cols] Q_P' (in place: every entry belongs to one item)
      const int nA = np * np, nItems = nA + (n / kJP) * np;
      for (int it = blockIdx.x; it < nItems; it += gridDim.x) {
        if (it < nA && it / np == it % np) continue;  // diagonal blocks came from step (1)
        const bool isA = it < nA;
        const int P2 = isA ? it % np : (it - nA) % np;
        int ci, cj;
        pair_of(br, P2, nb, ci, cj);
        const int gc = lc_ < kJW ? ci * kJW + lc_ : cj * kJW + lc_ - kJW;
        int gr;
        if (isA) {
          int bi, bj;
          pair_of(br, it / np, nb, bi, bj);
          gr = lr_ < kJW ? bi * kJW + lr_ : bj * kJW + lr_ - kJW;
          S.x[lr_][lc_] = __ldcg(A + static_cast<size_t>(gr) * m + gc);
          S.qa[lr_][lc_] = __ldcg(J.q + static_cast<size_t>(it / np) * kJP * kJP + tid);
        } else {
          gr = ((it - nA) / np) * kJP + lr_;
          S.x[lr_][lc_] = __ldcg(V + static_cast<size_t>(gr) * m + gc);
        }
        S.qb[lr_][lc_] = __ldcg(J.q + static_cast<size_t>(P2) * kJP * kJP + tid);
        __syncthreads();
        if (isA) {
          double t = 0.0;
#pragma unroll
          for (int k = 0; k < kJP; ++k) t = fma(S.qa[k][lr_], S.x[k][lc_], t);
          S.t[lr_][lc_] = t;
          __syncthreads();
        }
        double(*L)[kJP + 1] = isA ? S.t : S.x;
        double y = 0.0;
#pragma unroll
        for (int k = 0; k < kJP; ++k) y = fma(L[lr_][k], S.qb[k][lc_], y);
        __stcg((isA ? B : V) + static_cast<size_t>(gr) * m + gc, y);
        __syncthreads();
      }
      double* t = A;
      A = B;
      B = t;
      if (!grid.sync()) return -1;
    }
  }
  return sweep;
}

}  // namespace

// a, b, v, w, g, x: m x m (a stays the matrix); the FP64 rotations (a quarter of that is the FP32 ones'); the
// seed; slots
size_t jacobi_scratch_doubles(int pa) {
  const size_t m = jacobi_order(pa);
  return 6 * m * m + static_cast<size_t>(pa) * pa + (m / kJP) * kJP * kJP + 1024 + 8;
}

int jacobi_grid_blocks(int pa, int sms) {
  const int np = jacobi_order(pa) / kJP;
  int g = 2 * np * np;
  if (g > sms) g = sms;
  if (g > 256) g = 256;  // three partial sums per block, at 0, 256 and 512 of the 1024 slots
  return g < 1 ? 1 : g;
}

__global__ void __launch_bounds__(kThreads, 1) jacobi_grid_kernel(const __grid_constant__ JacobiParams J) {
  extern __shared__ __align__(16) float dyn[];
  __shared__ Shared S;
  if (__ldcg(J.ctl) == 0) return;  // the finalize kernel found the eigenpairs undefined
  const int tid = threadIdx.x, pa = J.pa, m = J.m;
  const int nthreads = gridDim.x * kThreads, gtid = blockIdx.x * kThreads + tid;
  Grid grid{J.bar, 0u, J.wait_ns > 0 ? static_cast<unsigned long long>(J.wait_ns) : kGridWaitNs, &S.ok};
  double* flags = J.out + J.flags_off;
  double* A = J.a;
  double* V = J.v;
  const double* T = J.a;  // what step 2 diagonalises
  bool seeded = false;
  int sweeps = 0;
  // a block told to be absent leaves before its first arrival: the other blocks' waits at that
  // barrier run out after wait_ns and the call reports the timeout (the failure path of a stalled
  // block, taken without a fault)
  bool alive = static_cast<int>(blockIdx.x) != J.absent_block;
  auto at = [m](int i, int j) { return static_cast<size_t>(i) * m + j; };

  // ||A||_F^2, and the seed into V
  if (alive) {
    double f = 0.0;
    for (int i = gtid; i < m * m; i += nthreads) {
      const double x = __ldcg(A + i);
      f = fma(x, x, f);
      if (J.basis) {
        const int r = i / m, c = i % m;
        __stcg(V + i, r < pa && c < pa ? J.basis[static_cast<size_t>(c) * pa + r] : r == c ? 1.0 : 0.0);
      }
    }
    f = block_total(f, S.red);
    if (tid == 0) __stcg(J.slots + blockIdx.x, f);
    alive = grid.sync();
  }
  const double fro2 = alive ? slots_total<double>(J.slots, S) : 0.0;
  const Variances var = variances(A, m, pa, S.diag, reinterpret_cast<int*>(S.red));
  if (alive && J.basis) {
    // the seed is used only if its columns are orthonormal: max |V^T V - I| <= 1e-9
    double dev = 0.0;
    grid_product(
        m, S, [&](int i, int k) { return __ldcg(V + at(k, i)); }, [&](int k, int j) { return __ldcg(V + at(k, j)); },
        [&](int i, int j, double v) {
          const double x = fabs(v - (i == j ? 1.0 : 0.0));
          dev = fmax(dev, x == x ? x : 1.0);
        });
    dev = block_max(dev, S.red);
    if (tid == 0) __stcg(J.slots + 512 + blockIdx.x, dev);
    alive = grid.sync();
    seeded = alive && slots_max(J.slots + 512, S) <= 1e-9;
    if (seeded) {  // T = V^T A V
      grid_product(
          m, S, [&](int i, int k) { return __ldcg(A + at(i, k)); }, [&](int k, int j) { return __ldcg(V + at(k, j)); },
          [&](int i, int j, double v) { __stcg(J.w + at(i, j), v); });
      alive = grid.sync();
      if (alive)
        grid_product(
            m, S, [&](int i, int k) { return __ldcg(V + at(k, i)); }, [&](int k, int j) { return __ldcg(J.w + at(k, j)); },
            [&](int i, int j, double v) { __stcg(J.b + at(i, j), v); });
      alive = alive && grid.sync();
      T = J.b;
    }
  }

  double* X = J.w;
  double* Xn = V;
  double* W = J.x;  // A X, then the corrections
  // FP32 has to hold the matrix scaled to order one, FP64 the squares of its entries
  const bool in_range = fro2 > 1e-280 && fro2 < 1e280;
  if (alive && in_range) {
    const int E = scale_exponent(fro2);
    float* F = reinterpret_cast<float*>(J.g);  // two m x m FP32 matrices
    float* Q32 = reinterpret_cast<float*>(J.x);  // V of step 2
    auto t32 = [&](int r, int c) {
      if (T == J.a) return scaled32(__ldcg(T + at(r, c)), E - kUp32);
      return scaled32(0.5 * (__ldcg(T + at(r, c)) + __ldcg(T + at(c, r))), E - kUp32);
    };
    if (m <= k32Max) {
      if (blockIdx.x == 0) {
        float* sA = dyn;
        float* sV = dyn + 2 * m * m;
        for (int i = tid; i < m * m; i += kThreads) {
          sA[i] = t32(i / m, i % m);
          sV[i] = i / m == i % m ? 1.f : 0.f;
        }
        __syncthreads();
        int n = 0, copy = 0;
        switch (m) {
          case 16: n = jacobi32<16>(sA, sV, 20, floor32(var.least, E), S.s32, copy); break;
          case 32: n = jacobi32<32>(sA, sV, 20, floor32(var.least, E), S.s32, copy); break;
          case 48: n = jacobi32<48>(sA, sV, 20, floor32(var.least, E), S.s32, copy); break;
          default: n = jacobi32<64>(sA, sV, 20, floor32(var.least, E), S.s32, copy); break;
        }
        sV += copy * m * m;
        for (int i = tid; i < m * m; i += kThreads) __stcg(Q32 + i, sV[i]);
        if (tid == 0) __stcg(J.slots + 1023, static_cast<double>(n));
      }
      alive = grid.sync();
      sweeps = alive ? static_cast<int>(__ldcg(J.slots + 1023)) : 0;
    } else {
      for (int i = gtid; i < m * m; i += nthreads) {
        __stcg(F + i, t32(i / m, i % m));
        __stcg(Q32 + i, i / m == i % m ? 1.f : 0.f);
      }
      alive = grid.sync();
      if (alive) {
        sweeps = grid_jacobi32(J, grid, S, dyn, F, F + static_cast<size_t>(m) * m, Q32, floor32(var.least, E));
        alive = sweeps >= 0;
      }
    }
    // X = V Q (into w first: Q lies where X goes)
    if (alive) {
      if (seeded)
        grid_product(
            m, S, [&](int i, int k) { return __ldcg(V + at(i, k)); },
            [&](int k, int j) { return f32_to_f64(__ldcg(Q32 + at(k, j))); },
            [&](int i, int j, double v) { __stcg(J.w + at(i, j), v); });
      else
        for (int i = gtid; i < m * m; i += nthreads) __stcg(J.w + i, f32_to_f64(__ldcg(Q32 + i)));
      alive = grid.sync();
    }
  }
  // the refinement; if need be FP64 rotations, and its late steps for what they leave
  const Noise noise = noise_of(var.E, pa);
  float* weights = reinterpret_cast<float*>(J.slots + 256);
  int it = 0;
  for (bool rotated = false; alive; rotated = true) {
    bool refined = false;  // lambda and X hold the result
    bool warm = false;     // X is orthonormal, but some eigenvalues are too close for the refinement
    for (; in_range && it < kSteps; ++it) {
      grid_product(
          m, S, [&](int i, int k) { return __ldcg(A + at(i, k)); }, [&](int k, int j) { return __ldcg(X + at(k, j)); },
          [&](int i, int j, double v) { __stcg(W + at(i, j), v); });
      if (!(alive = grid.sync())) break;
      grid_grams(m, S, X, W, J.b, J.g, A, noise.E, weights);
      if (!(alive = grid.sync())) break;
      if (tid < m) {
        const double l = __ldcg(J.b + at(tid, tid)) / __ldcg(J.g + at(tid, tid));
        S.lambda[tid] = l;
        S.noise[tid] = noise.column(l, __ldcg(weights + tid), S.nf[tid], S.ni[tid]);
      }
      __syncthreads();
      int found = 0;
      for (int i = gtid; i < m * m; i += nthreads) {
        const int r = i / m, c = i % m;
        const double e = correction(r, c, __ldcg(J.b + i), __ldcg(J.g + i), S.lambda[r], S.lambda[c],
                                    S.noise[r] * S.noise[c], S.nf[r] * S.ni[c], S.nf[c] * S.ni[r], it, it == 0, found);
        __stcg(W + i, e);
      }
      found = block_or(found, reinterpret_cast<int*>(S.red));
      if (tid == 0) __stcg(reinterpret_cast<int*>(J.slots + blockIdx.x), found);
      if (!(alive = grid.sync())) break;
      found = slots_or(J.slots, S);
      if (found & kFailed) break;
      grid_product(
          m, S, [&](int i, int k) { return __ldcg(X + at(i, k)); }, [&](int k, int j) { return __ldcg(W + at(k, j)); },
          [&](int i, int j, double v) { __stcg(Xn + at(i, j), __ldcg(X + at(i, j)) + v); });
      if (!(alive = grid.sync())) break;
      double* t = X;
      X = Xn;
      Xn = t;
      if (!(found & kMore)) {
        refined = !(found & kClose);
        warm = !refined;
        break;
      }
    }
    if (!alive || refined || rotated) break;
    double* R = J.g;  // what is rotated: X^T A X, symmetrised, or A
    if (warm) {
      grid_product(
          m, S, [&](int i, int k) { return __ldcg(A + at(i, k)); }, [&](int k, int j) { return __ldcg(X + at(k, j)); },
          [&](int i, int j, double v) { __stcg(W + at(i, j), v); });
      if (!(alive = grid.sync())) break;
      grid_product(
          m, S, [&](int i, int k) { return __ldcg(X + at(k, i)); }, [&](int k, int j) { return __ldcg(W + at(k, j)); },
          [&](int i, int j, double v) { __stcg(J.b + at(i, j), v); });
      if (!(alive = grid.sync())) break;
      for (int i = gtid; i < m * m; i += nthreads)
        __stcg(R + i, 0.5 * (__ldcg(J.b + i) + __ldcg(J.b + at(i % m, i / m))));
    } else {
      X = V;
      for (int i = gtid; i < m * m; i += nthreads) {
        __stcg(X + i, (i / m == i % m) ? 1.0 : 0.0);
        __stcg(R + i, __ldcg(A + i));
      }
      seeded = false;
    }
    if (!(alive = grid.sync())) break;
    const int n = grid_jacobi64(J, grid, S, R, J.b, X, var.E);
    if (!(alive = n >= 0)) break;
    sweeps += n;
    if (tid < m) S.lambda[tid] = __ldcg(R + at(tid, tid));
    __syncthreads();
    Xn = X == V ? J.w : V;
    it = kPolish;
    if (!(alive = grid.sync())) break;  // b and g are free again
  }
  if (!alive) {
    if (tid == 0) flags[5] = 1.0;
    return;
  }
  // descending order (ties by index), eigenvector signs: largest-magnitude component positive
  if (tid < pa) {
    S.key[tid] = order_key(S.lambda[tid]);
    S.order[tid] = tid;
  }
  __syncthreads();
  if (tid < pa) {
    int rank = 0;
    const unsigned long long k = S.key[tid];
    for (int d = 0; d < pa; ++d) rank += (S.key[d] > k || (S.key[d] == k && d < tid)) ? 1 : 0;
    S.order[rank] = tid;
  }
  __syncthreads();
  double* evals = J.out + J.evals_off;
  double* evecs = J.out + J.evecs_off;
  for (int k = blockIdx.x; k < pa; k += gridDim.x) {
    const int col = S.order[k];
    double vi = 0.0;
    unsigned long long best = 0;
    int bi = kThreads;
    if (tid < pa) {
      vi = __ldcg(X + at(tid, col));
      best = magnitude_key(vi);
      bi = tid;
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
    if ((tid & 31) == 0) {
      S.best[tid >> 5] = best;
      S.best_i[tid >> 5] = bi;
    }
    __syncthreads();
    if (tid == 0) {
      unsigned long long bb = S.best[0];
      int ii = S.best_i[0];
      for (int w = 1; w < kThreads / 32; ++w)
        if (S.best[w] > bb || (S.best[w] == bb && S.best_i[w] < ii)) {
          bb = S.best[w];
          ii = S.best_i[w];
        }
      S.val = __ldcg(X + at(ii, col)) < 0.0 ? -1.0 : 1.0;
      evals[k] = S.lambda[col];
    }
    __syncthreads();
    if (tid < pa) evecs[static_cast<size_t>(k) * pa + tid] = S.val * vi;
    __syncthreads();
  }
  if (blockIdx.x == 0 && tid == 0) {
    flags[2] = sweeps;
    flags[3] = 1.0;
    flags[6] = seeded ? 1.0 : 0.0;
  }
}

cudaError_t launch_jacobi_grid(const JacobiParams& J, int grid, cudaStream_t stream) {
  if (grid < 1 || J.m > 256 || J.m < 16) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(jacobi_grid_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(kDynBytes));
  if (e != cudaSuccess) return e;
  void* args[] = {const_cast<JacobiParams*>(&J)};
  return cudaLaunchCooperativeKernel(reinterpret_cast<void*>(jacobi_grid_kernel), dim3(grid), dim3(kThreads), args,
                                     kDynBytes, stream);
}

}  // namespace ss
