// k_core64.cu -- the plain FP64 CUDA-core pass (STATS_FP64 with raw moments, as in the paper;
// STATS_FP64_SHIFTED on x - c), arxiv 2604.23826, "Data Representation and Sufficient
// Statistics" with the shift of "Numerical Considerations".
//
// Bound: the FP64 unit, 2 operations per clock and SM on GB300 (64 cycles a warp instruction,
// conversions and additions alike), so p (p + 1) / 2 FMAs plus 2 p additions a row set the time and
// everything else only has to stay off that unit and keep it fed:
//   - the output's upper triangle is cut into register micro-tiles of 4 x 4 or 2 x 2 entries, one
//     per thread, so little is multiplied that nobody reads (48 columns: 1248 of 1176);
//   - the rows of a stage are dealt to slices of a block's threads, so a few tiles fill all lanes;
//     core64_plan picks micro-tile, block size, slices and groups by the FP64 cycles a row costs;
//   - values are read as they lie (lanes = rows), turned into FP64 by integer instructions, shifted
//     and stored as rows of an odd stride (conflict-free); several blocks per SM overlap the
//     loads of one with the FMAs of another.
// 250,001 rows x 48 columns: 6.60 ms as 64 x 64 tiles on 61 blocks, 0.67 ms now (FMAs, shift and
// sums of those rows alone: 0.50 ms), plus 12 us to add the slots.  Up to 12 columns one thread kept a
// row's 90 sums in registers (2e7 rows of Table 1: 5.08 ms); its eight warps an SM spent half their
// time on loads and conversions.  This way: 3.88 ms (90 operations a row alone: 2.9 ms).
// Each block writes one slot; a second kernel adds an entry's slots in row order into the ctx's
// double-double accumulators (a fixed order: a given grid reproduces its bits).
// Sums are kept in blocks: a 2 x 2 tile's and a column's go to a second sum every kChain of a thread's rows
// or less (one addition in 128 FMAs or more), so the roundings on the way to a slot are at most kChain, the
// number of those blocks and the slices' tree: fewer at any row count than the 300 and a 78,000th of the
// rows that a grid of row-per-thread sums had (unblocked: an 8,000th; 12 columns x 1e7 rows 1.98 ms, 2.00 so).  4 x 4 tiles, from 13 columns on, have no registers
// for it and more threads to a row than 64 x 64 tiles had.
#include <algorithm>

#include "core.cuh"

namespace ss {

namespace {

using namespace core;

constexpr int kMaxThreads = 512;
constexpr int kBatch = 4;  // loads a lane has in flight
constexpr int kChain = 256;

__host__ __device__ inline int row_stride(int p, int MI) { return ((p + MI - 1) / MI * MI) | 1; }

// 32 nchunks rows of a column from row r0 on (those below `rows`) as x - c into X; a lane has
// kBatch loads in flight.  The type is the template's, so a value costs a load, about ten integer
// instructions and a store.
template <int DT>
__device__ __forceinline__ void convert_rows(const void* col, int64_t r0, int rows, int nchunks, bool shifted, double c,
                                             double* X, int S) {
  const int lane = threadIdx.x & 31;
  for (int k0 = lane; k0 < 32 * nchunks; k0 += 32 * kBatch) {
    uint64_t v[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) v[u] = k0 + 32 * u < rows ? load_bits(col, DT, r0 + k0 + 32 * u) : 0;
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
      if (k0 + 32 * u < rows) {
        const double x = bits_to_f64(v[u], DT);
        X[(k0 + 32 * u) * S] = shifted ? x - c : x;
      }
  }
}

template <int MI>
constexpr bool kBlocked = MI == 2;
// shared memory ahead of the second sums: a stage's rows, or the slices' partial sums
__host__ __device__ inline size_t first_bytes(const Core64Params& P, int MI) {
  const size_t rows = (size_t(1) << P.log_rows) * row_stride(P.p, MI), tree = static_cast<size_t>(MI) * MI * (P.threads / 2);
  return (rows > tree ? rows : tree) * sizeof(double);
}

// (registers: blocks of 384 threads fit three and two times on an SM)
template <int MI>
__global__ void __maxnreg__(MI == 2 ? 56 : 80) core64_kernel(const __grid_constant__ Core64Params P) {
  constexpr int kE = MI * MI;
  extern __shared__ __align__(16) uint8_t smem[];
  double* X = reinterpret_cast<double*>(smem);  // [R][S], rows of x - c
  const int p = P.p, R = 1 << P.log_rows, S = row_stride(p, MI);
  const int tid = threadIdx.x, NT = blockDim.x, warp = tid >> 5, nwarps = NT >> 5;
  const int g = blockIdx.x % P.groups, range = blockIdx.x / P.groups;
  const int64_t nst = (P.nrows + R - 1) >> P.log_rows;
  const int64_t st0 = nst * range / P.ranges, st1 = nst * (range + 1) / P.ranges;

  const int tg = P.tiles_per_group, slice = tid / tg, tl = tid % tg;
  const int tile = g * tg + tl;
  const bool active = slice < P.slices && tile < P.ntiles;
  int bi = 0, bj = 0;
  if (active) tile_of<MI, MI>(tile, p, bi, bj);
  double acc[MI][MI];
#pragma unroll
  for (int i = 0; i < MI; ++i)
#pragma unroll
    for (int j = 0; j < MI; ++j) acc[i][j] = 0.0;
  const int cc = tid % p, cq = tid / p, ncq = NT / p;  // column sums: this thread's column and rows
  double s = 0.0;
  // second sums of this thread's entries and column, in shared memory (registers would cost a block an SM)
  double* second = reinterpret_cast<double*>(smem + first_bytes(P, MI)) + tid;
  if (kBlocked<MI>)
    for (int e = 0; e <= kE; ++e) second[e * NT] = 0.0;
  // the columns that pad the last micro-tile are zero
  for (int i = tid; i < R * (S - p); i += NT) X[(i / (S - p)) * S + p + i % (S - p)] = 0.0;

  for (int64_t st = st0; st < st1; ++st) {
    const int64_t r0 = st << P.log_rows;
    const int rows = static_cast<int>(min(static_cast<int64_t>(R), P.nrows - r0));
    const int ng = (R + 127) / 128, nitems = p * ng;  // items: 128 rows of a column, fewer in a shorter stage
    __syncthreads();  // the last stage's rows have been read
    for (int it = warp; it < nitems; it += nwarps) {
      const int c = it / ng, k = (it - c * ng) * 128, nch = min(R - k, 128) / 32;
      const void* col = P.cols[c];
      const double sh = P.shift ? P.shift[c] : 0.0;
      double* dst = X + k * S + c;
      switch (P.dtype[c]) {
        case I16: convert_rows<I16>(col, r0 + k, rows - k, nch, P.shift, sh, dst, S); break;
        case I32: convert_rows<I32>(col, r0 + k, rows - k, nch, P.shift, sh, dst, S); break;
        case I64: convert_rows<I64>(col, r0 + k, rows - k, nch, P.shift, sh, dst, S); break;
        case F32: convert_rows<F32>(col, r0 + k, rows - k, nch, P.shift, sh, dst, S); break;
        default: convert_rows<F64>(col, r0 + k, rows - k, nch, P.shift, sh, dst, S); break;
      }
    }
    __syncthreads();
    if (g == 0 && cq < ncq)
      for (int k = cq; k < rows; k += ncq) s += X[k * S + cc];
    if (active) {
      const double* xa = X + MI * bi;
      const double* xb = X + MI * bj;
#pragma unroll 2
      for (int k = slice; k < rows; k += P.slices) {
        double a[MI], b[MI];
#pragma unroll
        for (int i = 0; i < MI; ++i) a[i] = xa[k * S + i];
#pragma unroll
        for (int j = 0; j < MI; ++j) b[j] = xb[k * S + j];
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
          for (int j = 0; j < MI; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
      }
    }
    if (kBlocked<MI> && (st & P.chain_mask) == 0) {
#pragma unroll
      for (int e = 0; e < kE; ++e) {
        second[e * NT] += acc[e / MI][e % MI];
        acc[e / MI][e % MI] = 0.0;
      }
      second[kE * NT] += s;
      s = 0.0;
    }
  }
  if (kBlocked<MI>) {
#pragma unroll
    for (int e = 0; e < kE; ++e) acc[e / MI][e % MI] += second[e * NT];
    s += second[kE * NT];
  }
  // the slices' partial sums, added in a fixed tree through shared memory
  double* buf = X;
  for (int n = P.slices; n > 1;) {
    const int h = (n + 1) / 2;
    __syncthreads();
    if (slice >= h && slice < n) {
#pragma unroll
      for (int e = 0; e < kE; ++e) buf[e * (NT / 2) + (slice - h) * tg + tl] = acc[e / MI][e % MI];
    }
    __syncthreads();
    if (slice < n - h) {
#pragma unroll
      for (int e = 0; e < kE; ++e) acc[e / MI][e % MI] += buf[e * (NT / 2) + slice * tg + tl];
    }
    n = h;
  }
  double* slot = P.slots + static_cast<size_t>(blockIdx.x) * core64_slot_doubles(p, tg, MI);
  if (slice == 0) {
#pragma unroll
    for (int e = 0; e < kE; ++e) slot[static_cast<size_t>(e) * tg + tl] = acc[e / MI][e % MI];
  }
  __syncthreads();
  if (cq < ncq) buf[cq * p + cc] = s;
  __syncthreads();
  if (g == 0 && tid < p) {
    double t = 0.0;
    for (int i = 0; i < ncq; ++i) t += buf[i * p + tid];
    slot[static_cast<size_t>(kE) * tg + tid] = t;
  }
}

// Adds the ranges' slots of 32 entries per block, kSeg consecutive runs of ranges at once, in
// double-double; the runs in order, then into the accumulators.
constexpr int kSeg = 16;

template <int MI>
__global__ void __launch_bounds__(32 * kSeg) core64_merge_kernel(const __grid_constant__ Core64Params P) {
  __shared__ double sh[kSeg][32], sl[kSeg][32];
  constexpr int kE = MI * MI;
  const int p = P.p, tg = P.tiles_per_group, lane = threadIdx.x & 31, seg = threadIdx.x >> 5;
  const int nS = P.ntiles * kE;
  const int x = blockIdx.x * 32 + lane;
  const size_t sd = core64_slot_doubles(p, tg, MI);
  int j = -1, k = -1;
  size_t off = 0;
  if (x < nS) {
    const int e = x / P.ntiles, t = x % P.ntiles, g = t / tg;
    int bi, bj;
    tile_of<MI, MI>(t, p, bi, bj);
    j = MI * bi + e / MI;
    k = MI * bj + e % MI;
    if (j > k || k >= p) j = -1;
    off = static_cast<size_t>(g) * sd + static_cast<size_t>(e) * tg + (t - g * tg);
  } else if (x < nS + p) {
    j = k = x - nS;
    off = static_cast<size_t>(kE) * tg + j;
  }
  double h = 0.0, l = 0.0;
  if (j >= 0) {
    const double* src = P.slots + off;
    const size_t step = static_cast<size_t>(P.groups) * sd;
    const int r0 = P.ranges * seg / kSeg, r1 = P.ranges * (seg + 1) / kSeg;
#pragma unroll 4
    for (int r = r0; r < r1; ++r) pair_add(h, l, __ldcg(src + r * step));
  }
  sh[seg][lane] = h;
  sl[seg][lane] = l;
  __syncthreads();
  if (seg == 0 && j >= 0) {
    for (int i = 1; i < kSeg; ++i) {
      pair_add(h, l, sh[i][lane]);
      l += sl[i][lane];
    }
    const int idx = x < nS ? j * p - j * (j - 1) / 2 + (k - j) : j;
    double* ah = (x < nS ? P.acc_S : P.acc_s) + idx;
    double* al = (x < nS ? P.acc_S_lo : P.acc_s_lo) + idx;
    double vh = *ah, vl = *al;
    pair_add(vh, vl, h);
    *ah = vh;
    *al = vl + l;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *P.acc_n += P.nrows;
}

size_t smem_bytes(const Core64Params& P) {
  return first_bytes(P, P.micro) + (P.micro == 2 ? 5 * sizeof(double) * P.threads : 0);
}

const void* kernel_of(int micro) {
  return micro == 4 ? reinterpret_cast<const void*>(core64_kernel<4>) : reinterpret_cast<const void*>(core64_kernel<2>);
}

}  // namespace

// The cut of p columns and nrows rows for `sms` SMs (or `blocks` blocks, when positive).
cudaError_t core64_plan(int p, int64_t nrows, bool shifted, int sms, int blocks, Core64Params& P) {
  double best = 0;
  for (int micro : {4, 2}) {
    if (micro == 4 && p <= 12) continue;
    const int M = core::tile_count(p, micro, micro);
    for (int nt = 128; nt <= kMaxThreads; nt += 128) {
      if (nt < p) continue;  // the column sums take a thread per column
      const int G0 = (M + nt - 1) / nt;
      for (int G = G0; G <= G0 + 8; ++G) {
        const int tg = (M + G - 1) / G, ks = nt / tg;
        if (tg * (G - 1) >= M) continue;
        // FP64 warp instructions a row costs one of the SM's four schedulers: the tiles' FMAs, in every
        // group the shift and (a quarter of one a value) loading and converting, the column sums in one
        const double fmas = ((tg * ks + 31) / 32 + 3) / 4 * double(micro * micro) / ks;
        const double cost = G * (fmas + (shifted ? 1.25 : 0.25) * p / 128.0) + double(nt) / (nt / p * p) * p / 128.0;
        if (best == 0 || cost < best) {
          best = cost;
          P.micro = micro;
          P.threads = nt;
          P.ntiles = M;
          P.groups = G;
          P.tiles_per_group = tg;
          P.slices = ks;
        }
      }
    }
  }
  // rows of a stage: about 32 KB, fewer while that would leave SMs without one
  int lr = 5;
  while (lr < 9 && (row_stride(p, P.micro) << (lr + 1)) <= 4096 &&
         (nrows >> (lr + 1)) >= 4 * int64_t(std::max(1, sms / P.groups)))
    ++lr;
  P.log_rows = lr;
  const int per_stage = ((1 << lr) + std::min(P.slices, P.threads / p) - 1) / std::min(P.slices, P.threads / p);
  P.chain_mask = 0;  // a thread's rows of chain_mask + 1 stages: at most kChain, or one stage's
  while (2 * (P.chain_mask + 1) * per_stage <= kChain) P.chain_mask = 2 * P.chain_mask + 1;
  const size_t smem = smem_bytes(P);
  cudaError_t e = cudaFuncSetAttribute(kernel_of(P.micro), cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  int per = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel_of(P.micro), P.threads, smem);
  if (e != cudaSuccess) return e;
  const int64_t nst = (nrows + (int64_t(1) << lr) - 1) >> lr;
  const int64_t want = blocks > 0 ? blocks : int64_t(sms) * std::max(1, std::min(per, 4));
  P.ranges = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(want / P.groups, nst)));
  return cudaSuccess;
}

size_t core64_slot_bytes(const Core64Params& P) {
  return static_cast<size_t>(P.groups) * P.ranges * core64_slot_doubles(P.p, P.tiles_per_group, P.micro) * sizeof(double);
}

cudaError_t launch_core64(const Core64Params& P, cudaStream_t stream) {
  const size_t smem = smem_bytes(P);
  const int grid = P.groups * P.ranges, mgrid = (P.ntiles * P.micro * P.micro + P.p + 31) / 32;
  cudaError_t e = cudaFuncSetAttribute(kernel_of(P.micro), cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  if (P.micro == 4) {
    core64_kernel<4><<<grid, P.threads, smem, stream>>>(P);
    core64_merge_kernel<4><<<mgrid, 32 * kSeg, 0, stream>>>(P);
  } else {
    core64_kernel<2><<<grid, P.threads, smem, stream>>>(P);
    core64_merge_kernel<2><<<mgrid, 32 * kSeg, 0, stream>>>(P);
  }
  return cudaGetLastError();
}

}  // namespace ss
