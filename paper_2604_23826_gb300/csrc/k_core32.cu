// k_core32.cu -- the FP32-core pass (STATS_FP32): n, X^T 1 and X^T X of x - c with FP32 FMA on the
// CUDA cores, flushed into FP32 (hi, lo) pairs at least every 64 rows (arxiv 2604.23826, "Data
// Representation and Sufficient Statistics" with the shift of "Numerical Considerations").
//
// Bound: FP32 FMA for more than about fifty columns (p (p + 1) / 2 per row at 128 per clock and
// SM), HBM below.  So the layout spends issue slots, shared-memory reads and barriers on as little
// else as possible:
//   - the output's upper triangle is cut into 8 x 4 register micro-tiles, one per thread: three
//     128-bit shared loads and four register pairs feed 16 packed FMAs of two entries each (which
//     take two cycles, so the other instructions issue beside them).  Only tiles on or above the
//     diagonal exist, so 100 columns cost 5408 FMAs a row for 5050 entries (8 x 8 tiles would want
//     192 registers for the sums and their (hi, lo) pairs);
//   - when there are fewer tiles than threads, the rows of a stage are dealt to several slices of
//     threads; when there are more, groups of blocks take a part of the tiles each.  core32_plan
//     picks the number of groups by the instructions a row costs;
//   - columns are copied as they lie (cp.async, 16 bytes, two stages ahead), then one pass turns a
//     stage into rows of x - c (lanes = columns: conflict-free both ways) and adds the column sums,
//     while other warps still multiply the stage before: one barrier a stage.
// Columns of other types, or not 16-byte aligned, are converted (x - c in FP64) into the same
// stage by plain loads.
// 1e6 rows x 100 columns: 0.427 ms (its FMAs alone: 0.135; as 64 x 64 tiles of scalar loads 8.78).
// Each block writes one slot of (hi, lo) pairs; a second kernel adds the slots of an entry in row
// order, in three-term FP32 expansions and then FP64 pairs (a fixed order: a given grid
// reproduces its bits).  Sums that leave FP32's range on the way are added in FP64 instead, so only a
// thread's own rows have to stay within it.
#include <algorithm>

#include "core.cuh"

namespace ss {

namespace {

using namespace core;

constexpr int kMI = 8, kMJ = 4, kE = kMI * kMJ;
constexpr int kNT = 512;
constexpr size_t kSmemMax = 226 * 1024;
constexpr size_t kTreeBytes = (kNT / 2) * kE * 8;  // the slices' pairs on their way to one slot

__host__ __device__ inline int width_of(int p) { return (p + kMI - 1) / kMI * kMI; }
__host__ __device__ inline size_t raw_bytes(int W, int R) { return static_cast<size_t>(W) * (R + 4) * 4; }
__host__ __device__ inline size_t row_bytes(int W, int R) { return static_cast<size_t>(R) * (W + 4) * 4; }

// two FP32 values in a 64-bit register: one instruction works on both, each rounded as by itself
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 twice(float v) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(v));
  return d;
}
__device__ __forceinline__ float2 parts(f32x2 v) {
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(v));
  return d;
}
__device__ __forceinline__ void fma2(f32x2& d, f32x2 a, f32x2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

__global__ void __launch_bounds__(kNT, 1) core32_kernel(const __grid_constant__ Core32Params P) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int p = P.p, W = width_of(p), R = 1 << P.log_rows, S = W + 4, K = R + 4;
  float* raw = reinterpret_cast<float*>(smem);                     // [2][W][K], as the columns lie
  float* X = reinterpret_cast<float*>(smem + 2 * raw_bytes(W, R));  // [2][R][S], rows of x - c
  const int tid = threadIdx.x;
  const int g = blockIdx.x % P.groups, range = blockIdx.x / P.groups;
  const int64_t nst = (P.nrows + R - 1) >> P.log_rows;
  const int64_t st0 = nst * range / P.ranges, st1 = nst * (range + 1) / P.ranges;

  // compute: slice tid / tg takes rows slice, slice + slices, ... of a stage for tile tid % tg
  const int tg = P.tiles_per_group, slice = tid / tg, tl = tid % tg;
  const int tile = g * tg + tl;
  const bool active = slice < P.slices && tile < P.ntiles;
  int bi = 0, bj = 0;
  if (active) tile_of<kMI, kMJ>(tile, p, bi, bj);
  f32x2 acc[kMI / 2][kMJ], hi[kMI / 2][kMJ], lo[kMI / 2][kMJ];  // rows 2 i, 2 i + 1 of the tile together
#pragma unroll
  for (int i = 0; i < kMI / 2; ++i)
#pragma unroll
    for (int j = 0; j < kMJ; ++j) acc[i][j] = hi[i][j] = lo[i][j] = 0;
  int since = 0;
  auto flush = [&] {
    since = 0;
#pragma unroll
    for (int i = 0; i < kMI / 2; ++i)
#pragma unroll
      for (int j = 0; j < kMJ; ++j) {  // pair_add
        const f32x2 s = add2(hi[i][j], acc[i][j]), bp = sub2(s, hi[i][j]);
        lo[i][j] = add2(lo[i][j], add2(sub2(hi[i][j], sub2(s, bp)), sub2(acc[i][j], bp)));
        hi[i][j] = s;
        acc[i][j] = 0;
      }
  };

  // conversion: this thread's column and its share of the stage's row quads
  const int cc = tid % W, cq = tid / W, ncq = kNT / W;
  const bool quick = cc < p && (P.quick[cc >> 5] >> (cc & 31) & 1u);
  const float shift = quick ? static_cast<float>(P.shift[cc]) : 0.f;
  float shi = 0.f, slo = 0.f;

  auto issue = [&](int64_t st) {
    float* dst = raw + (st & 1) * (raw_bytes(W, R) / 4);
    const int64_t r0 = st << P.log_rows;
    const int rows = static_cast<int>(min(static_cast<int64_t>(R), P.nrows - r0));
    const int lq = P.log_rows - 2;  // quads of a column: 2^lq
    for (int i = tid; i < (p << lq); i += kNT) {
      const int c = i >> lq, k = (i & ((1 << lq) - 1)) * 4;
      if (!(P.quick[c >> 5] >> (c & 31) & 1u)) continue;
      const int have = min(4, max(0, rows - k));
      const float* src = static_cast<const float*>(P.cols[c]) + r0 + (have ? k : 0);
      cp_async16(smem_u32(dst + c * K + k), src, 4 * have);
    }
    if (P.any_slow)
      for (int i = tid; i < (p << P.log_rows); i += kNT) {
        const int c = i >> P.log_rows, k = i & (R - 1);
        if (P.quick[c >> 5] >> (c & 31) & 1u) continue;
        if (k < rows) {
          float v;
          if (P.dtype[c] == F32)
            v = static_cast<const float*>(P.cols[c])[r0 + k] - static_cast<float>(P.shift[c]);
          else
            v = static_cast<float>(load_as_double(P.cols[c], P.dtype[c], r0 + k) - P.shift[c]);
          dst[c * K + k] = v;
        }
      }
  };
  auto convert = [&](int64_t st) {
    if (cq >= ncq) return;
    const int rows = static_cast<int>(min(static_cast<int64_t>(R), P.nrows - (st << P.log_rows)));
    const float* src = raw + (st & 1) * (raw_bytes(W, R) / 4) + cc * K;
    float* dst = X + (st & 1) * (row_bytes(W, R) / 4) + cc;
    float s = 0.f;
#pragma unroll 2
    for (int k = 4 * cq; k < R; k += 4 * ncq) {
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      if (cc < p) {
        const float4 x = *reinterpret_cast<const float4*>(src + k);
        v[0] = k < rows ? x.x - shift : 0.f;
        v[1] = k + 1 < rows ? x.y - shift : 0.f;
        v[2] = k + 2 < rows ? x.z - shift : 0.f;
        v[3] = k + 3 < rows ? x.w - shift : 0.f;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) dst[(k + i) * S] = v[i];
      s += (v[0] + v[1]) + (v[2] + v[3]);
    }
    pair_add(shi, slo, s);
  };

  // One barrier a stage: while stage st is multiplied, st + 1 is turned into rows by whichever warps
  // are done, and st + 2 is on its way.
  if (st0 < st1) issue(st0);
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  if (st0 + 1 < st1) issue(st0 + 1);
  cp_async_commit();
  if (st0 < st1) convert(st0);
  for (int64_t st = st0; st < st1; ++st) {
    cp_async_wait<0>();
    __syncthreads();  // st is rows, st + 1 has landed, and st's columns and st - 1's rows are free
    if (st + 2 < st1) issue(st + 2);
    cp_async_commit();
    if (active) {
      const int rows = static_cast<int>(min(static_cast<int64_t>(R), P.nrows - (st << P.log_rows)));
      const float* x = X + (st & 1) * (row_bytes(W, R) / 4) + slice * S;
      const float* xa = x + kMI * bi;
      const float* xb = x + kMJ * bj;
      const int step = P.slices * S;
      for (int left = (rows - slice + P.slices - 1) / P.slices; left > 0;) {
        if (since == P.flush_rows) flush();
        const int m = min(left, P.flush_rows - since);
        since += m;
        left -= m;
#pragma unroll 2
        for (int i = 0; i < m; ++i, xa += step, xb += step) {
          const ulonglong2 a01 = *reinterpret_cast<const ulonglong2*>(xa);
          const ulonglong2 a23 = *reinterpret_cast<const ulonglong2*>(xa + 4);
          const float4 b4 = *reinterpret_cast<const float4*>(xb);
          const f32x2 a[4] = {a01.x, a01.y, a23.x, a23.y};
          const f32x2 b[4] = {twice(b4.x), twice(b4.y), twice(b4.z), twice(b4.w)};
#pragma unroll
          for (int u = 0; u < kMI / 2; ++u)
#pragma unroll
            for (int v = 0; v < kMJ; ++v) fma2(acc[u][v], a[u], b[v]);
        }
      }
    }
    if (st + 1 < st1) convert(st + 1);
  }
  flush();
  auto at = [](const f32x2(&v)[kMI / 2][kMJ], int e) {  // entry e = 4 row + column of the tile
    const float2 w = parts(v[e / kMJ / 2][e % kMJ]);
    return (e / kMJ) & 1 ? w.y : w.x;
  };
  // the slices' pairs, added in a fixed tree through shared memory; near the end of FP32's range all of the
  // block's are taken at 2^-10 (at most 512 slices)
  float2* buf = reinterpret_cast<float2*>(smem);
  float scale = 1.f;
  if (P.slices > 1) {
    float top = 0.f;
#pragma unroll
    for (int e = 0; e < kE; ++e) top = fmaxf(top, fabsf(at(hi, e)));
    if (__syncthreads_or(top >= 0x1p117f)) {
      scale = 0x1p10f;
#pragma unroll
      for (int i = 0; i < kMI / 2; ++i)
#pragma unroll
        for (int j = 0; j < kMJ; ++j) {
          hi[i][j] = mul2(hi[i][j], twice(0x1p-10f));
          lo[i][j] = mul2(lo[i][j], twice(0x1p-10f));
        }
    }
  }
  for (int n = P.slices; n > 1;) {
    const int h = (n + 1) / 2;
    __syncthreads();
    if (slice >= h && slice < n) {
#pragma unroll
      for (int e = 0; e < kE; ++e)
        buf[e * (kNT / 2) + (slice - h) * tg + tl] = make_float2(at(hi, e), at(lo, e));
    }
    __syncthreads();
    if (slice < n - h) {
#pragma unroll
      for (int i = 0; i < kMI / 2; ++i)
#pragma unroll
        for (int j = 0; j < kMJ; ++j) {
          const float2 v = buf[(2 * i * kMJ + j) * (kNT / 2) + slice * tg + tl];
          const float2 w = buf[((2 * i + 1) * kMJ + j) * (kNT / 2) + slice * tg + tl];
          float2 h = parts(hi[i][j]), l = parts(lo[i][j]);
          pair_add(h.x, l.x, v.x);
          pair_add(h.y, l.y, w.x);
          l.x += v.y;
          l.y += w.y;
          asm("mov.b64 %0, {%1, %2};" : "=l"(hi[i][j]) : "f"(h.x), "f"(h.y));
          asm("mov.b64 %0, {%1, %2};" : "=l"(lo[i][j]) : "f"(l.x), "f"(l.y));
        }
    }
    n = h;
  }
  float2* slot = reinterpret_cast<float2*>(P.slots) + static_cast<size_t>(blockIdx.x) * core32_slot_pairs(p, tg);
  if (slice == 0) {
#pragma unroll
    for (int e = 0; e < kE; ++e)
      slot[static_cast<size_t>(e) * tg + tl] = make_float2(at(hi, e), at(lo, e));
  }
  __syncthreads();
  if (cq < ncq) buf[cq * W + cc] = make_float2(shi, slo);
  __syncthreads();
  if (tid < W) {
    float h = 0.f, l = 0.f;
    for (int i = 0; i < ncq; ++i) {
      const float2 v = buf[i * W + tid];
      pair_add(h, l, v.x);
      l += v.y;
    }
    slot[static_cast<size_t>(kE) * tg + tid] = make_float2(h, l);
  }
  if (tid == 0) slot[static_cast<size_t>(kE) * tg + W] = make_float2(scale, 0.f);
}

// Adds the ranges' slots of 32 entries per block (kSeg consecutive runs of ranges at once) into
// the accumulators.  Within a run a three-term FP32 expansion keeps every rounding of the pairs'
// additions (72 bits; FP64 adds would cost 64 cycles a warp each); the runs are added in order in
// FP64 pairs.  A run that leaves FP32's range, and all runs when some block scaled its sums, are added
// in FP64 pairs throughout.
constexpr int kSeg = 8;
__device__ __forceinline__ float two_sum32(float& s, float v) {
  const float t = s + v, bp = t - s, e = (s - (t - bp)) + (v - bp);
  s = t;
  return e;
}

__global__ void __launch_bounds__(32 * kSeg, 8) core32_merge_kernel(const __grid_constant__ Core32Params P) {
  __shared__ double sh[kSeg][32], sl[kSeg][32];
  const int p = P.p, tg = P.tiles_per_group, lane = threadIdx.x & 31, seg = threadIdx.x >> 5;
  const int nS = P.ntiles * kE;
  const int x = blockIdx.x * 32 + lane;  // entry: tiles' values, then the column sums
  const size_t sp = core32_slot_pairs(p, tg);
  const float2* slots = reinterpret_cast<const float2*>(P.slots);
  const size_t at_scale = static_cast<size_t>(kE) * tg + width_of(p);
  bool scaled = false;
  for (int b = threadIdx.x; P.slices > 1 && b < P.groups * P.ranges; b += blockDim.x)
    scaled |= __ldcg(slots + b * sp + at_scale).x != 1.f;
  scaled = __syncthreads_or(scaled);
  int j = -1, k = -1, group = 0;
  size_t off = 0;
  if (x < nS) {
    const int e = x / P.ntiles, t = x % P.ntiles, g = t / tg;
    int bi, bj;
    tile_of<kMI, kMJ>(t, p, bi, bj);
    j = kMI * bi + e / kMJ;
    k = kMJ * bj + e % kMJ;
    if (j > k || k >= p) j = -1;
    group = g;
    off = static_cast<size_t>(e) * tg + (t - g * tg);
  } else if (x < nS + p) {
    j = k = x - nS;
    off = static_cast<size_t>(kE) * tg + j;
  }
  float h = 0.f, l = 0.f, ll = 0.f;
  const float2* src = slots + group * sp + off;
  const size_t step = static_cast<size_t>(P.groups) * sp;
  const int r0 = P.ranges * seg / kSeg, r1 = P.ranges * (seg + 1) / kSeg;
  if (j >= 0 && !scaled) {
#pragma unroll 8
    for (int r = r0; r < r1; ++r) {
      const float2 v = __ldcg(src + r * step);
      const float e1 = two_sum32(h, v.x);
      const float e2 = two_sum32(l, e1);
      ll += e2 + two_sum32(l, v.y);
    }
  }
  double dh = h, dl = 0.0;
  if (j >= 0 && (scaled || !(fabsf(h) <= 0x1.fffffep127f))) {
    const float2* scales = slots + group * sp + at_scale;
    dh = 0.0;
    for (int r = r0; r < r1; ++r) {
      const float2 v = __ldcg(src + r * step);
      const double s = x < nS ? __ldcg(scales + r * step).x : 1.0;
      pair_add(dh, dl, v.x * s);
      dl += v.y * s;
    }
  } else {
    pair_add(dh, dl, static_cast<double>(l));
    dl += ll;
  }
  sh[seg][lane] = dh;
  sl[seg][lane] = dl;
  __syncthreads();
  if (seg == 0 && j >= 0) {
    for (int s = 1; s < kSeg; ++s) {
      pair_add(dh, dl, sh[s][lane]);
      dl += sl[s][lane];
    }
    const int idx = x < nS ? j * p - j * (j - 1) / 2 + (k - j) : j;
    double* ah = (x < nS ? P.acc_S : P.acc_s) + idx;
    double* al = (x < nS ? P.acc_S_lo : P.acc_s_lo) + idx;
    double vh = *ah, vl = *al;
    pair_add(vh, vl, dh);
    *ah = vh;
    *al = vl + dl;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *P.acc_n += P.nrows;
}

size_t smem_bytes(int W, int R) {
  return std::max<size_t>(2 * raw_bytes(W, R) + 2 * row_bytes(W, R), kTreeBytes);
}

}  // namespace

// The cut of p columns and nrows rows for `sms` SMs (or `blocks` blocks, when positive).
void core32_plan(int p, int64_t nrows, int sms, int blocks, Core32Params& P) {
  const int W = width_of(p), M = tile_count(p, kMI, kMJ);
  P.ntiles = M;
  // groups of blocks over the tiles: the fewest warp instructions a row costs the SMs together,
  // ~42 per warp of tiles (16 double FMAs of two cycles, 3 loads, 4 copies; warps run four at a time) and ~14 per 128
  // converted values in every group
  double best = 0;
  for (int G = (M + kNT - 1) / kNT; G <= 4 * ((M + kNT - 1) / kNT); ++G) {
    const int tg = (M + G - 1) / G, ks = kNT / tg;
    if (tg * (G - 1) >= M) continue;
    const int quads = ((tg * ks + 31) / 32 + 3) / 4;
    const double cost = G * (quads * 4 * 42.0 / ks + W * 14.0 / 128);
    if (best == 0 || cost < best) {
      best = cost;
      P.groups = G;
      P.tiles_per_group = tg;
      P.slices = ks;
    }
  }
  // rows of a stage: as many as shared memory takes, fewer while that would leave SMs without one
  int lr = 5;
  const int want = std::max(1, (blocks > 0 ? blocks : sms) / P.groups);
  while (lr < 11 && smem_bytes(W, 1 << (lr + 1)) <= kSmemMax && (nrows >> (lr + 1)) >= 2 * int64_t(want)) ++lr;
  P.log_rows = lr;
  const int64_t nst = (nrows + (int64_t(1) << lr) - 1) >> lr;
  P.ranges = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(want, nst)));
  // Sums of squares up to FP32's range are promised for a thread's rows as 64 x 64 tiles of four blocks an SM
  // dealt them, 4096 rows a block at least.  Wide tables of few slices (176..192 columns and from 252 on)
  // give a thread up to a third more, and take their rows in two launches.
  const int nb = (p + 63) / 64, tiles = nb * (nb + 1) / 2;
  const int64_t dealt = std::min<int64_t>(nrows / 4096, (4 * int64_t(sms) + tiles - 1) / tiles);
  P.launches = blocks <= 0 && int64_t(P.ranges) * P.slices < dealt ? 2 : 1;
  P.ranges *= P.launches;
}

size_t core32_slot_bytes(const Core32Params& P) {
  return static_cast<size_t>(P.groups) * P.ranges * core32_slot_pairs(P.p, P.tiles_per_group) * sizeof(float2);
}

cudaError_t launch_core32(const Core32Params& P, cudaStream_t stream) {
  const size_t smem = smem_bytes(width_of(P.p), 1 << P.log_rows);
  cudaError_t e = cudaFuncSetAttribute(core32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  const int64_t nst = (P.nrows + (int64_t(1) << P.log_rows) - 1) >> P.log_rows;
  for (int i = 0; i < P.launches; ++i) {  // whole stages: the columns stay as aligned as they were
    const int64_t first = nst * i / P.launches << P.log_rows;
    Core32Params Q = P;
    Q.ranges = P.ranges / P.launches;
    Q.nrows = std::min(P.nrows, nst * (i + 1) / P.launches << P.log_rows) - first;
    Q.slots = P.slots + 2 * core32_slot_pairs(P.p, P.tiles_per_group) * P.groups * Q.ranges * i;
    for (int c = 0; c < P.p; ++c) Q.cols[c] = static_cast<const char*>(P.cols[c]) + first * dtype_bytes(P.dtype[c]);
    core32_kernel<<<P.groups * Q.ranges, kNT, smem, stream>>>(Q);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  core32_merge_kernel<<<(P.ntiles * kE + P.p + 31) / 32, 32 * kSeg, 0, stream>>>(P);
  return cudaGetLastError();
}

}  // namespace ss
