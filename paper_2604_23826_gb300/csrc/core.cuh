// core.cuh -- what the two CUDA-core passes (k_core32.cu, k_core64.cu) share: the cut of the
// output's upper triangle into register micro-tiles, loads of any column type, and bounded
// copies into shared memory.
#pragma once

#include "common.cuh"
#include "kernels.h"

namespace ss {
namespace core {

// Micro-tile t of the upper triangle: MI x MJ entries at columns (MI * bi, MJ * bj), MI a multiple
// of MJ, bj >= bi * (MI / MJ); tiles of one bi are consecutive.
__host__ __device__ constexpr int tile_count(int p, int MI, int MJ) {
  const int nI = (p + MI - 1) / MI, nJ = (p + MJ - 1) / MJ;
  int m = 0;
  for (int b = 0; b < nI; ++b) m += nJ - b * (MI / MJ);
  return m;
}
template <int MI, int MJ>
__device__ __forceinline__ void tile_of(int t, int p, int& bi, int& bj) {
  const int nJ = (p + MJ - 1) / MJ;
  bi = 0;
  while (t >= nJ - bi * (MI / MJ)) {
    t -= nJ - bi * (MI / MJ);
    ++bi;
  }
  bj = bi * (MI / MJ) + t;
}

// hi + lo += v, the rounding of the addition kept in lo
template <typename Acc>
__device__ __forceinline__ void pair_add(Acc& hi, Acc& lo, Acc v) {
  const Acc s = hi + v;
  const Acc bp = s - hi;
  lo += (hi - (s - bp)) + (v - bp);
  hi = s;
}

// Exact conversions to FP64 on the integer pipe.  GB300 runs every FP64 instruction, conversions
// included, at 2 per clock and SM (64 cycles per warp instruction, measured), where the FP64
// passes have no slot to spare; these take about ten integer instructions instead.
__device__ __forceinline__ double i32_to_f64(int32_t v) {
  const uint32_t m = v < 0 ? 0u - static_cast<uint32_t>(v) : static_cast<uint32_t>(v);
  const int lz = __clz(static_cast<int>(m));  // 32 when v = 0
  const uint32_t n = lz < 32 ? m << lz : 0u;
  const uint32_t hi = (static_cast<uint32_t>(v) & 0x80000000u) + (static_cast<uint32_t>(1023 + 30 - lz) << 20) + (n >> 11);
  return v == 0 ? 0.0 : __hiloint2double(static_cast<int>(hi), static_cast<int>(n << 21));
}
__device__ __forceinline__ double load_as_double(const void* col, int dt, int64_t r) {
  switch (dt) {
    case I16: return i32_to_f64(static_cast<const int16_t*>(col)[r]);
    case I32: return i32_to_f64(static_cast<const int32_t*>(col)[r]);
    case I64: return static_cast<double>(static_cast<const int64_t*>(col)[r]);
    case F32: return f32_to_f64(static_cast<const float*>(col)[r]);
    default: return static_cast<const double*>(col)[r];
  }
}

// 16-byte asynchronous copy to shared memory of which only the first `bytes` are read, the rest
// written as zeros
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

}  // namespace core
}  // namespace ss
