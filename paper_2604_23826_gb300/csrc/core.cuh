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
__device__ __forceinline__ double i64_to_f64(int64_t v) {
  const uint64_t m = v < 0 ? 0ull - static_cast<uint64_t>(v) : static_cast<uint64_t>(v);
  const int lz = __clzll(static_cast<long long>(m));
  if (lz < 11) return static_cast<double>(v);  // more than 53 bits: rounds
  if (v == 0) return 0.0;
  // n: the significand with its leading one at bit 52, which the exponent's field adds back
  const uint64_t n = m << (lz - 11);
  const uint64_t bits = (static_cast<uint64_t>(v) & (1ull << 63)) + (static_cast<uint64_t>(1023 + 62 - lz) << 52) + n;
  return __longlong_as_double(static_cast<long long>(bits));
}

// the bits of value r of a column, sign-extended integers below 64 bits; bits_to_f64 turns them into
// the value.  Two steps, so that a thread can have many loads in flight.
__device__ __forceinline__ uint64_t load_bits(const void* col, int dt, int64_t r) {
  if (dt == F64 || dt == I64) return static_cast<const uint64_t*>(col)[r];
  if (dt == I16) return static_cast<uint32_t>(static_cast<const int16_t*>(col)[r]);
  return static_cast<const uint32_t*>(col)[r];
}
__device__ __forceinline__ double bits_to_f64(uint64_t b, int dt) {
  if (dt == F64) return __longlong_as_double(static_cast<long long>(b));
  if (dt == F32) return f32_to_f64(__uint_as_float(static_cast<uint32_t>(b)));
  if (dt == I64) return i64_to_f64(static_cast<int64_t>(b));
  return i32_to_f64(static_cast<int32_t>(b));
}

__device__ __forceinline__ double load_as_double(const void* col, int dt, int64_t r) {
  return bits_to_f64(load_bits(col, dt, r), dt);
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
