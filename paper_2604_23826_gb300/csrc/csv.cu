// csv.cu -- CSV text tables: a host writer, and a parser on the GPU for the first k
// fields of every line (arxiv 2604.23826, "Validation and Infrastructure Verification":
// the validation program streamed the CSV file in chunks and parsed its first column on
// the GPUs; "Data Representation and Sufficient Statistics": text parsing dominated, so
// the table was converted to binary).
//
// Device parse of a text buffer, four launches:
//   csv_count_kernel   newlines per 4 KB tile, a warp each (eight 16-byte loads a lane in flight,
//                      four bytes compared at a time);
//   csv_scan_kernel    one block: exclusive prefix of the tile counts, the line count
//                      (plus one for a last line without '\n');
//   csv_index_kernel   each tile again: the offsets of its newlines, in order;
//   csv_parse_kernel   one thread per line: the first k fields, converted and stored in
//                      column j at the line's row (adjacent lines -> adjacent rows, so
//                      the stores of a warp are contiguous).
// Bound: instruction issue in the parse.  Fields are taken eight characters at a time: one
// comparison finds the digits' end, three multiplications give their value; a character loop takes
// the rest (exponents, more than 19 digits) and every error.  1.5e6 lines of Table 1 (115 MB):
// parse 353 us a character at a time, 184 now; counting, scanning and indexing 142 us, 68 now.
// Number conversion is exact.  A real field is M * 10^E with M < 10^19 (the significant
// digits as an integer, trailing zeros moved into E) and -38 <= E <= 19.  For E >= 0 the product M * 10^E is formed in
// 128-bit integers; for E < 0 the quotient M * 2^s / 10^-E (a 64-bit quotient and a sticky
// remainder bit) comes, for -E <= 27, from one division by the normalised 5^-E with its
// precomputed reciprocal (exact quotient and remainder), and below that from binary long
// division.  Either way the exact value is
// a 64-bit integer q plus a sticky fraction times a power of two, rounded once to
// nearest, ties to even, to the 53 (FP64) or 24 (FP32) bits of the column type, and
// assembled bit by bit.
#include <fcntl.h>
#include <stdio.h>
#include <string.h>
#include <unistd.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <thread>
#include <vector>

#include "../../include/stats_csv.h"
#include "common.cuh"
#include "kernels.h"

namespace ss {

namespace {

constexpr int kCsvThreads = 256;  // a warp per tile in the counting and indexing kernels

// One warp per tile: lane l holds bytes 16 l .. 16 l + 15 of each of its kChunks 512-byte chunks.
constexpr int kChunks = kCsvTile / 512;

// newlines of a lane's 16 bytes of every chunk, a bit per byte; all loads in flight at once
__device__ __forceinline__ void newline_masks(const char* __restrict__ t, int64_t n, int64_t tile, bool aligned,
                                              uint32_t (&mask)[kChunks]) {
  const int64_t p0 = tile * kCsvTile + (threadIdx.x & 31) * 16;
  if (aligned && (tile + 1) * kCsvTile <= n) {
    uint4 v[kChunks];
#pragma unroll
    for (int c = 0; c < kChunks; ++c) v[c] = __ldg(reinterpret_cast<const uint4*>(t + p0 + c * 512));
#pragma unroll
    for (int c = 0; c < kChunks; ++c) {
      const uint32_t w[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
      mask[c] = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t hit = __vcmpeq4(w[i], 0x0A0A0A0Au) & 0x01010101u;  // a 1 in each newline's byte
        mask[c] |= ((hit * 0x10204080u) >> 28) << (4 * i);                // gathered into four bits
      }
    }
    return;
  }
#pragma unroll
  for (int c = 0; c < kChunks; ++c) {
    mask[c] = 0;
    for (int i = 0; i < 16; ++i) {
      const int64_t p = p0 + c * 512 + i;
      if (p < n && t[p] == '\n') mask[c] |= 1u << i;
    }
  }
}

__global__ void __launch_bounds__(kCsvThreads) csv_count_kernel(const char* __restrict__ t, int64_t n, int64_t ntiles,
                                                               uint32_t* __restrict__ counts) {
  const bool aligned = (reinterpret_cast<uintptr_t>(t) & 15u) == 0;
  const int64_t tile = blockIdx.x * static_cast<int64_t>(kCsvThreads / 32) + (threadIdx.x >> 5);
  if (tile >= ntiles) return;
  uint32_t mask[kChunks];
  newline_masks(t, n, tile, aligned, mask);
  int c = 0;
#pragma unroll
  for (int i = 0; i < kChunks; ++i) c += __popc(mask[i]);
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0) counts[tile] = static_cast<uint32_t>(c);
}

// one block of 1024 threads, 4096 tiles a step; offs[i] = newlines before tile i; *total = lines
__global__ void __launch_bounds__(1024) csv_scan_kernel(const char* __restrict__ t, int64_t n,
                                                       const uint32_t* __restrict__ counts, int64_t ntiles,
                                                       int64_t* __restrict__ offs, int64_t* __restrict__ ends,
                                                       int64_t ends_cap, int64_t* __restrict__ total) {
  __shared__ uint32_t s_warp[2][32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int64_t before = 0;
  int buf = 0;
  for (int64_t i0 = 0; i0 < ntiles; i0 += 4096, buf ^= 1) {
    const int64_t i = i0 + 4 * tid;
    uint4 c = make_uint4(0, 0, 0, 0);
    if (i + 4 <= ntiles) {
      c = *reinterpret_cast<const uint4*>(counts + i);
    } else {
      if (i < ntiles) c.x = counts[i];
      if (i + 1 < ntiles) c.y = counts[i + 1];
      if (i + 2 < ntiles) c.z = counts[i + 2];
    }
    const uint32_t own = c.x + c.y + c.z + c.w;  // 4096 tiles hold at most 2^24 newlines
    uint32_t x = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[buf][warp] = x;
    __syncthreads();
    uint32_t w = s_warp[buf][lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    const uint32_t ahead = __shfl_sync(0xffffffffu, w, (warp + 31) & 31), all = __shfl_sync(0xffffffffu, w, 31);
    int64_t run = before + (warp ? ahead : 0) + (x - own);
    const uint32_t cs[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i + u < ntiles) {
        offs[i + u] = run;
        run += cs[u];
      }
    before += all;
  }
  if (tid == 0) {
    int64_t lines = before;
    if (n > 0 && t[n - 1] != '\n') {  // a last line without its newline ends at the text's end
      if (lines < ends_cap) ends[lines] = n;
      ++lines;
    }
    *total = lines;
  }
}

__global__ void __launch_bounds__(kCsvThreads) csv_index_kernel(const char* __restrict__ t, int64_t n, int64_t ntiles,
                                                               const int64_t* __restrict__ offs,
                                                               int64_t* __restrict__ ends, int64_t ends_cap) {
  const bool aligned = (reinterpret_cast<uintptr_t>(t) & 15u) == 0;
  const int lane = threadIdx.x & 31;
  const int64_t tile = blockIdx.x * static_cast<int64_t>(kCsvThreads / 32) + (threadIdx.x >> 5);
  if (tile >= ntiles) return;
  uint32_t mask[kChunks];
  newline_masks(t, n, tile, aligned, mask);
  int64_t line = offs[tile];
  // two chunks' counts (at most 512 each) to a scan
#pragma unroll
  for (int c = 0; c < kChunks; c += 2) {
    const uint32_t own = static_cast<uint32_t>(__popc(mask[c])) | static_cast<uint32_t>(__popc(mask[c + 1])) << 16;
    uint32_t x = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    const uint32_t all = __shfl_sync(0xffffffffu, x, 31);
    x -= own;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      int64_t at = line + (u ? (all & 0xFFFFu) + (x >> 16) : (x & 0xFFFFu));
      const int64_t p = tile * kCsvTile + (c + u) * 512 + lane * 16;
      for (uint32_t m = mask[c + u]; m; m &= m - 1, ++at)
        if (at < ends_cap) ends[at] = p + __ffs(static_cast<int>(m)) - 1;
    }
    line += (all & 0xFFFFu) + (all >> 16);
  }
}

// ------------------------------- exact decimal -> binary -------------------------------
constexpr int kCsvFastK = 27;  // 5^27 < 2^63: one-word divisors for 10^-k, k <= 27
struct CsvTables {
  uint64_t p10[20];
  uint64_t dn[kCsvFastK + 1];
  uint64_t v[kCsvFastK + 1];
  int32_t z[kCsvFastK + 1];
  int32_t pad;
};
static_assert(sizeof(CsvTables) % 8 == 0, "copied as 64-bit words");

// Built on the host in exact integer arithmetic.
CsvTables make_csv_tables() {
  CsvTables T{};
  uint64_t p = 1;
  for (int i = 0; i < 20; ++i, p *= 10u) T.p10[i] = p;
  uint64_t f = 1;
  for (int k = 1; k <= kCsvFastK; ++k) {
    f *= 5u;
    const int z = __builtin_clzll(f);
    const uint64_t dn = f << z;
    const unsigned __int128 all = ~static_cast<unsigned __int128>(0);
    T.dn[k] = dn;
    T.z[k] = z;
    T.v[k] = static_cast<uint64_t>(all / dn - (static_cast<unsigned __int128>(1) << 64));
  }
  return T;
}

struct U128 {
  uint64_t lo, hi;
};
__device__ __forceinline__ int bitlen64(uint64_t x) { return x ? 64 - __clzll(static_cast<long long>(x)) : 0; }
__device__ __forceinline__ int bitlen128(const U128& x) { return x.hi ? 64 + bitlen64(x.hi) : bitlen64(x.lo); }
__device__ __forceinline__ bool ge128(const U128& a, const U128& b) { return a.hi != b.hi ? a.hi > b.hi : a.lo >= b.lo; }
__device__ __forceinline__ U128 sub128(const U128& a, const U128& b) {
  U128 r;
  r.lo = a.lo - b.lo;
  r.hi = a.hi - b.hi - (a.lo < b.lo ? 1u : 0u);
  return r;
}
__device__ __forceinline__ U128 shl128(const U128& a, int s) {  // 0 <= s < 128
  if (s == 0) return a;
  if (s >= 64) return U128{0, a.lo << (s - 64)};
  return U128{a.lo << s, (a.hi << s) | (a.lo >> (64 - s))};
}
__device__ __forceinline__ U128 mul64x64(uint64_t a, uint64_t b) { return U128{a * b, __umul64hi(a, b)}; }
__device__ __forceinline__ U128 mul128x10(const U128& a) {  // a < 2^124
  const U128 lo = mul64x64(a.lo, 10u);
  return U128{lo.lo, lo.hi + a.hi * 10u};
}

// Round (q + f) * 2^e2 (0 <= f < 1, f > 0 iff sticky) to t bits, nearest, ties to even, and
// return the IEEE bits of the column type (53: FP64, 24: FP32).  status: kCsvRange when
// the result overflows or would be subnormal.
__device__ uint64_t round_assemble(uint64_t q, bool sticky, int e2, int t, bool neg, uint32_t& status) {
  const int bq = bitlen64(q);  // q > 0
  uint64_t mant;
  if (bq > t) {
    const int sh = bq - t;
    mant = q >> sh;
    const uint64_t rem = q & ((uint64_t(1) << sh) - 1), half = uint64_t(1) << (sh - 1);
    const bool up = rem > half || (rem == half && (sticky || (mant & 1u)));
    mant += up ? 1u : 0u;
    e2 += sh;
    if (mant >> t) {  // carried into a new bit
      mant >>= 1;
      ++e2;
    }
  } else {
    mant = q << (t - bq);  // exact (sticky is 0 here: see the callers)
    e2 -= t - bq;
  }
  const int etop = e2 + t - 1;  // exponent of the leading bit
  const int emax = t == 53 ? 1023 : 127, emin = t == 53 ? -1022 : -126;
  if (etop > emax || etop < emin) {
    status |= kCsvRange;
    return 0;
  }
  if (t == 53) {
    const uint64_t bits = (static_cast<uint64_t>(etop + 1023) << 52) | (mant & ((uint64_t(1) << 52) - 1));
    return bits | (neg ? (uint64_t(1) << 63) : 0);
  }
  const uint32_t bits = (static_cast<uint32_t>(etop + 127) << 23) | static_cast<uint32_t>(mant & ((1u << 23) - 1));
  return bits | (neg ? (1u << 31) : 0u);
}

// M * 10^E correctly rounded to t bits (M > 0, -38 <= E <= 19), as IEEE bits.  T holds
// 10^0 .. 10^19 and, for 1 <= k <= kCsvFastK, 5^k normalised (shifted left until its top
// bit is set) with its reciprocal v = floor((2^128 - 1) / (5^k << z)) - 2^64.
__device__ uint64_t decimal_to_bits(uint64_t M, int E, int t, bool neg, uint32_t& status, const CsvTables& T) {
  if (E >= 0) {
    const U128 P = mul64x64(M, T.p10[E]);  // 10^19 < 2^64, the product < 2^128
    const int bl = bitlen128(P);
    uint64_t q;
    bool sticky = false;
    int e2 = 0;
    if (bl > 64) {
      const int sh = bl - 64;  // 1 .. 63
      q = (P.lo >> sh) | (P.hi << (64 - sh));
      sticky = (P.lo & ((uint64_t(1) << sh) - 1)) != 0;
      e2 = sh;
    } else {
      q = P.lo;
    }
    return round_assemble(q, sticky, e2, t, neg, status);
  }
  const int k = -E, bM = bitlen64(M);
  if (k <= kCsvFastK) {
    // M / 10^k = (M 2^a / 5^k) 2^-(a + k) with a = 63 + bitlen(5^k) - bitlen(M), so that
    // q = floor(M 2^a / 5^k) lies in [2^62, 2^64).  With 5^k normalised to dn = 5^k 2^z,
    // q = floor(u / dn) for u = M 2^(a + z) = M 2^(127 - bitlen(M)) (a 128-bit numerator
    // whose high word is below dn): one division by an invariant word with its
    // precomputed reciprocal (Moller and Granlund 2011) and the exact remainder.
    const uint64_t dn = T.dn[k], v = T.v[k];
    const int bD = 64 - T.z[k];
    const int sh = 127 - bM;  // 63 .. 126
    const uint64_t u1 = sh >= 64 ? M << (sh - 64) : M >> 1;
    const uint64_t u0 = sh >= 64 ? 0 : M << 63;
    const U128 qq = mul64x64(v, u1);
    const uint64_t q0 = qq.lo + u0;
    uint64_t q1 = qq.hi + u1 + (q0 < qq.lo ? 1u : 0u) + 1u;
    uint64_t r = u0 - q1 * dn;
    if (r > q0) {
      q1 -= 1u;
      r += dn;
    }
    if (r >= dn) {
      q1 += 1u;
      r -= dn;
    }
    return round_assemble(q1, r != 0, -(63 + bD - bM + k), t, neg, status);
  }
  // 10^k above 2^64: binary long division, one quotient bit per step
  U128 D{1, 0};
  for (int i = 0; i < k; ++i) D = mul128x10(D);  // 10^38 < 2^127
  const int bD = bitlen128(D);
  const int s = 63 + bD - bM;  // M 2^s / D lies in [2^62, 2^64)
  U128 R = shl128(U128{M, 0}, bD - 1 - bM);  // M < 2^64 < D here: the leading quotient bits are zero
  const int steps = s - (bD - 1 - bM);
  uint64_t q = 0;
  for (int i = 0; i < steps; ++i) {
    R = shl128(R, 1);
    q <<= 1;
    if (ge128(R, D)) {
      R = sub128(R, D);
      q |= 1u;
    }
  }
  return round_assemble(q, (R.lo | R.hi) != 0, -s, t, neg, status);
}

__device__ __forceinline__ bool is_digit(char c) { return c >= '0' && c <= '9'; }

// Parse the field that starts at p (ended by ',' or the line end e) as column type dt and
// store it at dst.  Returns the terminator's position, or -1 (status set) on an error.
__device__ int64_t parse_field(const char* t, int64_t p, int64_t e, int32_t dt, void* dst, uint32_t& status,
                               const CsvTables& T) {
  char c = p < e ? t[p] : ',';
  bool neg = false;
  if (c == '+' || c == '-') {
    neg = c == '-';
    ++p;
    c = p < e ? t[p] : ',';
  }
  if (dt == STATS_I16 || dt == STATS_I32 || dt == STATS_I64) {
    uint64_t v = 0;
    int nd = 0;
    while (c != ',') {
      if (!is_digit(c) || ++nd > STATS_CSV_MAX_DIGITS) {
        status |= kCsvFormat;
        return -1;
      }
      v = v * 10u + static_cast<uint64_t>(c - '0');
      ++p;
      c = p < e ? t[p] : ',';
    }
    if (nd == 0) {
      status |= kCsvFormat;
      return -1;
    }
    const uint64_t lim = dt == STATS_I16 ? 32767u : dt == STATS_I32 ? 2147483647u : 9223372036854775807ull;
    if (v > lim + (neg ? 1u : 0u)) {
      status |= kCsvRange;
      return -1;
    }
    const int64_t x = neg ? static_cast<int64_t>(0 - v) : static_cast<int64_t>(v);
    if (dt == STATS_I16)
      *static_cast<int16_t*>(dst) = static_cast<int16_t>(x);
    else if (dt == STATS_I32)
      *static_cast<int32_t*>(dst) = static_cast<int32_t>(x);
    else
      *static_cast<int64_t*>(dst) = x;
    return p;
  }
  // real: digits [. digits] [e|E [+-] digits]
  uint64_t M = 0;
  int nsig = 0, E = 0, ndig = 0, tz = 0;  // tz: trailing zero digits of M
  bool point = false;
  for (;; ++p, c = p < e ? t[p] : ',') {
    if (c == '.') {
      if (point) break;
      point = true;
      continue;
    }
    if (!is_digit(c)) break;
    ++ndig;
    const int d = c - '0';
    if (nsig == 0 && d == 0) {  // leading zeros
      if (point) --E;
      continue;
    }
    if (nsig < STATS_CSV_MAX_DIGITS) {
      M = M * 10u + static_cast<uint64_t>(d);
      ++nsig;
      tz = d == 0 ? tz + 1 : 0;
      if (point) --E;
    } else if (d != 0) {
      status |= kCsvFormat;  // more significant digits than supported
      return -1;
    } else if (!point) {
      ++E;  // a zero past the kept digits, before the point
    }
  }
  if (ndig == 0) {
    status |= kCsvFormat;
    return -1;
  }
  if (c == 'e' || c == 'E') {
    ++p;
    c = p < e ? t[p] : ',';
    bool eneg = false;
    if (c == '+' || c == '-') {
      eneg = c == '-';
      ++p;
      c = p < e ? t[p] : ',';
    }
    int x = 0, nx = 0;
    for (; is_digit(c); ++p, c = p < e ? t[p] : ',', ++nx) x = x * 10 + (c - '0');
    if (nx == 0 || nx > 4) {
      status |= kCsvFormat;
      return -1;
    }
    E += eneg ? -x : x;
  }
  if (c != ',') {
    status |= kCsvFormat;
    return -1;
  }
  const bool f64 = dt == STATS_F64;
  uint64_t bits = 0;
  if (M == 0) {
    bits = neg ? (f64 ? (uint64_t(1) << 63) : (uint64_t(1) << 31)) : 0;
  } else {
    // the same value with the exponent moved toward the supported range
    if (E < 0 && tz > 0) {  // trailing zeros of M (counted while parsing: no 64-bit remainders)
      const int n = min(tz, -E);
      M /= T.p10[n];
      E += n;
    }
    while (E > 19 && M < 1000000000000000000ull) {
      M *= 10u;
      --E;
    }
    if (E < -38 || E > 19) {
      status |= kCsvFormat;  // outside the supported exponent range
      return -1;
    }
    uint32_t st = 0;
    bits = decimal_to_bits(M, E, f64 ? 53 : 24, neg, st, T);
    if (st) {
      status |= st;
      return -1;
    }
  }
  if (f64)
    *static_cast<uint64_t*>(dst) = bits;
  else
    *static_cast<uint32_t*>(dst) = static_cast<uint32_t>(bits);
  return p;
}

// ------------------------------- eight characters at a time -------------------------------
// The eight bytes at p (the first in the lowest byte).  Two aligned words where both lie inside the
// text; next to its ends byte by byte, with zeros past it.
__device__ __forceinline__ uint64_t load8(const char* t, int64_t p, int64_t n) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(t + p);
  const int sh = static_cast<int>(a & 7u);
  if (p >= sh && p - sh + 16 <= n) {
    const uint64_t* w = reinterpret_cast<const uint64_t*>(a - sh);
    const uint64_t lo = __ldg(w);
    if (sh == 0) return lo;
    return lo >> (8 * sh) | __ldg(w + 1) << (64 - 8 * sh);
  }
  uint64_t v = 0;
  for (int i = 0; i < 8; ++i)
    if (p + i < n) v |= static_cast<uint64_t>(static_cast<unsigned char>(t[p + i])) << (8 * i);
  return v;
}

// Eight digits in a word, the well-known way: a byte is no digit if XOR '0' leaves it above 9, and the digits are
// joined two, four and eight at a time by multiplications with 10 * 2^8 + 1, 100 * 2^16 + 1 and 10000 * 2^32 + 1.
// how many of the eight characters, from the first on, are digits; d: the bytes XOR '0'
__device__ __forceinline__ int leading_digits(uint64_t d) {
  const uint64_t other = (((d & 0x7F7F7F7F7F7F7F7Full) + 0x7676767676767676ull) | d) & 0x8080808080808080ull;
  return other ? (__ffsll(static_cast<long long>(other)) - 1) >> 3 : 8;
}
// value of the first nd (1..8) digits: moved to the high bytes, then digits, pairs and fours joined
__device__ __forceinline__ uint32_t digits_value(uint64_t d, int nd) {
  uint64_t v = d << (64 - 8 * nd);
  v = (v * (10u << 8 | 1u) >> 8) & 0x00FF00FF00FF00FFull;
  v = (v * (100u << 16 | 1u) >> 16) & 0x0000FFFF0000FFFFull;
  return static_cast<uint32_t>(v * (10000ull << 32 | 1ull) >> 32);
}

// A run of digits from p on into v (at most 19 of them kept count of; more overflow v, and the
// caller refuses them).  Returns their number.
__device__ __forceinline__ int digit_run(const char* t, int64_t p, int64_t n, const CsvTables& T, uint64_t& v,
                                         uint64_t& next) {
  int total = 0;
  for (;;) {
    const uint64_t w = load8(t, p + total, n), d = w ^ 0x3030303030303030ull;
    const int nd = leading_digits(d);
    if (nd) v = v * T.p10[nd] + digits_value(d, nd);
    total += nd;
    if (nd < 8) {
      next = w >> (8 * nd);  // the characters that follow the run, the first in the low byte
      return total;
    }
    if (total > 2 * STATS_CSV_MAX_DIGITS) return total;
  }
}

// parse_field for the forms nearly all fields have -- an integer of at most 19 digits; a real of
// digits and a point whose significant digits are at most 19 -- with the same result.  Anything
// else (an exponent, more digits, a stray character) goes to parse_field from its start, which also
// gives the error.
__device__ __forceinline__ int64_t parse_field_fast(const char* t, int64_t n, int64_t p, int64_t e, int32_t dt, void* dst,
                                                    uint32_t& status, const CsvTables& T) {
  const int64_t start = p;
  const char c = p < e ? t[p] : ',';
  const bool neg = c == '-';
  if (neg || c == '+') ++p;
  uint64_t v = 0, next = 0;
  int nd = digit_run(t, p, n, T, v, next);
  p += nd;
  if (dt == STATS_I16 || dt == STATS_I32 || dt == STATS_I64) {
    const bool ends = p == e || (p < e && (next & 0xFF) == ',');
    const uint64_t lim = dt == STATS_I16 ? 32767u : dt == STATS_I32 ? 2147483647u : 9223372036854775807ull;
    if (nd == 0 || nd > STATS_CSV_MAX_DIGITS || !ends || v > lim + (neg ? 1u : 0u))
      return parse_field(t, start, e, dt, dst, status, T);
    const int64_t x = static_cast<int64_t>(neg ? 0 - v : v);
    if (dt == STATS_I16)
      *static_cast<int16_t*>(dst) = static_cast<int16_t>(x);
    else if (dt == STATS_I32)
      *static_cast<int32_t*>(dst) = static_cast<int32_t>(x);
    else
      *static_cast<int64_t*>(dst) = x;
    return p;
  }
  int E = 0, sig = v ? nd : 0;  // digits that v may hold, leading zeros of the integer part left out
  bool plain = nd > 0 && nd <= STATS_CSV_MAX_DIGITS;
  if (p < e && (next & 0xFF) == '.') {
    ++p;
    const int nf = digit_run(t, p, n, T, v, next);
    p += nf;
    E = -nf;
    sig += nf;
    nd += nf;
  }
  plain = plain && sig <= STATS_CSV_MAX_DIGITS && (p == e || (p < e && (next & 0xFF) == ','));
  if (!plain) return parse_field(t, start, e, dt, dst, status, T);
  const bool f64 = dt == STATS_F64;
  uint64_t bits = neg ? (f64 ? (uint64_t(1) << 63) : (uint64_t(1) << 31)) : 0;
  if (v) {
    uint32_t st = 0;
    bits = decimal_to_bits(v, E, f64 ? 53 : 24, neg, st, T);
    if (st) {
      status |= st;
      return -1;
    }
  }
  if (f64)
    *static_cast<uint64_t*>(dst) = bits;
  else
    *static_cast<uint32_t*>(dst) = static_cast<uint32_t>(bits);
  return p;
}

__device__ __forceinline__ int dtype_size(int32_t dt) {
  return dt == STATS_I16 ? 2 : (dt == STATS_I32 || dt == STATS_F32) ? 4 : 8;
}

__global__ void __launch_bounds__(256) csv_parse_kernel(const char* __restrict__ t, int64_t nbytes, CsvScratch S, int k,
                                                       int64_t row_cap, int64_t max_lines,
                                                       const __grid_constant__ CsvTables TP) {
  if (*S.total > max_lines) return;
  __shared__ CsvTables T;
  for (int i = threadIdx.x; i < static_cast<int>(sizeof(CsvTables) / 8); i += blockDim.x)
    reinterpret_cast<uint64_t*>(&T)[i] = reinterpret_cast<const uint64_t*>(&TP)[i];
  __syncthreads();
  const int64_t nl = min(*S.total, S.ends_cap);
  for (int64_t row = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; row < nl;
       row += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    int64_t p = row == 0 ? 0 : S.ends[row - 1] + 1;
    int64_t e = S.ends[row];
    if (e > p && t[e - 1] == '\r') --e;
    uint32_t status = 0;
    const bool store = row < row_cap;
    for (int j = 0; j < k; ++j) {
      const int32_t dt = S.dts[j];
      uint64_t scratch;
      void* dst = store ? static_cast<void*>(static_cast<char*>(S.cols[j]) + row * dtype_size(dt))
                        : static_cast<void*>(&scratch);
      const int64_t f = parse_field_fast(t, nbytes, p, e, dt, dst, status, T);
      if (f < 0) break;
      if (j + 1 < k) {
        if (f >= e) {  // fewer than k fields
          status |= kCsvFormat;
          break;
        }
        p = f + 1;
      }
    }
    if (status) {  // one error bit per line (its parse stops there); the smallest line wins
      atomicOr(S.status, status);
      atomicMin(S.bad, (static_cast<unsigned long long>(row) << 2) | status);
    }
  }
}

size_t pad256(size_t b) { return (b + 255) / 256 * 256; }

}  // namespace

size_t csv_scratch_bytes(int64_t nbytes, int64_t ends_cap, int k) {
  const int64_t ntiles = (nbytes + kCsvTile - 1) / kCsvTile + 1;
  return pad256(4 * ntiles) + pad256(8 * ntiles) + pad256(8 * (ends_cap + 1)) + pad256(sizeof(CsvHead) + 12 * k);
}

void csv_scratch_carve(void* base, int64_t nbytes, int64_t ends_cap, int k, CsvScratch& s) {
  const int64_t ntiles = (nbytes + kCsvTile - 1) / kCsvTile + 1;
  char* b = static_cast<char*>(base);
  s.counts = reinterpret_cast<uint32_t*>(b);
  b += pad256(4 * ntiles);
  s.offs = reinterpret_cast<int64_t*>(b);
  b += pad256(8 * ntiles);
  s.ends = reinterpret_cast<int64_t*>(b);
  s.ends_cap = ends_cap;
  b += pad256(8 * (ends_cap + 1));
  s.head = reinterpret_cast<CsvHead*>(b);
  s.total = &s.head->total;
  s.status = &s.head->status;
  s.bad = &s.head->bad;
  b += sizeof(CsvHead);
  s.cols = reinterpret_cast<void**>(b);
  b += 8 * k;
  s.dts = reinterpret_cast<int32_t*>(b);
}

cudaError_t launch_csv_lines(const char* d_text, int64_t nbytes, const CsvScratch& s, cudaStream_t st) {
  const int64_t ntiles = (nbytes + kCsvTile - 1) / kCsvTile;
  if (ntiles == 0) return cudaMemsetAsync(s.total, 0, sizeof(int64_t), st);
  if (ntiles > 0x7fffffff) return cudaErrorInvalidValue;
  const unsigned blocks = static_cast<unsigned>((ntiles + kCsvThreads / 32 - 1) / (kCsvThreads / 32));
  csv_count_kernel<<<blocks, kCsvThreads, 0, st>>>(d_text, nbytes, ntiles, s.counts);
  csv_scan_kernel<<<1, 1024, 0, st>>>(d_text, nbytes, s.counts, ntiles, s.offs, s.ends, s.ends_cap, s.total);
  csv_index_kernel<<<blocks, kCsvThreads, 0, st>>>(d_text, nbytes, ntiles, s.offs, s.ends, s.ends_cap);
  return cudaGetLastError();
}

cudaError_t launch_csv_parse(const char* d_text, int64_t nbytes, const CsvScratch& s, int k, int64_t row_cap,
                             int64_t max_lines, int sms, cudaStream_t st) {
  const int64_t want = (s.ends_cap + 255) / 256;
  const int grid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(want, int64_t(sms) * 8)));
  static const CsvTables tables = make_csv_tables();
  csv_parse_kernel<<<grid, 256, 0, st>>>(d_text, nbytes, s, k, row_cap, max_lines, tables);
  return cudaGetLastError();
}

}  // namespace ss

// ------------------------------------------------------------------------ host side
using namespace ss;

namespace {

bool valid_dtype(int32_t d) { return d >= STATS_I16 && d <= STATS_F64; }
int host_dtype_bytes(int32_t d) { return d == STATS_I16 ? 2 : (d == STATS_I32 || d == STATS_F32) ? 4 : 8; }

// decimal text of an integer
char* put_int(char* o, int64_t v) {
  char buf[24];
  int n = 0;
  uint64_t u = v < 0 ? 0 - static_cast<uint64_t>(v) : static_cast<uint64_t>(v);
  do {
    buf[n++] = static_cast<char>('0' + u % 10u);
    u /= 10u;
  } while (u);
  if (v < 0) *o++ = '-';
  while (n) *o++ = buf[--n];
  return o;
}

// Format rows [r0, r1) of the columns into out; false if a real value is not finite.
bool format_rows(int p, const int32_t* dt, const void* const* cols, int64_t r0, int64_t r1, std::string& out) {
  out.clear();
  out.reserve(static_cast<size_t>(r1 - r0) * (p * 12 + 8));
  char line[STATS_MAX_P * 28 + 4];
  for (int64_t r = r0; r < r1; ++r) {
    char* o = line;
    for (int j = 0; j < p; ++j) {
      if (j) *o++ = ',';
      switch (dt[j]) {
        case STATS_I16: o = put_int(o, static_cast<const int16_t*>(cols[j])[r]); break;
        case STATS_I32: o = put_int(o, static_cast<const int32_t*>(cols[j])[r]); break;
        case STATS_I64: o = put_int(o, static_cast<const int64_t*>(cols[j])[r]); break;
        case STATS_F32: {
          const float v = static_cast<const float*>(cols[j])[r];
          if (!std::isfinite(v)) return false;
          o += snprintf(o, 24, "%.9g", static_cast<double>(v));
          break;
        }
        default: {
          const double v = static_cast<const double*>(cols[j])[r];
          if (!std::isfinite(v)) return false;
          o += snprintf(o, 28, "%.17g", v);
          break;
        }
      }
    }
    *o++ = '\n';
    out.append(line, static_cast<size_t>(o - line));
  }
  return true;
}

bool write_all(int fd, const char* b, size_t len, off_t off) {
  while (len > 0) {
    const ssize_t w = pwrite(fd, b, len, off);
    if (w <= 0) return false;
    b += w;
    len -= static_cast<size_t>(w);
    off += w;
  }
  return true;
}

// Append rows [0, nrows) of the host columns at *off, formatted by parallel threads.
stats_status append_rows(int fd, off_t* off, int p, const int32_t* dt, const void* const* cols, int64_t nrows) {
  const int nt = static_cast<int>(std::max(1u, std::min(16u, std::thread::hardware_concurrency())));
  const int64_t block = int64_t(1) << 20;
  std::vector<std::string> bufs(nt);
  for (int64_t b0 = 0; b0 < nrows; b0 += block) {
    const int64_t b1 = std::min(nrows, b0 + block);
    std::vector<char> ok(nt, 1);
    std::vector<std::thread> th;
    const int64_t per = (b1 - b0 + nt - 1) / nt;
    for (int i = 0; i < nt; ++i) {
      const int64_t r0 = std::min(b1, b0 + i * per), r1 = std::min(b1, r0 + per);
      th.emplace_back([&, i, r0, r1] { ok[i] = format_rows(p, dt, cols, r0, r1, bufs[i]); });
    }
    for (auto& x : th) x.join();
    for (int i = 0; i < nt; ++i)
      if (!ok[i]) return STATS_EINVAL;
    std::vector<off_t> at(nt);
    for (int i = 0; i < nt; ++i) {
      at[i] = *off;
      *off += static_cast<off_t>(bufs[i].size());
    }
    std::vector<char> wok(nt, 1);
    th.clear();
    for (int i = 0; i < nt; ++i)
      th.emplace_back([&, i] { wok[i] = write_all(fd, bufs[i].data(), bufs[i].size(), at[i]); });
    for (auto& x : th) x.join();
    for (int i = 0; i < nt; ++i)
      if (!wok[i]) return STATS_EIO;
  }
  return STATS_OK;
}

stats_status open_out(const char* path, const char* header, int* fd, off_t* off) {
  *fd = open(path, O_CREAT | O_TRUNC | O_WRONLY, 0644);
  if (*fd < 0) return STATS_EIO;
  *off = 0;
  if (header) {
    std::string h(header);
    h.push_back('\n');
    if (!write_all(*fd, h.data(), h.size(), 0)) return STATS_EIO;
    *off = static_cast<off_t>(h.size());
  }
  return STATS_OK;
}

}  // namespace

extern "C" {

stats_status stats_csv_write(const char* path, int32_t p, const int32_t* dtypes, int64_t nrows,
                             const void* const* hcols, const char* header) {
  if (!path || p < 1 || p > STATS_MAX_P || !dtypes || nrows < 0) return STATS_EINVAL;
  for (int j = 0; j < p; ++j) {
    if (!valid_dtype(dtypes[j])) return STATS_EINVAL;
    if (nrows > 0 && (!hcols || !hcols[j])) return STATS_EINVAL;
  }
  int fd = -1;
  off_t off = 0;
  stats_status st = open_out(path, header, &fd, &off);
  if (st == STATS_OK) st = append_rows(fd, &off, p, dtypes, hcols, nrows);
  if (fd >= 0 && close(fd) != 0 && st == STATS_OK) st = STATS_EIO;
  return st;
}

stats_status stats_csv_write_table1(const char* path, uint64_t seed, uint64_t row0, int64_t nrows, int32_t layout,
                                    int64_t chunk_rows) {
  int32_t dt[STATS_T1_P];
  double lo[STATS_T1_P], hi[STATS_T1_P];
  uint8_t ident[STATS_T1_P];
  if (!path || nrows < 0 || chunk_rows < 0 || stats_table1_config(layout, 1, dt, ident, lo, hi) != STATS_OK)
    return STATS_EINVAL;
  if (chunk_rows == 0) chunk_rows = int64_t(1) << 22;
  chunk_rows = std::max<int64_t>(1, std::min<int64_t>(chunk_rows, std::max<int64_t>(nrows, 1)));
  std::vector<size_t> coff(STATS_T1_P);
  size_t bytes = 0;
  for (int j = 0; j < STATS_T1_P; ++j) {
    coff[j] = bytes;
    bytes += pad256(static_cast<size_t>(chunk_rows) * host_dtype_bytes(dt[j]));
  }
  void* d = nullptr;
  void* h = nullptr;
  if (cudaMalloc(&d, bytes) != cudaSuccess) {
    cudaGetLastError();
    return STATS_ENOMEM;
  }
  if (cudaHostAlloc(&h, bytes, cudaHostAllocDefault) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(d);
    return STATS_ENOMEM;
  }
  std::vector<void*> dcols(STATS_T1_P);
  std::vector<const void*> hcols(STATS_T1_P);
  for (int j = 0; j < STATS_T1_P; ++j) {
    dcols[j] = static_cast<char*>(d) + coff[j];
    hcols[j] = static_cast<char*>(h) + coff[j];
  }
  int fd = -1;
  off_t off = 0;
  stats_status st = open_out(path, "A,B,C,D,E,F,G,H,cotC,I,J,K", &fd, &off);
  for (int64_t r = 0; st == STATS_OK && r < nrows; r += chunk_rows) {
    const int64_t m = std::min(chunk_rows, nrows - r);
    st = stats_gen_table1(seed, row0 + static_cast<uint64_t>(r), m, layout, dcols.data(), nullptr);
    if (st == STATS_OK && cudaMemcpy(h, d, bytes, cudaMemcpyDeviceToHost) != cudaSuccess) st = STATS_ECUDA;
    if (st == STATS_OK) st = append_rows(fd, &off, STATS_T1_P, dt, hcols.data(), m);
  }
  if (fd >= 0 && close(fd) != 0 && st == STATS_OK) st = STATS_EIO;
  cudaFreeHost(h);
  cudaFree(d);
  return st;
}

stats_status stats_csv_parse(const char* d_text, int64_t nbytes, int32_t k, const int32_t* dtypes,
                             void* const* d_cols, int64_t max_rows, int64_t* nrows, int64_t* bad_line,
                             void* stream) {
  if (bad_line) *bad_line = -1;
  if (nrows) *nrows = 0;
  if (nbytes < 0 || k < 1 || k > STATS_MAX_P || !dtypes || !d_cols || max_rows < 0 || (nbytes > 0 && !d_text))
    return STATS_EINVAL;
  for (int j = 0; j < k; ++j)
    if (!valid_dtype(dtypes[j]) || !d_cols[j]) return STATS_EINVAL;
  if (nbytes == 0) return STATS_OK;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t ends_cap = std::min<int64_t>(max_rows, nbytes / 2 + 1);
  void* scratch = nullptr;
  if (cudaMallocAsync(&scratch, csv_scratch_bytes(nbytes, ends_cap, k), st) != cudaSuccess) {
    cudaGetLastError();
    return STATS_ENOMEM;
  }
  CsvScratch S;
  csv_scratch_carve(scratch, nbytes, ends_cap, k, S);
  // one copy in (the error words' start, the columns and their types), one out and one wait: a table of
  // more lines than it may have is left alone by the parse itself
  char in[sizeof(CsvHead) + 12 * STATS_MAX_P];
  const CsvHead start{0, ~0ull, 0u, 0u};
  memcpy(in, &start, sizeof(start));
  memcpy(in + sizeof(start), d_cols, sizeof(void*) * k);
  memcpy(in + sizeof(start) + sizeof(void*) * k, dtypes, sizeof(int32_t) * k);
  CsvHead out{};
  stats_status res = STATS_OK;
  cudaError_t e = cudaMemcpyAsync(S.head, in, sizeof(start) + 12 * k, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = launch_csv_lines(d_text, nbytes, S, st);
  if (e == cudaSuccess) e = launch_csv_parse(d_text, nbytes, S, k, max_rows, max_rows, sms, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&out, S.head, sizeof(out), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess && out.total > max_rows) res = STATS_EINVAL;
  cudaFreeAsync(scratch, st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return STATS_ECUDA;
  }
  if (res != STATS_OK) return res;
  if (out.status) {
    if (bad_line) *bad_line = static_cast<int64_t>(out.bad >> 2);
    return (out.bad & kCsvFormat) ? STATS_EFORMAT : STATS_ERANGE;
  }
  if (nrows) *nrows = out.total;
  return STATS_OK;
}

}  // extern "C"
