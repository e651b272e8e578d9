// digits.cuh -- FP64 blocks as signed base-256 digits (bsm_internal.h has the
// layout): what the symbolic fill pass writes and the digit kernel reads.
#pragma once

#include "bsm_internal.h"

namespace bsm {

__host__ __device__ __forceinline__ int64_t digit_base(int64_t off, int64_t b, const DigitSide &o) {
  return kDigitZeros + (off * o.mul >> 6) + b * o.pad;
}

// X + 128 * (1 + 256 + ... + 256^7): byte i (from the top) is digit d_i + 128.
// field: the exponent field of the row's largest value, less 8 per class; zero: no
// scale, the digits are zeros. In integers: x = f * 2^(e - 1075) with a 53-bit f,
// X = f * 2^(e - field + 9) rounded to nearest.
__device__ __forceinline__ uint64_t digit_word(double x, int field) {
  const uint64_t bias = 0x8080808080808080ull;
  const int64_t b = __double_as_longlong(x);
  const int e = (int)((uint64_t)b >> 52) & 0x7FF;
  const int up = e - field + 9;  // <= 9
  if (e == 0 || up < -54 || up > 9 || field == 0) return bias;
  uint64_t f = ((uint64_t)b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  if (up >= 0) {
    f <<= up;
  } else {
    const uint64_t h = f >> (-up - 1);  // and the bit below, for rounding
    f = (h >> 1) + (h & 1);
    // a tie goes up: half a unit of 2^-62 of the scale either way
  }
  return (b < 0 ? (uint64_t)0 - f : f) + bias;
}

// |X| in units of 2^48, rounded up.
__device__ __forceinline__ int digit_top(uint64_t word) {
  const int64_t x = (int64_t)(word - 0x8080808080808080ull);
  return (int)((uint64_t)((x < 0 ? -x : x) + ((1ll << 48) - 1)) >> 48);
}

// A sum of these (below 2^30) over 2^14 in 7 bits: rounded up to two bits behind the leading
// one, as an FP32 number's exponent (2^-15, which stands for less too, to 2^16) and mantissa.
__device__ __forceinline__ uint32_t digit_sum_code(uint32_t sum) {
  const float f = fmaxf(__uint2float_ru(sum) * 0x1p-14f, 0x1p-15f);
  return ((__float_as_uint(f) + (1u << 21) - 1) >> 21) - (112u << 2);
}
__device__ __forceinline__ float digit_sum_of(uint32_t code) {
  return __uint_as_float((code + (112u << 2)) << 21);
}

__device__ __forceinline__ int digit_field(double x) {
  const int f = (int)(((uint32_t)__double2hiint(x) >> 20) & 0x7FF);
  return f ? f : (x != 0.0 ? 1 : 0);
}

// Two bytes of a word (sel: byte, 4, byte, 4) as FP16 integers: u = d + 128 below
// the exponent of 1024 is 1024 + u; minus 1152.
__device__ __forceinline__ uint32_t digit_half2(uint32_t word, uint32_t sel) {
  uint32_t h = __byte_perm(word, 0x64646464u, sel);
  asm("add.f16x2 %0, %0, %1;\n" : "+r"(h) : "r"(0xE480E480u));
  return h;
}

// The unit of two values, from their digit words.
__device__ __forceinline__ uint4 digit_unit(uint64_t x, uint64_t y) {
  const uint32_t xh = (uint32_t)(x >> 32), yh = (uint32_t)(y >> 32);
  const uint32_t xl = (uint32_t)x, yl = (uint32_t)y;
  return make_uint4(__byte_perm(xh, yh, 0x6273), __byte_perm(xh, yh, 0x4051),
                    __byte_perm(xl, yl, 0x6273), __byte_perm(xl, yl, 0x4051));
}

// One layout of a block: element (r, k) at r * rs + k * ks, `rows` rows, k up to s
// (rs = 1, ks = rows; or rs = s, ks = 1). seg: 2 kDigitMaxRows words of the warp's own.
__device__ __forceinline__ void digit_layout(const double *__restrict__ x, int rows, int s, int rs,
                                             int ks, const DigitSide &o, int64_t first, int64_t b,
                                             int64_t base, int32_t *seg, int lane) {
  const int octets = (s + 7) >> 3;
  const int32_t *expo = o.expo + first;
  uint4 *units = o.units + base;
  bool outside = rows > kDigitMaxRows || octets > kDigitMaxOctets;
  int cls = 0;
  uint32_t most = 0;  // the largest sum of a row's absolute values, in 2^-14 of its scale
  if (!outside) {
    // the largest exponent field of each row of the block
    int32_t *sum = seg + kDigitMaxRows;
    for (int r = lane; r < rows; r += 32) seg[r] = sum[r] = 0;
    __syncwarp();
    const int len = rows * s;
    for (int z = lane; z < len; z += 32) {  // in the order of the values
      const int hi = (int)((uint32_t)z / (uint32_t)(rs == 1 ? rows : s));
      const int lo = z - hi * (rs == 1 ? rows : s);
      atomicMax(&seg[rs == 1 ? lo : hi], digit_field(__ldg(x + z)));
    }
    __syncwarp();
    int room = 8 * kDigitMaxClass;  // bits that every row of the block leaves free
    for (int r = lane; r < rows; r += 32) {
      const int f = seg[r], field = expo[r];
      outside |= f && (field < kDigitExpLo || field > kDigitExpHi);
      if (f) room = min(room, field - f);
    }
    room = __reduce_min_sync(0xffffffffu, room);
    cls = room >> 3;
    for (int r = lane; r < rows; r += 32)
      outside |= seg[r] && seg[r] < expo[r] - 8 * cls - kDigitRange;
    outside = __any_sync(0xffffffffu, outside);
    const int total = 4 * octets * rows;
    for (int z = lane; z < total && !outside; z += 32) {
      const int q = (int)((uint32_t)z / (uint32_t)rows), r = z - q * rows;  // values 2 q, 2 q + 1 of row r
      const double *p = x + (int64_t)r * rs + (int64_t)(2 * q) * ks;
      const double v0 = (2 * q < s) ? __ldg(p) : 0.0;
      const double v1 = (2 * q + 1 < s) ? __ldg(p + ks) : 0.0;
      const int field = seg[r] ? expo[r] - 8 * cls : 0;
      const uint64_t w0 = digit_word(v0, field), w1 = digit_word(v1, field);
      units[((q >> 2) * rows + r) * 4 + (q & 3)] = digit_unit(w0, w1);
      atomicAdd(&sum[r], digit_top(w0) + digit_top(w1));
    }
    __syncwarp();
    for (int r = lane; r < rows; r += 32) most = max(most, (uint32_t)sum[r]);
    most = __reduce_max_sync(0xffffffffu, most);
  }
  outside = __any_sync(0xffffffffu, outside);
  if (lane == 0)
    o.meta[b] = make_uint2((uint32_t)base,
                           outside ? kDigitOutside
                                   : (uint32_t)octets | (uint32_t)(8 * octets - s) << kDigitPadAt |
                                         (uint32_t)cls << kDigitClassAt |
                                         digit_sum_code(most) << kDigitSumAt);
}

// The digits of M as a left and / or right operand, one warp per block.
__device__ __forceinline__ void digits_of(const DevMat &M, const DigitSide *left,
                                          const DigitSide *right, int32_t *seg, int64_t w0,
                                          int64_t nw, int lane) {
  const int64_t nblk = M.hdr[0];
  for (int64_t b = w0; b < nblk; b += nw) {
    const int i = M.blk_row[b], j = M.col_idx[b];
    const int m = M.row_sizes[i], n = M.col_sizes[j];
    const int64_t off = M.blk_off[b];
    const double *x = M.vals + off;
    if (left)
      digit_layout(x, m, n, 1, m, *left, left->first[i], b, digit_base(off, b, *left), seg, lane);
    if (right)
      digit_layout(x, n, m, m, 1, *right, right->first[j], b, digit_base(off, b, *right), seg,
                   lane);
  }
}

}  // namespace bsm
