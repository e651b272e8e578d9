// k_split.cu -- the numeric phase in split precision: every block product
// A_ik . B_kj is carried out on the tensor cores as a sum of products of
// low-precision slices of the operands (Ozaki-style multi-term products),
// accumulated in FP32; C is formed in FP64:
//
//     C_ij = beta * C_in_ij + alpha * sum_k sum_{(p,q)} A_ik^(p) . B_kj^(q)
//
//   BF16x3: a = a1 + a2 + a3 (three BF16 slices of 8 significant bits each),
//           the six slice products with p + q <= 4 (1-based) are kept;
//   TF32x2: a = a1 + a2 (two TF32 slices of 11 significant bits),
//           the three products a1 b1, a1 b2, a2 b1 are kept.
//
// The slices are cut by integer operations on the FP64 bit pattern
// (truncation: each slice takes the next BITS significant bits of what the
// previous slices left), so no FP64 arithmetic is spent on splitting; the
// filter and the norms stay in FP64 (k_symbolic.cu).
//
// Slice layout. For every block b of r x c values (FP64 offset blk_off[b]),
// the slices live at a fixed multiple of the FP64 offset (no extra offset
// table). An operand is seen as `rows` rows along the k index:
//   "left" layout (the block as a left operand, k = its columns): r rows of
//         c values; "right" layout (as a right operand, k = its rows): c rows
//         (the block's columns) of r values.
// k is cut into 16-byte pieces (8 BF16 or 4 TF32 values, zero past the end),
// and a plane stores the pieces k-piece-major: piece (row, kp) at
// (kp * rows + row) * 16 bytes. Eight consecutive rows of one k-piece, the
// 8 x 8 unit of the tensor cores' fragment loads (ldmatrix), are then 128
// contiguous bytes (no shared-memory bank conflict), and a whole operand (all
// planes) is one contiguous, 16-byte aligned run for a bulk copy.
//   BF16: 3 planes of rows * ceil8(k) halfwords at halfword 24*blk_off[b];
//   TF32: 2 planes of rows * ceil4(k) words at word 8*blk_off[b].
#include <cstdint>

#include "bsm_internal.h"

namespace bsm {

// ---------------------------------------------------------------------------
// Splitting an FP64 value into slices of BITS significant bits (truncation).
// Zeros and FP64 subnormals give zero slices; inf/NaN go to the first slice.
// ---------------------------------------------------------------------------
template <int NS, int BITS>
struct Slices {
  uint32_t s[NS];  // bf16 in the low 16 bits, or tf32 as FP32 bits
};

template <int NS, int BITS>
__device__ __forceinline__ Slices<NS, BITS> split_value(double x) {
  Slices<NS, BITS> out;
#pragma unroll
  for (int q = 0; q < NS; q++) out.s[q] = 0u;
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const uint32_t sign = (uint32_t)(b >> 63);
  const int E = (int)((b >> 52) & 0x7FF);
  if (E == 0) return out;
  if (E == 0x7FF) {  // inf / NaN
    const bool nan = (b & 0xFFFFFFFFFFFFFull) != 0;
    out.s[0] = (BITS == 8) ? ((sign << 15) | 0x7F80u | (nan ? 0x40u : 0u))
                           : ((sign << 31) | 0x7F800000u | (nan ? 0x400000u : 0u));
    return out;
  }
  uint64_t rem = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);  // 53-bit significand
  const int e = E - 1023;  // value = rem * 2^(e - 52)
#pragma unroll
  for (int q = 0; q < NS; q++) {
    if (rem == 0) break;
    const int p = 63 - __clzll((long long)rem);  // leading one
    uint32_t h;
    uint64_t low;
    if (p >= BITS - 1) {
      h = (uint32_t)(rem >> (p - (BITS - 1)));
      low = rem & ((1ull << (p - (BITS - 1))) - 1ull);
    } else {
      h = (uint32_t)(rem << ((BITS - 1) - p));
      low = 0;
    }
    // slice value = h * 2^(e - 52 + p - (BITS-1)), h has BITS bits, top bit set
    const int ef = e - 52 + p + 127;  // biased exponent of the slice
    if (ef >= 1 && ef <= 254) {
      if (BITS == 8)
        out.s[q] = (sign << 15) | ((uint32_t)ef << 7) | (h & 0x7Fu);
      else
        out.s[q] = (sign << 31) | ((uint32_t)ef << 23) | ((h & 0x3FFu) << 13);
    } else if (ef > 254) {  // beyond the 8-bit exponent range: infinity
      out.s[q] = (BITS == 8) ? ((sign << 15) | 0x7F80u) : ((sign << 31) | 0x7F800000u);
      break;
    }
    rem = low;
  }
  return out;
}

// ---------------------------------------------------------------------------
// Split every block of a matrix into the left and/or right slice layouts.
// One warp per block (grid-stride), lanes over the positions of the block
// padded to whole pieces in both directions (ceil8(r) x ceil8(c) for BF16,
// ceil4 for TF32, column-major): each value is split once and its slices are
// written to both layouts; the padding positions write the zeros.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int round_up(int x, int q) { return (x + q - 1) / q * q; }

template <int NS, int BITS, int PIECE, typename T>
__device__ __forceinline__ void split_block(const double *__restrict__ x, int r, int c, int lane,
                                            T *__restrict__ left, T *__restrict__ right) {
  const int rp = round_up(r, PIECE), cp = round_up(c, PIECE);
  const int lplane = r * cp, rplane = c * rp;  // elements per plane
  for (int e = lane; e < rp * cp; e += 32) {
    const int yc = e / rp, xr = e - yc * rp;  // (row xr, column yc), column-major
    const bool in = xr < r && yc < c;
    const Slices<NS, BITS> sl = split_value<NS, BITS>(in ? x[xr + (int64_t)yc * r] : 0.0);
    // left: row xr along k = yc; right: row yc along k = xr; pieces k-major
    const int li = ((yc / PIECE) * r + xr) * PIECE + (yc % PIECE);
    const int ri = ((xr / PIECE) * c + yc) * PIECE + (xr % PIECE);
#pragma unroll
    for (int q = 0; q < NS; q++) {
      if (left && xr < r) left[(int64_t)q * lplane + li] = (T)sl.s[q];
      if (right && yc < c) right[(int64_t)q * rplane + ri] = (T)sl.s[q];
    }
  }
}

__global__ void k_split_bf16x3(const int32_t *__restrict__ row_sizes,
                               const int32_t *__restrict__ col_sizes,
                               const int32_t *__restrict__ blk_row,
                               const int32_t *__restrict__ col_idx,
                               const int64_t *__restrict__ blk_off,
                               const double *__restrict__ vals, const int64_t *__restrict__ hdr,
                               uint16_t *__restrict__ left, uint16_t *__restrict__ right) {
  const int lane = threadIdx.x & 31;
  const int64_t nblk = hdr[0];
  const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t b = w0; b < nblk; b += nw) {
    const int64_t base = kBf16HalfwordsPerValue * blk_off[b];
    split_block<3, 8, 8>(vals + blk_off[b], row_sizes[blk_row[b]], col_sizes[col_idx[b]], lane,
                         left ? left + base : nullptr, right ? right + base : nullptr);
  }
}

__global__ void k_split_tf32x2(const int32_t *__restrict__ row_sizes,
                               const int32_t *__restrict__ col_sizes,
                               const int32_t *__restrict__ blk_row,
                               const int32_t *__restrict__ col_idx,
                               const int64_t *__restrict__ blk_off,
                               const double *__restrict__ vals, const int64_t *__restrict__ hdr,
                               uint32_t *__restrict__ left, uint32_t *__restrict__ right) {
  const int lane = threadIdx.x & 31;
  const int64_t nblk = hdr[0];
  const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t b = w0; b < nblk; b += nw) {
    const int64_t base = kTf32WordsPerValue * blk_off[b];
    split_block<2, 11, 4>(vals + blk_off[b], row_sizes[blk_row[b]], col_sizes[col_idx[b]], lane,
                          left ? left + base : nullptr, right ? right + base : nullptr);
  }
}

cudaError_t launch_split(int precision, const int32_t *row_sizes, const int32_t *col_sizes,
                         const int32_t *blk_row, const int32_t *col_idx, const int64_t *blk_off,
                         const double *vals, const int64_t *hdr, void *left, void *right,
                         int grid, cudaStream_t stream) {
  if (precision == BSM_PREC_SPLIT_BF16X3)
    k_split_bf16x3<<<grid, 256, 0, stream>>>(row_sizes, col_sizes, blk_row, col_idx, blk_off, vals,
                                             hdr, (uint16_t *)left, (uint16_t *)right);
  else
    k_split_tf32x2<<<grid, 256, 0, stream>>>(row_sizes, col_sizes, blk_row, col_idx, blk_off, vals,
                                             hdr, (uint32_t *)left, (uint32_t *)right);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Tensor-core fragments (mma.sync, FP32 accumulation).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mma_bf16_k16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                             uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma_bf16_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(b0));
}

__device__ __forceinline__ void mma_tf32_k8(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                            uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// ---------------------------------------------------------------------------
// Numeric kernels (below). A warp computes one C block at a time, or its
// transpose, whichever needs fewer 16x8 MMA tiles. Operands: L (Mp rows along
// k) and R (Np rows along k), both k-piece-major. Not transposed: L = A_ik (A's
// left layout), R = B_kj (B's right layout); transposed (C^T = B^T A^T): L =
// B_kj^T (B's right layout), R = A_ik^T (A's left layout). A k step is 16 (BF16;
// 8 for a last piece) or 8 (TF32) values of k with all slice products of every
// tile.
//
// Accumulation: the products are summed in FP32 by the tensor cores, a few at
// a time, then added to a running sum kept as an unevaluated pair hi + lo of
// FP32 numbers (TwoSum, error-free), so the long sum over the products of a C
// block loses no more than FP32 rounding of each partial sum; hi + lo is
// formed in FP64 at the end (FP32 -> FP64 is exact).
// ---------------------------------------------------------------------------
// hi + lo += x, exactly (Knuth's TwoSum in FP32, no fused operations).
__device__ __forceinline__ void two_sum_acc(float &hi, float &lo, float x) {
  const float s = __fadd_rn(hi, x);
  const float bp = __fsub_rn(s, hi);
  const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
  hi = s;
  lo = __fadd_rn(lo, err);
}

__device__ __forceinline__ void ldsm_x4(uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3,
                                        uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2(uint32_t &r0, uint32_t &r1, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];\n"
               : "=r"(r0), "=r"(r1)
               : "r"(addr));
}

// ---------------------------------------------------------------------------
// Per-block kernel. The operands' slices go from L1/L2 straight into the MMA's
// registers. Of the four lanes that share a row of an MMA operand, lanes 0 and 1 take
// the halves of a 16-byte piece, lanes 2 and 3 those of the next: their values are the
// MMA's k positions of these lanes (2t, 2t + 1, 2t + 8, 2t + 9 of a BF16 k16 step, t and
// t + 4 of a TF32 k8 step), as an MMA's sum does not depend on the order of its k
// positions if both operands have the same. So two pieces of k are a k step, and eight
// rows of a plane one load instruction over two runs of 128 bytes; nothing is staged.
// (Whole pieces, a 16-byte load a lane over four runs: each quarter of a load touches
// four lines, and the L1 is busy 0.78 of the time. Single words in the order of the
// MMA's registers: the same time. Loads of a step ahead, or 24 warps per SM: registers
// spill, slower.)
//
// The products of a C block follow one another in steps of two pieces, 16 of which are
// looked up at a time (a lane each piece, into shared memory); a product's last step is
// filled up with a piece of zeros. (Steps across products would be fewer, 4.6 instead of
// 6.3 ms below, but would change the order of the roundings: sums stay the bits that the
// products one after another give.) L is the operand on the MMA's 16 rows, R on its 8
// columns; a warp takes a tile of up to 16 x 16:
//   kHalf: up to 8 x 8 (the lower half of the MMA's rows repeats the upper one);
//   kOne:  up to 16 x 8;  kTwo: up to 16 x 16.
// With a second destination in host memory the blocks of a warp's run that follow one
// another in C are gathered and leave in 256-byte stores, which the link needs (a block at a
// time: 141 of its 193 GB/s). Without one (DIRECT) a tile goes from the registers into C:
// numeric phase, gathered -> direct, water of 512 molecules 3.19 -> 3.05 ms, 10000 rows with about
// one product for each C block of 6, 13, 16, 24 1.94 -> 1.64, 0.85 -> 0.78, 0.95 -> 0.78, 2.53 ->
// 2.35 (the ring below 2.27, 0.75, 0.75, 3.27).
//
// Against one bulk copy per operand and product into a ring in shared memory and
// ldmatrix, which cost 45 clocks of an SM per copy; numeric phase: water of 1024
// molecules, BF16x3, values also to host memory 10.4 -> 6.28 ms, without 7.8 -> 6.27;
// amorphous of 600 atoms, TF32x2 8.96 -> 6.87. Bound by the L1 (0.61 of its load slots:
// the runs are not aligned to lines) and the latency of its misses; 16 warps per SM
// issue 1.9 instructions a clock, 24 no more; the MMAs are 0.2 of the time.
// ---------------------------------------------------------------------------
constexpr int kSbWarps = 8;
constexpr int kSbBlocksPerSm = 2;
constexpr int kSbStage = 512;    // values gathered at most
constexpr int kSbCarveout = 60;  // % of an SM's L1 as shared memory: what two blocks need
constexpr int kSbGrab = 8;  // C blocks a warp takes at a time, at most
// Units of work per warp up to which C blocks are split into parts of their tiles (32 x 32
// blocks of 32, BF16x3: 0.151 ms with whole blocks, 0.086 with parts; 8 units gain no more).
constexpr int kSbUnits = 4;

__device__ const uint4 g_zero_pieces[32] = {};  // a piece of zeros for each row

struct SbItem {  // a C block of a warp's run
  const int2 *prods;
  int64_t coff, cin;  // cin: offset of its C_in block, or -1
  int32_t np, m, n, part;  // part: every nparts-th tile from this one on
};
struct SbPiece {  // a piece of k: where row 0's lies in both operands' first planes, and
  const uint4 *a, *b;  // the distance of the planes in rows
};
struct SbOut {  // a tile's element (0, 0) in C and in C_in (null: none), column-major, ld rows
  double *c;
  const double *cin;
  double alpha, beta;
  int ld;
  bool plain;  // alpha = 1 and no C_in
};
struct SbWarp {  // a warp's shared memory
  float2 tile[16 * 16];  // hi and lo of a tile, column-major as in C
  double stage[kSbStage];  // values of finished blocks that follow one another in C
  SbPiece piece[32];
  int32_t pieces[32];  // the product's pieces (0: a piece of zeros)
  SbItem item[kSbGrab];
};

constexpr int kSbFold = 1 << 8;  // in SbWarp::pieces: the sums are folded after the step
// Products summed plainly in FP32 before each compensated fold: a partial sum
// of kFold products carries kFold times the rounding of one, still far below
// the slice truncation error.
constexpr int kFold = 4;

enum SbTile { kHalf, kOne, kTwo };

// One tile, into w.tile: rows l0 to l0 + tl - 1 of L, r0 to r0 + tr - 1 of R (swap: L is
// B). a, b, pc: where the operands of product `lane` start, and its pieces of k (0: none).
// DIRECT: into C (out) instead.
template <int PREC, SbTile TILE, bool DIRECT>
__device__ __forceinline__ void sb_tile(SbWarp &w, const uint4 *a, const uint4 *b, int pc,
                                        const SbItem &it, int l0, int tl, int r0, int tr, bool swap,
                                        const DevMat &A, const DevMat &B,
                                        const uint4 *__restrict__ a_left,
                                        const uint4 *__restrict__ b_right, const SbOut &out, int lane) {
  constexpr bool BF = (PREC == BSM_PREC_SPLIT_BF16X3);
  constexpr int NSL = BF ? 3 : 2, NPQ = BF ? 6 : 3, VPP = BF ? 8 : 4;
  constexpr int64_t kUnit = BF ? 3 : 2;  // pieces per FP64 value of an operand's offset
  constexpr int NT = TILE == kTwo ? 2 : 1;
  // slice products, smallest first: (3,1) (2,2) (1,3) (2,1) (1,2) (1,1); (2,1) (1,2) (1,1)
  constexpr int PA[6] = {BF ? 2 : 1, BF ? 1 : 0, 0, 1, 0, 0};
  constexpr int PB[6] = {0, 1, BF ? 2 : 0, 0, 1, 0};
  const int g = lane >> 2, t = lane & 3;
  const int nl = swap ? it.n : it.m, nr = swap ? it.m : it.n;
  // the lane's rows (past the last one: the last one again)
  const int rl = l0 + min(g, tl - 1), rl8 = l0 + min(g + 8, tl - 1) - rl;
  const int rr = r0 + min(g, tr - 1), rr8 = r0 + min(g + 8, tr - 1) - rr;
  float hi[NT][4], lo[NT][4], acc[NT][4];
#pragma unroll
  for (int nt = 0; nt < NT; nt++)
#pragma unroll
    for (int x = 0; x < 4; x++) hi[nt][x] = lo[nt][x] = acc[nt][x] = 0.f;
  for (int pb = 0; pb < it.np; pb += 32) {
    if (pb > 0) {
      pc = 0;
      if (pb + lane < it.np) {
        const int2 pr = __ldg(it.prods + pb + lane);
        a = a_left + kUnit * A.blk_off[pr.x];
        b = b_right + kUnit * B.blk_off[pr.y];
        pc = (A.col_sizes[A.col_idx[pr.x]] + VPP - 1) / VPP;
      }
    }
    const int even = (pc + 1) & ~1;
    int incl = even;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += y;
    }
    const int slots = __shfl_sync(0xffffffffu, incl, 31);
    // where the product's piece number 0 of the whole batch would be
    const uint4 *a0 = a - (int64_t)(incl - even) * it.m, *b0 = b - (int64_t)(incl - even) * it.n;
#pragma unroll 1
    for (int s0 = 0; s0 < slots; s0 += 32) {
      const int s = s0 + lane;
      int p = 0;  // products that end at or before slot s
#pragma unroll
      for (int step = 16; step; step >>= 1)
        if (__shfl_sync(0xffffffffu, incl, p + step - 1) <= s) p += step;
      SbPiece e;
      e.a = (const uint4 *)__shfl_sync(0xffffffffu, (unsigned long long)a0, p) + s * it.m;
      e.b = (const uint4 *)__shfl_sync(0xffffffffu, (unsigned long long)b0, p) + s * it.n;
      int num = __shfl_sync(0xffffffffu, pc, p);
      const int begin = __shfl_sync(0xffffffffu, incl - even, p);
      // the step of this slot is the last one before a fold: of every kFold-th product
      // and of the last one
      const bool fold = s - begin >= num - 2 && ((p % kFold) == kFold - 1 || pb + p == it.np - 1);
      if (s - begin >= num) e.a = e.b = g_zero_pieces, num = 0;
      if (fold) num |= kSbFold;
      __syncwarp();
      w.piece[lane] = swap ? SbPiece{e.b, e.a} : e;
      w.pieces[lane] = num;
      __syncwarp();
      const int end = min(32, slots - s0);
      struct Raw {  // two pieces of k of both operands
        uint2 l[NSL], l8[NSL], r[NSL][NT];
      };
      auto load = [&](Raw &f, int o) {
        const SbPiece at = w.piece[o + (t >> 1)];
        const int np = w.pieces[o + (t >> 1)] & (kSbFold - 1);
        const uint2 *xl = reinterpret_cast<const uint2 *>(at.a + rl) + (t & 1);
        const uint2 *xr = reinterpret_cast<const uint2 *>(at.b + rr) + (t & 1);
#pragma unroll
        for (int q = 0; q < NSL; q++) {
          f.l[q] = __ldg(xl + 2 * q * np * nl);
          f.l8[q] = TILE == kHalf ? f.l[q] : __ldg(xl + 2 * (q * np * nl + rl8));
          f.r[q][0] = __ldg(xr + 2 * q * np * nr);
          if (TILE == kTwo) f.r[q][NT - 1] = __ldg(xr + 2 * (q * np * nr + rr8));
        }
      };
      auto mma = [&](const Raw &f, bool fold) {
#pragma unroll
        for (int pq = 0; pq < NPQ; pq++)
#pragma unroll
          for (int nt = 0; nt < NT; nt++) {
            const uint2 &x = f.l[PA[pq]], &y = f.l8[PA[pq]], &z = f.r[PB[pq]][nt];
            const uint32_t u[4] = {x.x, y.x, x.y, y.y};
            if (BF)
              mma_bf16_k16(acc[nt], u, z.x, z.y);
            else
              mma_tf32_k8(acc[nt], u, z.x, z.y);
          }
        if (fold) {
#pragma unroll
          for (int nt = 0; nt < NT; nt++)
#pragma unroll
            for (int x = 0; x < 4; x++) {
              two_sum_acc(hi[nt][x], lo[nt][x], acc[nt][x]);
              acc[nt][x] = 0.f;
            }
        }
      };
#pragma unroll 1
      for (int o = 0; o < end; o += 4) {
        Raw f0, f1;
        load(f0, o);
        const bool d0 = w.pieces[o] & kSbFold;
        if (o + 2 < end) {
          load(f1, o + 2);
          const bool d1 = w.pieces[o + 2] & kSbFold;
          mma(f0, d0);
          mma(f1, d1);
        } else {
          mma(f0, d0);
        }
      }
    }
  }
  if (DIRECT) {
#pragma unroll
    for (int nt = 0; nt < NT; nt++)
#pragma unroll
      for (int x = 0; x < (TILE == kHalf ? 2 : 4); x++) {
        const int u = g + (x >> 1) * 8, v = nt * 8 + 2 * t + (x & 1);
        if (u >= tl || v >= tr) continue;
        const int64_t at = swap ? (int64_t)u * out.ld + v : (int64_t)v * out.ld + u;
        // FP32 -> FP64 is exact; hi + lo rounded once in FP64
        double y = (double)hi[nt][x] + (double)lo[nt][x];
        if (!out.plain) {
          y = out.alpha * y;
          if (out.cin) y = fma(out.beta, out.cin[at], y);
        }
        __stcs(out.c + at, y);
      }
    return;
  }
  // the tile as it lies in C: row + rows of the tile * column
  __syncwarp();
  const int ld = swap ? tr : tl;
#pragma unroll
  for (int nt = 0; nt < NT; nt++)
#pragma unroll
    for (int x = 0; x < (TILE == kHalf ? 2 : 4); x++) {
      const int u = g + (x >> 1) * 8, v = nt * 8 + 2 * t + (x & 1);
      if (u < tl && v < tr) w.tile[swap ? u * ld + v : v * ld + u] = make_float2(hi[nt][x], lo[nt][x]);
    }
  __syncwarp();
}

// sel: 0 every C block, 2 those beyond 16 x 16. DIRECT: there is no second destination.
template <int PREC, bool DIRECT>
__global__ void __launch_bounds__(kSbWarps * 32, kSbBlocksPerSm)
    k_numeric_split_blocks(DevMat A, DevMat B, DevOut C, DevMat Cin,
                           const uint4 *__restrict__ a_left, const uint4 *__restrict__ b_right,
                           double alpha, double beta, DevWs ws, const DevStatus *st,
                           const int32_t *__restrict__ items, const int64_t *__restrict__ seg,
                           int sel, int ntiles, unsigned long long *work) {
  if (st->overflow) return;
  constexpr bool BF = (PREC == BSM_PREC_SPLIT_BF16X3);
  constexpr int VPP = BF ? 8 : 4;
  constexpr int64_t kUnit = BF ? 3 : 2;
  extern __shared__ __align__(16) unsigned char smem_sb[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  SbWarp &w = reinterpret_cast<SbWarp *>(smem_sb)[warp];
  int64_t wb = 0, we = st->nblk_c;
  if (seg) wb = seg[0], we = seg[1];
  double *hout = (!DIRECT && C.host_vals && st->nnz_c <= C.host_cap) ? C.host_vals : nullptr;
  const bool plain = (alpha == 1.0 && beta == 0.0);
  // fewer at a time where that would leave warps without work
  const int64_t warps = (int64_t)gridDim.x * kSbWarps;
  // the parts of a C block, a unit of work each
  const int nparts =
      (int)min((int64_t)ntiles, max((int64_t)1, kSbUnits * warps / max((int64_t)1, we - wb)));
  we = wb + (we - wb) * nparts;
  const int64_t share = (we - wb) / (warps * 4);
  const int grab = share >= kSbGrab ? kSbGrab : share < 1 ? 1 : (int)share;

  for (;;) {
    unsigned long long got = 0;
    if (lane == 0) got = atomicAdd(work, (unsigned long long)grab);
    const int64_t base = wb + (int64_t)__shfl_sync(0xffffffffu, got, 0);
    if (base >= we) break;
    const int count = we - base < grab ? (int)(we - base) : grab;
    if (lane < count) {
      const int64_t unit = base + lane - wb, blk = nparts > 1 ? wb + unit / nparts : base + lane;
      const int64_t gb = items ? items[blk] : blk;
      SbItem it;
      it.part = nparts > 1 ? (int)(unit % nparts) : 0;
      const int64_t p0 = ws.prod_ptr[gb];
      it.prods = ws.prods + p0;
      it.np = (int)(ws.prod_ptr[gb + 1] - p0);
      it.m = C.row_sizes[C.blk_row[gb]];
      it.n = C.col_sizes[C.col_idx[gb]];
      it.coff = C.blk_off[gb];
      const int cin = ws.c_cin[gb];
      it.cin = cin >= 0 ? Cin.blk_off[cin] : -1;
      w.item[lane] = it;
    }
    __syncwarp();
    // a block's first products and where their operands lie are loaded while the
    // block before is computed
    int2 pr = make_int2(-1, -1);
    auto products = [&](int x) {
      pr = make_int2(-1, -1);
      if (x < count && lane < w.item[x].np) pr = __ldg(w.item[x].prods + lane);
    };
    const uint4 *a = nullptr, *b = nullptr;
    int pc = 0;
    auto operands = [&]() {
      pc = 0;
      if (pr.x >= 0) {
        a = a_left + kUnit * A.blk_off[pr.x];
        b = b_right + kUnit * B.blk_off[pr.y];
        pc = (A.col_sizes[A.col_idx[pr.x]] + VPP - 1) / VPP;
      }
    };
    products(0);
    operands();
    int64_t first = 0;  // where the staged values start in C, and how many there are
    int held = 0;
    auto flush = [&]() {
      // from the start of the 128-byte line that they begin in
      for (int e = lane - (int)(first & 15); e < held; e += 32)
        if (e >= 0) {
          const double v = w.stage[e];
          __stcs(C.vals + first + e, v);
          if (hout) __stcs(hout + first + e, v);
        }
      held = 0;
      __syncwarp();
    };
    for (int x = 0; x < count; x++) {
      const SbItem &it = w.item[x];
      const int m = it.m, n = it.n;
      const uint4 *ca = a, *cb = b;
      const int cp = pc;
      products(x + 1);
      if (sel == 2 && m <= 16 && n <= 16) {
        operands();
        continue;
      }
      const bool staged = !DIRECT && nparts == 1 && m * n <= kSbStage;
      int number = 0;
      if (held > 0 && (!staged || held + m * n > kSbStage || it.coff != first + held)) flush();
      if (held == 0) first = it.coff;
      // the orientation with fewer MMA tiles
      const bool swap = ((n + 15) >> 4) * ((m + 7) >> 3) < ((m + 15) >> 4) * ((n + 7) >> 3);
      for (int m0 = 0; m0 < m; m0 += 16)
        for (int n0 = 0; n0 < n; n0 += 16) {
          if (nparts > 1 && number++ % nparts != it.part) continue;
          const int tm = min(16, m - m0), tn = min(16, n - n0);
          const int l0 = swap ? n0 : m0, tl = swap ? tn : tm, r0 = swap ? m0 : n0, tr = swap ? tm : tn;
          const double *cinv = it.cin >= 0 ? Cin.vals + it.cin : nullptr;
          const int64_t corner = (int64_t)n0 * m + m0;
          const SbOut out{C.vals + it.coff + corner,
                          cinv ? cinv + corner : nullptr, alpha, beta, m, plain};
          if (tr > 8)
            sb_tile<PREC, kTwo, DIRECT>(w, ca, cb, cp, it, l0, tl, r0, tr, swap, A, B, a_left, b_right, out, lane);
          else if (tl > 8)
            sb_tile<PREC, kOne, DIRECT>(w, ca, cb, cp, it, l0, tl, r0, tr, swap, A, B, a_left, b_right, out, lane);
          else
            sb_tile<PREC, kHalf, DIRECT>(w, ca, cb, cp, it, l0, tl, r0, tr, swap, A, B, a_left, b_right, out, lane);
          if (DIRECT) continue;
          const int dc = 32 / tm, dr = 32 - dc * tm;
          int c = lane / tm, r = lane - c * tm;
          for (int e = lane; e < tm * tn; e += 32) {
            const float2 s = w.tile[e];
            // FP32 -> FP64 is exact; hi + lo rounded once in FP64
            double v = (double)s.x + (double)s.y;
            const int64_t loc = (int64_t)(n0 + c) * m + m0 + r;
            if (!plain) {
              v = alpha * v;
              if (cinv) v = fma(beta, cinv[loc], v);
            }
            if (staged) {
              w.stage[held + (int)loc] = v;
            } else {
              __stcs(C.vals + it.coff + loc, v);
              if (hout) __stcs(hout + it.coff + loc, v);
            }
            r += dr, c += dc;
            if (r >= tm) r -= tm, c++;
          }
          __syncwarp();
        }
      operands();
      if (staged) held += m * n;
    }
    if (held > 0) flush();
    __syncwarp();  // the items are read before the next ones are written
  }
}

// ---------------------------------------------------------------------------
// Chunked kernel: the products of a C block concatenated along k. A warp
// computes one C block at a time (or its transpose, as the per-block kernel
// chooses), for the C blocks whose MMA problem fits 16 x 16. The k pieces of
// the block's products, in ascending k, are staged chunk by chunk into shared
// memory. A chunk holds whole products, at most PCMAX 16-byte pieces of k, and
// each slice plane of L (and of R) is one k-piece-major plane of Mp (Np) rows
// in it, so the MMA loop runs over the chunk's pieces as over one long k
// whatever the products' boundaries: every product's pieces are zero past its
// own k. The copies are 16-byte cp.async from all lanes (one loop per operand
// and product over all its planes), double buffered as in the FP64 packed
// kernel, and the tensor cores' FP32 sums are folded into the compensated
// running sum once per chunk. Per product this leaves the copy loop and a
// table entry; the waits, the fold and the loop control come per chunk.
// ---------------------------------------------------------------------------
constexpr int kCatWarps = 4;
constexpr int kCatMeta = 32;  // product table entries (one batch)

// Bytes of one operand buffer: every plane of up to 16 rows and PCMAX pieces,
// and 256 bytes beyond, which the fragment loads of rows past Mp (or Np) in the
// last plane may touch (their results are never used).
template <int PREC, int PCMAX>
__host__ __device__ constexpr int cat_operand_bytes() {
  return (PREC == BSM_PREC_SPLIT_BF16X3 ? 3 : 2) * 16 * PCMAX * 16 + 256;
}
template <int PREC, int PCMAX>
__host__ __device__ constexpr int cat_warp_bytes() {
  return 2 * 2 * cat_operand_bytes<PREC, PCMAX>() + kCatMeta * (8 + 8 + 4);
}

__device__ __forceinline__ void cpa16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cpa_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

template <int PREC, int PCMAX>
__global__ void __launch_bounds__(kCatWarps * 32)
    k_numeric_split_cat(DevMat A, DevMat B, DevOut C, DevMat Cin, const void *__restrict__ a_left,
                        const void *__restrict__ b_right, double alpha, double beta, DevWs ws,
                        const DevStatus *st, const int32_t *__restrict__ items,
                        const int64_t *__restrict__ seg, unsigned long long *work) {
  if (st->overflow) return;
  constexpr bool BF = (PREC == BSM_PREC_SPLIT_BF16X3);
  constexpr int NSL = BF ? 3 : 2;
  constexpr int VPP = BF ? 8 : 4;  // k values per 16-byte piece
  // a product's k (at most 16 for the small instances, 32 for the others)
  // fits one chunk; the launcher picks the instance by the largest k
  static_assert(PCMAX * VPP >= 16, "a chunk must hold the longest product (k <= 16 or 32)");
  constexpr int64_t kUnit = BF ? 2 * kBf16HalfwordsPerValue : 4 * kTf32WordsPerValue;
  constexpr int OPB = cat_operand_bytes<PREC, PCMAX>();
  extern __shared__ __align__(16) unsigned char smem_cat[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  unsigned char *wbase = smem_cat + warp * cat_warp_bytes<PREC, PCMAX>();
  const unsigned char **meta_a = reinterpret_cast<const unsigned char **>(wbase + 4 * OPB);
  const unsigned char **meta_b = meta_a + kCatMeta;
  int *meta_k = reinterpret_cast<int *>(meta_b + kCatMeta);  // pieces of k
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(wbase);
  // which 8 x 8 piece (rows 0-7 or 8-15, k piece 0 or 1 of the step) this lane
  // addresses in ldmatrix: "a" order for the left operand, "b" for the right one
  const int ra = (lane & 7) + ((lane >> 3) & 1) * 8, pa = lane >> 4;
  const int rb_ = (lane & 7) + (lane >> 4) * 8, pb = (lane >> 3) & 1;
  int64_t wb = 0, we = st->nblk_c;
  if (seg) {
    wb = seg[0];
    we = seg[1];
  }
  const bool plain = (alpha == 1.0 && beta == 0.0);
  double *hout = (C.host_vals && st->nnz_c <= C.host_cap) ? C.host_vals : nullptr;

  for (;;) {
    unsigned long long got = 0;
    if (lane == 0) got = atomicAdd(work, 1ull);
    const int64_t w = wb + (int64_t)__shfl_sync(0xffffffffu, got, 0);
    if (w >= we) break;
    const int64_t gb = items ? items[w] : w;
    const int i = C.blk_row[gb], j = C.col_idx[gb];
    const int m = C.row_sizes[i], n = C.col_sizes[j];
    const int tiles_n = ((m + 15) >> 4) * ((n + 7) >> 3);
    const int tiles_t = ((n + 15) >> 4) * ((m + 7) >> 3);
    const bool tr = tiles_t < tiles_n;
    const int Mp = tr ? n : m, Np = tr ? m : n;
    if (Mp > 16 || Np > 16) continue;  // the per-block kernel's
    const bool two = Np > 8;
    const int64_t p0 = ws.prod_ptr[gb], p1 = ws.prod_ptr[gb + 1];
    // chunk plane strides of L (Mp rows) and R (Np rows)
    const uint32_t lpl = (uint32_t)(Mp * PCMAX * 16), rpl = (uint32_t)(Np * PCMAX * 16);
    float hi[2][4], lo[2][4], acc[2][4];
#pragma unroll
    for (int nt = 0; nt < 2; nt++)
#pragma unroll
      for (int x = 0; x < 4; x++) hi[nt][x] = lo[nt][x] = acc[nt][x] = 0.f;

    // product cursor: the next product to stage and the table batch holding it
    int64_t pq = p0, tbase = p0;
    int tcount = 0;
    // all planes of one operand of a product (rows x pk pieces each,
    // contiguous, planes one after another) into the chunk at piece poff
    auto copy_operand = [&](uint32_t dst, uint32_t plane, const unsigned char *src, int rows, int pk,
                            int poff) {
      const int U = rows * pk;  // 16-byte units of one plane
      const uint32_t d0 = dst + 16u * (uint32_t)(poff * rows);
      for (int u = lane; u < NSL * U; u += 32) {
        const int q = (u >= U) + ((NSL == 3 && u >= 2 * U) ? 1 : 0);
        cpa16(d0 + (uint32_t)q * plane + 16u * (uint32_t)(u - q * U), src + 16 * (int64_t)u);
      }
    };
    // stage whole products into buffer buf while they fit; returns the pieces
    auto fill = [&](int buf) -> int {
      const uint32_t dL = sbase + (uint32_t)(buf * 2 * OPB), dR = dL + (uint32_t)OPB;
      int poff = 0;
      while (pq < p1) {
        if (pq == tbase + tcount) {  // the next batch of the product table
          tbase = pq;
          tcount = (p1 - pq < kCatMeta) ? (int)(p1 - pq) : kCatMeta;
          __syncwarp();  // every lane is past its reads of the old batch
          if (lane < tcount) {
            const int2 pr = ws.prods[pq + lane];
            meta_a[lane] = static_cast<const unsigned char *>(a_left) + kUnit * A.blk_off[pr.x];
            meta_b[lane] = static_cast<const unsigned char *>(b_right) + kUnit * B.blk_off[pr.y];
            meta_k[lane] = (A.col_sizes[A.col_idx[pr.x]] + VPP - 1) / VPP;
          }
          __syncwarp();
        }
        const int e = (int)(pq - tbase);
        const int pk = meta_k[e];
        if (pk > PCMAX) {  // longer than a chunk (the launcher rules it out): error, block skipped
          if (lane == 0) atomicOr(const_cast<int32_t *>(&st->error), 1);
          pq = p1;
          break;
        }
        if (poff + pk > PCMAX) break;
        // not transposed: L = A_ik (left layout, m rows), R = B_kj (right layout, n rows)
        const unsigned char *sa = meta_a[e], *sb = meta_b[e];
        copy_operand(dL, lpl, tr ? sb : sa, Mp, pk, poff);
        copy_operand(dR, rpl, tr ? sa : sb, Np, pk, poff);
        poff += pk;
        pq++;
      }
      return poff;
    };

    int cur = fill(0);
    cpa_commit();
    for (int ch = 0;; ch++) {
      const int buf = ch & 1;
      const int nxt = (pq < p1) ? fill(buf ^ 1) : 0;
      cpa_commit();
      cpa_wait<1>();  // the current chunk has landed
      __syncwarp();
      const uint32_t sL = sbase + (uint32_t)(buf * 2 * OPB), sR = sL + (uint32_t)OPB;
      const uint32_t adL = sL + 16u * (uint32_t)(pa * Mp + ra);
      const uint32_t adR = sR + 16u * (uint32_t)(pb * Np + rb_);
      const uint32_t adR2 = sR + 16u * (uint32_t)ra;  // "a" order on R (single pieces)
      if (BF) {
        // slice products, smallest first: (3,1) (2,2) (1,3) (2,1) (1,2) (1,1)
        constexpr int PA[6] = {2, 1, 0, 1, 0, 0};
        constexpr int PB[6] = {0, 1, 2, 0, 1, 0};
        for (int p = 0; p < cur; p += 2) {
          const uint32_t koL = 16u * (uint32_t)(p * Mp), koR = 16u * (uint32_t)(p * Np);
          if (cur - p == 1) {  // one piece left: m16n8k8
            uint32_t a[3][2], b[3][2];
#pragma unroll
            for (int q3 = 0; q3 < 3; q3++) {
              ldsm_x2(a[q3][0], a[q3][1], adL + q3 * lpl + koL);
              ldsm_x2(b[q3][0], b[q3][1], adR2 + q3 * rpl + koR);
            }
#pragma unroll
            for (int x = 0; x < 6; x++) {
              mma_bf16_k8(acc[0], a[PA[x]][0], a[PA[x]][1], b[PB[x]][0]);
              if (two) mma_bf16_k8(acc[1], a[PA[x]][0], a[PA[x]][1], b[PB[x]][1]);
            }
          } else {
            uint32_t a[3][4], b[3][4];
#pragma unroll
            for (int q3 = 0; q3 < 3; q3++) {
              ldsm_x4(a[q3][0], a[q3][1], a[q3][2], a[q3][3], adL + q3 * lpl + koL);
              ldsm_x4(b[q3][0], b[q3][1], b[q3][2], b[q3][3], adR + q3 * rpl + koR);
            }
#pragma unroll
            for (int x = 0; x < 6; x++) {
              mma_bf16_k16(acc[0], a[PA[x]], b[PB[x]][0], b[PB[x]][1]);
              if (two) mma_bf16_k16(acc[1], a[PA[x]], b[PB[x]][2], b[PB[x]][3]);
            }
          }
        }
      } else {
        // (2,1) (1,2) (1,1)
        constexpr int PA[3] = {1, 0, 0};
        constexpr int PB[3] = {0, 1, 0};
        for (int p = 0; p < cur; p += 2) {
          const uint32_t koL = 16u * (uint32_t)(p * Mp), koR = 16u * (uint32_t)(p * Np);
          uint32_t a[2][4], b[2][4];
          if (cur - p == 1) {  // one piece left: the other half of the k step is zero
#pragma unroll
            for (int q2 = 0; q2 < 2; q2++) {
              ldsm_x2(a[q2][0], a[q2][1], adL + q2 * lpl + koL);
              ldsm_x2(b[q2][0], b[q2][2], adR2 + q2 * rpl + koR);
              a[q2][2] = a[q2][3] = b[q2][1] = b[q2][3] = 0u;
            }
          } else {
#pragma unroll
            for (int q2 = 0; q2 < 2; q2++) {
              ldsm_x4(a[q2][0], a[q2][1], a[q2][2], a[q2][3], adL + q2 * lpl + koL);
              ldsm_x4(b[q2][0], b[q2][1], b[q2][2], b[q2][3], adR + q2 * rpl + koR);
            }
          }
#pragma unroll
          for (int x = 0; x < 3; x++) {
            mma_tf32_k8(acc[0], a[PA[x]], b[PB[x]][0], b[PB[x]][1]);
            if (two) mma_tf32_k8(acc[1], a[PA[x]], b[PB[x]][2], b[PB[x]][3]);
          }
        }
      }
      // the chunk's FP32 partial sums into the compensated running sum
#pragma unroll
      for (int nt = 0; nt < 2; nt++)
#pragma unroll
        for (int x = 0; x < 4; x++) {
          two_sum_acc(hi[nt][x], lo[nt][x], acc[nt][x]);
          acc[nt][x] = 0.f;
        }
      __syncwarp();  // the buffer is read before it is filled again
      if (nxt == 0) break;
      cur = nxt;
    }
    cpa_wait<0>();
    __syncwarp();

    const int cin = ws.c_cin[gb];
    const double *cinv = (cin >= 0) ? Cin.vals + Cin.blk_off[cin] : nullptr;
    double *out = C.vals + C.blk_off[gb];
    double *hblk = hout ? hout + C.blk_off[gb] : nullptr;
#pragma unroll
    for (int nt = 0; nt < 2; nt++)
#pragma unroll
      for (int x = 0; x < 4; x++) {
        const int rr = g + ((x >> 1) << 3);
        const int cc = nt * 8 + 2 * t + (x & 1);
        if (rr < Mp && cc < Np) {
          const int row = tr ? cc : rr, col = tr ? rr : cc;
          const int64_t e = (int64_t)col * m + row;
          // FP32 -> FP64 is exact; hi + lo rounded once in FP64
          double v = (double)hi[nt][x] + (double)lo[nt][x];
          if (!plain) {
            v = alpha * v;
            if (cinv) v = fma(beta, cinv[e], v);
          }
          out[e] = v;
          if (hblk) hblk[e] = v;
        }
      }
  }
}

cudaError_t launch_numeric_split(int precision, int sizes, DevMat A, DevMat B, DevOut C,
                                 DevMat Cin, const void *a_left, const void *b_right, double alpha,
                                 double beta, DevWs ws, const DevStatus *st, const int32_t *items,
                                 const int64_t *seg, int max_m, int max_n, int nsm,
                                 unsigned long long *work, cudaStream_t stream) {
  const int ntiles = ((max_m + 15) / 16) * ((max_n + 15) / 16);
  const size_t smem = kSbWarps * sizeof(SbWarp);
  const int grid = nsm * kSbBlocksPerSm;
  const uint4 *l = static_cast<const uint4 *>(a_left), *r = static_cast<const uint4 *>(b_right);
  const bool direct = !C.host_vals;
#define BSM_SPLIT_BLOCKS(P, D)                                                            \
  k_numeric_split_blocks<P, D><<<grid, kSbWarps * 32, smem, stream>>>(                    \
      A, B, C, Cin, l, r, alpha, beta, ws, st, items, seg, sizes, ntiles, work)
  if (precision == BSM_PREC_SPLIT_BF16X3) {
    if (direct) BSM_SPLIT_BLOCKS(BSM_PREC_SPLIT_BF16X3, true);
    else BSM_SPLIT_BLOCKS(BSM_PREC_SPLIT_BF16X3, false);
  } else {
    if (direct) BSM_SPLIT_BLOCKS(BSM_PREC_SPLIT_TF32X2, true);
    else BSM_SPLIT_BLOCKS(BSM_PREC_SPLIT_TF32X2, false);
  }
#undef BSM_SPLIT_BLOCKS
  return cudaGetLastError();
}

// Chunk capacity (16-byte pieces of k) of the chunked instances: the smaller
// where every k is at most 16 (the water blocks), the larger for k up to 32.
// Smaller chunks leave more warps per SM, which this kernel needs (water2048,
// BF16x3: 8 pieces 29.0 ms, 4 pieces 17.8 ms, 2 pieces 17.6 ms; TF32x2: 8
// pieces 23.4 ms, 4 pieces 18.8 ms).
constexpr int kCatPiecesBf16Small = 2, kCatPiecesBf16 = 4;
constexpr int kCatPiecesTf32Small = 4, kCatPiecesTf32 = 8;
template <int PREC, int PCMAX>
static const void *cat_fn() {
  return (const void *)k_numeric_split_cat<PREC, PCMAX>;
}

cudaError_t launch_numeric_split_cat(int precision, DevMat A, DevMat B, DevOut C, DevMat Cin,
                                     const void *a_left, const void *b_right, double alpha,
                                     double beta, DevWs ws, const DevStatus *st,
                                     const int32_t *items, const int64_t *seg, int smax, int nsm,
                                     unsigned long long *work, cudaStream_t stream) {
  const bool bf = precision == BSM_PREC_SPLIT_BF16X3, small = smax <= 16;
  constexpr int BF = BSM_PREC_SPLIT_BF16X3, TF = BSM_PREC_SPLIT_TF32X2;
  const void *fn = bf ? (small ? cat_fn<BF, kCatPiecesBf16Small>() : cat_fn<BF, kCatPiecesBf16>())
                      : (small ? cat_fn<TF, kCatPiecesTf32Small>() : cat_fn<TF, kCatPiecesTf32>());
  const size_t smem =
      (size_t)kCatWarps * (bf ? (small ? cat_warp_bytes<BF, kCatPiecesBf16Small>() : cat_warp_bytes<BF, kCatPiecesBf16>())
                              : (small ? cat_warp_bytes<TF, kCatPiecesTf32Small>() : cat_warp_bytes<TF, kCatPiecesTf32>()));
  int per_sm = 1;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kCatWarps * 32, smem);
  if (e != cudaSuccess) return e;
  const int grid = nsm * (per_sm > 0 ? per_sm : 1);
#define BSM_SPLIT_CAT(P, PC)                                                              \
  k_numeric_split_cat<P, PC><<<grid, kCatWarps * 32, smem, stream>>>(A, B, C, Cin, a_left, \
                                                                    b_right, alpha, beta, ws, \
                                                                    st, items, seg, work)
  if (bf) {
    if (small) BSM_SPLIT_CAT(BF, kCatPiecesBf16Small);
    else BSM_SPLIT_CAT(BF, kCatPiecesBf16);
  } else {
    if (small) BSM_SPLIT_CAT(TF, kCatPiecesTf32Small);
    else BSM_SPLIT_CAT(TF, kCatPiecesTf32);
  }
#undef BSM_SPLIT_CAT
  return cudaGetLastError();
}

cudaError_t numeric_split_init() {
  {
    constexpr int BF = BSM_PREC_SPLIT_BF16X3, TF = BSM_PREC_SPLIT_TF32X2;
    const void *fn[4] = {cat_fn<BF, kCatPiecesBf16Small>(), cat_fn<BF, kCatPiecesBf16>(),
                         cat_fn<TF, kCatPiecesTf32Small>(), cat_fn<TF, kCatPiecesTf32>()};
    const int bytes[4] = {kCatWarps * cat_warp_bytes<BF, kCatPiecesBf16Small>(),
                          kCatWarps * cat_warp_bytes<BF, kCatPiecesBf16>(),
                          kCatWarps * cat_warp_bytes<TF, kCatPiecesTf32Small>(),
                          kCatWarps * cat_warp_bytes<TF, kCatPiecesTf32>()};
    for (int x = 0; x < 4; x++) {
      cudaError_t e = cudaFuncSetAttribute(fn[x], cudaFuncAttributeMaxDynamicSharedMemorySize, bytes[x]);
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(fn[x], cudaFuncAttributePreferredSharedMemoryCarveout, 100);
      if (e != cudaSuccess) return e;
    }
  }
  // the per-block kernel's operands come through L1: no more shared memory than its own
  for (const void *fn : {(const void *)k_numeric_split_blocks<BSM_PREC_SPLIT_BF16X3, false>,
                         (const void *)k_numeric_split_blocks<BSM_PREC_SPLIT_BF16X3, true>,
                         (const void *)k_numeric_split_blocks<BSM_PREC_SPLIT_TF32X2, false>,
                         (const void *)k_numeric_split_blocks<BSM_PREC_SPLIT_TF32X2, true>}) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         kSbCarveout);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)(kSbWarps * sizeof(SbWarp)));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace bsm
