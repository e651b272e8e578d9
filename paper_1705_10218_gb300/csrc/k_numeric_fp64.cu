// k_numeric_fp64.cu -- the numeric phase in FP64: every C block accumulates
// its kept block products A_ik . B_kj (grouped and ordered by the symbolic
// phase, ascending k) in registers and is written once:
//
//     C_ij = beta * C_in_ij + alpha * sum_k A_ik . B_kj      (Sec. 2, Alg. 1)
//
// One warp owns one C block at a time and writes it once; no atomics. The
// kernels:
//   t16: 16 x 16 output tiles and k-chunks of 16; the operands of a (product,
//        chunk) step are copied to shared memory in their own layout (a
//        contiguous copy when a block fits one tile), and the next step's
//        operands are already in flight in registers while the current one is
//        multiplied. The (A offset, B offset, k) of up to 32 products are read
//        at once, one per lane, and handed out with warp shuffles. Compiled for
//        2 or 3 thread blocks of 8 warps per SM; C blocks are taken one at a
//        time from a work counter.
//   t32: 32 x 32 output tiles, synchronous staging, 4 warps per block.
//   pk:  "packed" lane slots for tiles of up to 16 x 16: a lane slot is a pair
//        (output element, k-group), so a tile of te elements is computed by
//        te * G slots in nT passes of 32 lanes, with nT and G chosen per tile
//        shape so that te * G nearly fills 32 * nT (13 x 5: 65 elements, 7
//        groups in 15 passes, 95% of the slots useful, where one element per
//        slot uses 68%). The products of a C block are concatenated along k
//        (the C block is one GEMM over the concatenated k), staged in chunks
//        with 8-byte asynchronous copies, double buffered; group g sums the
//        k positions congruent to g mod G, and the G partial sums of an
//        element are added in group order at the end.
//   dg:  the products on the tensor cores, from digits of the operands (below).
// All take an optional work list (C block indices, e.g. one shape class) and
// its [begin, end) range in device memory.
#include <algorithm>
#include <cstdlib>

#include "bsm_internal.h"
#include "digits.cuh"

namespace bsm {

// ----------------------------------------------------------------------------
// t32
// ----------------------------------------------------------------------------
constexpr int kNumWarps = 4;       // warps per thread block
constexpr int kLdA = kTile;        // sA[l * kLdA + r]
constexpr int kLdB = kTile + 1;    // sB[c * kLdB + l]
constexpr int kWarpSmem = kTile * kLdA + kTile * kLdB;  // doubles per warp

__device__ __forceinline__ void work_range(const DevStatus *st, const int64_t *seg, int64_t &b,
                                           int64_t &e) {
  if (seg) {
    b = seg[0];
    e = seg[1];
  } else {
    b = 0;
    e = st->nblk_c;
  }
}

__global__ void __launch_bounds__(kNumWarps * 32)
    k_numeric_fp64_t32(DevMat A, DevMat B, DevOut C, DevMat Cin, double alpha, double beta,
                       DevWs ws, const DevStatus *st, const int32_t *items, const int64_t *seg) {
  if (st->overflow) return;
  extern __shared__ double smem_num[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double *sA = smem_num + warp * kWarpSmem;
  double *sB = sA + kTile * kLdA;
  int64_t wb, we;
  work_range(st, seg, wb, we);
  const int64_t nwarp = (int64_t)gridDim.x * kNumWarps;

  for (int64_t w = wb + (int64_t)blockIdx.x * kNumWarps + warp; w < we; w += nwarp) {
    const int64_t g = items ? items[w] : w;
    const int i = C.blk_row[g], j = C.col_idx[g];
    const int m = C.row_sizes[i], n = C.col_sizes[j];
    const int64_t p0 = ws.prod_ptr[g], p1 = ws.prod_ptr[g + 1];
    const int cin = ws.c_cin[g];
    const int64_t coff = C.blk_off[g];
    const double *cinv = (cin >= 0) ? Cin.vals + Cin.blk_off[cin] : nullptr;

    for (int r0 = 0; r0 < m; r0 += kTile) {
      for (int c0 = 0; c0 < n; c0 += kTile) {
        const int tm = min(kTile, m - r0), tn = min(kTile, n - c0);
        const int te = tm * tn;
        const int nT = (te + 31) >> 5;
        double acc[32];
        int ar[32], bc[32];
#pragma unroll
        for (int t = 0; t < 32; t++) {
          acc[t] = 0.0;
          const int e = lane + 32 * t;
          // lanes past the tile read a valid dummy element; their sums are discarded
          ar[t] = (e < te) ? e % tm : 0;
          bc[t] = (e < te) ? (e / tm) * kLdB : 0;
        }
        for (int64_t p = p0; p < p1; p++) {
          const int2 pr = ws.prods[p];
          const int k = A.col_idx[pr.x];
          const int s = A.col_sizes[k];
          const double *Ab = A.vals + A.blk_off[pr.x];  // m x s, column-major
          const double *Bb = B.vals + B.blk_off[pr.y];  // s x n, column-major
          for (int l0 = 0; l0 < s; l0 += kTile) {
            const int kc = min(kTile, s - l0);
            __syncwarp();
            for (int e = lane; e < tm * kc; e += 32) {
              const int r = e % tm, l = e / tm;
              sA[l * kLdA + r] = __ldg(Ab + (int64_t)(l0 + l) * m + r0 + r);
            }
            for (int e = lane; e < kc * tn; e += 32) {
              const int l = e % kc, c = e / kc;
              sB[c * kLdB + l] = __ldg(Bb + (int64_t)(c0 + c) * s + l0 + l);
            }
            __syncwarp();
            for (int l = 0; l < kc; l++) {
#pragma unroll
              for (int t = 0; t < 32; t++) {
                if (t >= nT) break;
                acc[t] = fma(sA[l * kLdA + ar[t]], sB[bc[t] + l], acc[t]);
              }
            }
          }
        }
        // epilogue: C_ij = beta * C_in_ij + alpha * S_ij, written once
#pragma unroll
        for (int t = 0; t < 32; t++) {
          if (t >= nT) break;
          const int e = lane + 32 * t;
          if (e < te) {
            const int r = e % tm, c = e / tm;
            const int64_t loc = (int64_t)(c0 + c) * m + r0 + r;
            double v = alpha * acc[t];
            if (cinv) v = fma(beta, cinv[loc], v);
            C.vals[coff + loc] = v;
          }
        }
      }
    }
  }
}

// ----------------------------------------------------------------------------
// t16
// ----------------------------------------------------------------------------
constexpr int kS = 16;                 // output tile edge and k-chunk
constexpr int kSWarps = 8;             // warps per thread block
constexpr int kSElems = kS * kS / 32;  // operand elements per lane (8)

// Loads the A chunk (tm x kc, rows r0.., columns l0.. of the m x s block) and
// the B chunk (kc x tn, rows l0.., columns c0.. of the s x n block) of one
// step into registers, lane-strided in the chunks' own column-major order.
__device__ __forceinline__ void t16_load(const double *__restrict__ Ab,
                                         const double *__restrict__ Bb, int m, int s, int r0,
                                         int c0, int l0, int tm, int tn, int kc, int lane,
                                         double (&ra)[kSElems], double (&rb)[kSElems]) {
  const bool a_contig = (tm == m);  // whole columns of A: one contiguous range
  const bool b_contig = (kc == s);  // whole columns of B
#pragma unroll
  for (int u = 0; u < kSElems; u++) {
    const int e = lane + 32 * u;
    double va = 0.0, vb = 0.0;
    if (e < tm * kc) {
      const int64_t ia =
          a_contig ? (int64_t)l0 * m + e : (int64_t)(l0 + e / tm) * m + r0 + e % tm;
      va = __ldg(Ab + ia);
    }
    if (e < kc * tn) {
      const int64_t ib =
          b_contig ? (int64_t)c0 * s + e : (int64_t)(c0 + e / kc) * s + l0 + e % kc;
      vb = __ldg(Bb + ib);
    }
    ra[u] = va;
    rb[u] = vb;
  }
}

template <int MINB>
__global__ void __launch_bounds__(kSWarps * 32, MINB)
    k_numeric_fp64_t16(DevMat A, DevMat B, DevOut C, DevMat Cin, double alpha, double beta,
                       DevWs ws, const DevStatus *st, const int32_t *items, const int64_t *seg,
                       unsigned long long *work) {
  if (st->overflow) return;
  __shared__ double smem_t16[kSWarps][2 * kS * kS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double *sA = smem_t16[warp];
  double *sB = sA + kS * kS;
  int64_t wb, we;
  work_range(st, seg, wb, we);

  // C blocks come from the work counter (zero at launch), `grab` at a time:
  // one when there are few per warp, up to 8 when there are many (tiny C
  // blocks would otherwise queue on the counter)
  const int64_t per_warp = (we - wb) / ((int64_t)gridDim.x * kSWarps * 64);
  const int grab = per_warp < 1 ? 1 : (per_warp > 8 ? 8 : (int)per_warp);
  for (;;) {
    unsigned long long got = 0;
    if (lane == 0) got = atomicAdd(work, (unsigned long long)grab);
    const int64_t w0 = wb + (int64_t)__shfl_sync(0xffffffffu, got, 0);
    if (w0 >= we) break;
    const int64_t w1 = (w0 + grab < we) ? w0 + grab : we;
    for (int64_t w = w0; w < w1; w++) {
      const int64_t g = items ? items[w] : w;
      const int i = C.blk_row[g], j = C.col_idx[g];
      const int m = C.row_sizes[i], n = C.col_sizes[j];
      const int64_t p0 = ws.prod_ptr[g], p1 = ws.prod_ptr[g + 1];
      const int cin = ws.c_cin[g];
      const double *cinv = (cin >= 0) ? Cin.vals + Cin.blk_off[cin] : nullptr;
      double *out = C.vals + C.blk_off[g];

      for (int r0 = 0; r0 < m; r0 += kS) {
        for (int c0 = 0; c0 < n; c0 += kS) {
          const int tm = min(kS, m - r0), tn = min(kS, n - c0);
          const int te = tm * tn;
          const int nT = (te + 31) >> 5;
          int rc[kSElems];  // (row, col) in the tile of the lane's t-th output, r | c << 8
          double acc[kSElems];
#pragma unroll
          for (int t = 0; t < kSElems; t++) {
            const int e = lane + 32 * t;
            rc[t] = (e < te) ? (e % tm) | ((e / tm) << 8) : 0;  // past the tile: a valid dummy
            acc[t] = 0.0;
          }
          for (int64_t pb = p0; pb < p1; pb += 32) {
            const int nb = (p1 - pb < 32) ? (int)(p1 - pb) : 32;
            int64_t my_a = 0, my_b = 0;
            int my_s = 1;
            if (lane < nb) {
              const int2 pr = ws.prods[pb + lane];
              my_a = A.blk_off[pr.x];
              my_b = B.blk_off[pr.y];
              my_s = A.col_sizes[A.col_idx[pr.x]];
            }
            double ra[kSElems], rb[kSElems];
            int q = 0, l0 = 0;
            int s = __shfl_sync(0xffffffffu, my_s, 0);
            t16_load(A.vals + __shfl_sync(0xffffffffu, my_a, 0),
                     B.vals + __shfl_sync(0xffffffffu, my_b, 0), m, s, r0, c0, 0, tm, tn,
                     min(kS, s), lane, ra, rb);
            while (q < nb) {
              __syncwarp();
#pragma unroll
              for (int u = 0; u < kSElems; u++) {
                sA[lane + 32 * u] = ra[u];
                sB[lane + 32 * u] = rb[u];
              }
              __syncwarp();
              const int kc = min(kS, s - l0);
              // the next step: the next k-chunk of this product, or the next product
              int nq = q, nl0 = l0 + kS;
              if (nl0 >= s) {
                nq = q + 1;
                nl0 = 0;
              }
              // warp-uniform: every lane evaluates the same (nq, nl0)
              const int ns = __shfl_sync(0xffffffffu, my_s, nq < nb ? nq : 0);
              const int64_t na = __shfl_sync(0xffffffffu, my_a, nq < nb ? nq : 0);
              const int64_t nbo = __shfl_sync(0xffffffffu, my_b, nq < nb ? nq : 0);
              if (nq < nb)
                t16_load(A.vals + na, B.vals + nbo, m, ns, r0, c0, nl0, tm, tn, min(kS, ns - nl0),
                         lane, ra, rb);
              for (int l = 0; l < kc; l++) {
#pragma unroll
                for (int t = 0; t < kSElems; t++) {
                  if (t >= nT) break;
                  acc[t] = fma(sA[(rc[t] & 255) + l * tm], sB[(rc[t] >> 8) * kc + l], acc[t]);
                }
              }
              q = nq;
              l0 = nl0;
              s = ns;
            }
          }
          // epilogue: C_ij = beta * C_in_ij + alpha * S_ij
#pragma unroll
          for (int t = 0; t < kSElems; t++) {
            const int e = lane + 32 * t;
            if (t < nT && e < te) {
              const int64_t loc = (int64_t)(c0 + (rc[t] >> 8)) * m + r0 + (rc[t] & 255);
              double v = alpha * acc[t];
              if (cinv) v = fma(beta, cinv[loc], v);
              out[loc] = v;
            }
          }
        }
      }
    }
  }
}

// ----------------------------------------------------------------------------
// g8: tiny C blocks with few products (semi-empirical-style matrices: blocks
// of a few rows, about one product per C block). A group of 8 lanes computes
// one C block at a time, a lane per column, the rows in registers (MR = 4, 6
// or 8 rows and GS = 4, 6 or 8 lanes per group, chosen per launch from the
// largest C block: 5 groups of 6 lanes fill 30 of a warp's 32 lanes for
// 6-wide blocks, where groups of 8 would leave a quarter of the lanes without
// a column). A warp takes a run of C blocks at a time, whose descriptors and
// products its lanes look up at once; each group takes the run's next block when
// it has closed one, and walks its products one step per loop iteration. The
// finished blocks are gathered in shared memory and leave the warp together: the
// blocks of a run mostly follow one another in C, and a store instruction then
// covers 256 contiguous bytes. A lane's own columns would be 8 bytes apart from
// every other store, which the link to host memory (the second destination) takes
// at 25 GB/s of its 193.
// Measured, 20000 atoms, 2.2 M C blocks of 6, numeric phase with a second destination in
// host memory: 26.1 -> 3.40 ms, bound by the link (637 MB); without one 1.40 -> 1.32, bound
// by the FP64 pipe (0.68 without its instructions), if nothing is left to do at the stores
// (alpha = 1, no C_in). 16 warps per SM with runs of 30 blocks: 24 warps with runs of 15 took
// 0.15 ms more, 32 0.5 (the groups idle at a run's end).
// g8_direct has no runs: each group stores its blocks itself, in the iteration that closes
// them. It is the faster one without a second destination where the stores have work or the
// blocks are up to 4 x 4 (gathered -> direct, blocks of 4, 6, 8): alpha other than 1 0.59 ->
// 0.51, 1.47 -> 1.40, 1.73 -> 1.62 ms; with C_in 0.74 -> 0.63, 1.77 -> 1.60, 1.99 -> 1.82; plain
// 0.53 -> 0.52, but 1.32 -> 1.40, 1.58 -> 1.62. Both give the same bits. Larger blocks
// (below) are the gathering kernel's: two to four times as fast.
// A C block of more than MR rows or GS columns (only when the kernel is forced on
// larger blocks) is done in column and row chunks by its group and stored directly.
// ----------------------------------------------------------------------------
constexpr int kG8Warps = 8;
constexpr int kG8BlocksPerSm = 2;
constexpr int kG8Stage = 1152;  // doubles a warp gathers, at most
constexpr int kG8List = 64;     // products of a run that are listed
struct G8Item {  // a C block of a warp's run
  int64_t coff, p, cin;      // cin: offset of its C_in block, or -1
  int32_t np, m, n, at, q0;  // at: of its values in the stage, q0: its first product's entry
};
struct G8Product {  // where the two blocks of a product start, and their common size
  int64_t a, b;
  int32_t s;
};

size_t g8_smem_bytes() {
  return kG8Warps * (kG8Stage * sizeof(double) + kG8List * sizeof(G8Product) + 32 * sizeof(G8Item));
}

template <int MR, int GS>
__global__ void __launch_bounds__(kG8Warps * 32, kG8BlocksPerSm)
    k_numeric_fp64_g8(DevMat A, DevMat B, DevOut C, DevMat Cin, double alpha, double beta,
                      DevWs ws, const DevStatus *st, const int32_t *items, const int64_t *seg,
                      unsigned long long *work) {
  if (st->overflow) return;
  constexpr int kGroups = 32 / GS;
  constexpr int kFit = kG8Stage / (MR * GS);  // blocks of MR x GS that the stage holds
  constexpr int kRun = (kFit < 32 ? kFit : 32) / kGroups * kGroups;
  extern __shared__ double smem_g8[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int grp = lane / GS, cl = lane - grp * GS;
  double *stage = smem_g8 + warp * kG8Stage;
  G8Product *list = reinterpret_cast<G8Product *>(smem_g8 + kG8Warps * kG8Stage) + warp * kG8List;
  G8Item *item = reinterpret_cast<G8Item *>(
                     reinterpret_cast<G8Product *>(smem_g8 + kG8Warps * kG8Stage) +
                     kG8Warps * kG8List) + warp * 32;
  int64_t wb, we;
  work_range(st, seg, wb, we);
  // the second destination (host memory) when the whole result fits it
  double *hout = (C.host_vals && st->nnz_c <= C.host_cap) ? C.host_vals : nullptr;

  double acc[MR];
  auto entry = [&](int64_t q) -> G8Product {
    const int2 pr = ws.prods[q];
    return {A.blk_off[pr.x], B.blk_off[pr.y], A.col_sizes[A.col_idx[pr.x]]};
  };
  // rows [r0, r0 + MR) of column c of a product, added to acc
  auto product = [&](const G8Product &e, int m, int c, int r0) {
    const double *Ab = A.vals + e.a + r0;
    const double *Bb = B.vals + e.b + (int64_t)c * e.s;
#pragma unroll 2
    for (int kk = 0; kk < e.s; kk++) {
      const double bv = __ldg(Bb + kk);
      const double *a = Ab + (int64_t)kk * m;
#pragma unroll
      for (int r = 0; r < MR; r++)
        if (r0 + r < m) acc[r] = fma(__ldg(a + r), bv, acc[r]);
    }
  };
  // C_ij = beta * C_in_ij + alpha * S_ij of row r of acc, at loc of the block
  auto value = [&](const double *cinv, int r, int64_t loc) {
    const double v = alpha * acc[r];
    return cinv ? fma(beta, cinv[loc], v) : v;
  };
  auto scan = [&](int v) {  // inclusive sum over the lanes
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, v, d);
      if (lane >= d) v += y;
    }
    return v;
  };

  for (;;) {
    unsigned long long got = 0;
    if (lane == 0) got = atomicAdd(work, (unsigned long long)kRun);
    const int64_t base = wb + (int64_t)__shfl_sync(0xffffffffu, got, 0);
    if (base >= we) break;
    const int count = we - base < kRun ? (int)(we - base) : kRun;
    G8Item own{};
    own.cin = -1;
    if (lane < count) {
      const int64_t g = items ? items[base + lane] : base + lane;
      own.m = C.row_sizes[C.blk_row[g]];
      own.n = C.col_sizes[C.col_idx[g]];
      own.p = ws.prod_ptr[g];
      own.np = (int)(ws.prod_ptr[g + 1] - own.p);
      const int cin = ws.c_cin[g];
      own.cin = cin >= 0 ? Cin.blk_off[cin] : -1;
      own.coff = C.blk_off[g];
    }
    const bool gather = !__any_sync(0xffffffffu, own.m > MR || own.n > GS);
    const bool late = gather && !__any_sync(0xffffffffu, own.cin >= 0);  // alpha at the stores
    const int mn = own.m * own.n;
    own.at = scan(mn) - mn;
    const int np = own.np < kG8List ? own.np : kG8List;
    const int q1 = scan(np);
    own.q0 = q1 - np;
    if (lane < count) item[lane] = own;
    // blocks that do not follow the one before them in C
    const int64_t follows = __shfl_up_sync(0xffffffffu, own.coff + mn, 1);
    uint32_t starts = __ballot_sync(0xffffffffu, lane < count && (lane == 0 || own.coff != follows));
    // the products' entries, a lane each
    const int listed = min(__shfl_sync(0xffffffffu, q1, 31), kG8List);
    for (int q = lane; q - lane < listed; q += 32) {
      int b = 0;  // the block of product q: blocks that end at or before it
#pragma unroll
      for (int step = 16; step; step >>= 1)
        if (__shfl_sync(0xffffffffu, q1, b + step - 1) <= q) b += step;
      const int64_t p = __shfl_sync(0xffffffffu, own.p - own.q0, b) + q;
      if (q < listed) list[q] = entry(p);
    }
    __syncwarp();

    // a group takes the run's next block when it has closed one
    int k = grp < kGroups ? grp : count, taken = kGroups, p = 0;
    G8Item it{};
    if (k < count) it = item[k];
#pragma unroll
    for (int r = 0; r < MR; r++) acc[r] = 0.0;
    while (__any_sync(0xffffffffu, k < count)) {
      if (k < count) {
        const double *cinv = it.cin >= 0 ? Cin.vals + it.cin : nullptr;
        if (!gather) {  // column and row chunks, the products once per chunk
          for (int c = cl; c < it.n; c += GS)
            for (int r0 = 0; r0 < it.m; r0 += MR) {
#pragma unroll
              for (int r = 0; r < MR; r++) acc[r] = 0.0;
              for (int q = 0; q < it.np; q++) product(entry(it.p + q), it.m, c, r0);
#pragma unroll
              for (int r = 0; r < MR; r++)
                if (r0 + r < it.m) {
                  const int64_t loc = (int64_t)c * it.m + r0 + r;
                  const double v = value(cinv, r, loc);
                  C.vals[it.coff + loc] = v;
                  if (hout) hout[it.coff + loc] = v;
                }
            }
          p = it.np;
        } else {
          if (p < it.np) {  // one product of the block (products in ascending k)
            const G8Product e = it.q0 + p < listed ? list[it.q0 + p] : entry(it.p + p);
            if (cl < it.n) product(e, it.m, cl, 0);
            p++;
          }
          if (p >= it.np && cl < it.n) {  // the block is complete
            double *to = stage + it.at + cl * it.m;
            if (late) {
#pragma unroll
              for (int r = 0; r < MR; r++)
                if (r < it.m) to[r] = acc[r];
            } else {
#pragma unroll
              for (int r = 0; r < MR; r++)
                if (r < it.m) to[r] = value(cinv, r, cl * it.m + r);
            }
          }
        }
      }
      const bool closed = grp < kGroups && k < count && p >= it.np;
      const uint32_t heads = __ballot_sync(0xffffffffu, closed && cl == 0);
      if (closed) {
        k = taken + __popc(heads & ((1u << (grp * GS)) - 1u));
        p = 0;
        if (k < count) it = item[k];
#pragma unroll
        for (int r = 0; r < MR; r++) acc[r] = 0.0;
      }
      taken += __popc(heads);
    }
    __syncwarp();
    if (late && alpha != 1.0) {  // a loop of its own: no FP64 instruction without it
      const int all = __shfl_sync(0xffffffffu, own.at + mn, count - 1);
      for (int e = lane; e < all; e += 32) stage[e] *= alpha;
      __syncwarp();
    }
    while (gather && starts) {  // blocks x to y - 1, which follow one another in C
      const int x = __ffs(starts) - 1;
      starts &= starts - 1;
      const int y = starts ? __ffs(starts) - 1 : count;
      const int at = __shfl_sync(0xffffffffu, own.at, x);
      const int total = __shfl_sync(0xffffffffu, own.at + mn, y - 1) - at;
      const int64_t first = __shfl_sync(0xffffffffu, own.coff, x);
      // from the start of the 128-byte line that they begin in
      for (int e = lane - (int)(first & 15); e < total; e += 32)
        if (e >= 0) {
          const double v = stage[at + e];
          __stcs(C.vals + first + e, v);
          if (hout) __stcs(hout + first + e, v);
        }
    }
    __syncwarp();
  }
}

// The groups of a warp are independent streams: each takes kG8Grab C blocks at a time from
// the work counter and walks their products one step per loop iteration, closing a C block
// (epilogue, next block's metadata) in the iteration that ends it, so a group whose block
// has more products does not hold the other groups at a loop exit. The latency of each C
// block's chain of dependent loads is hidden by the many independent blocks in flight.
constexpr int kG8DirectBlocksPerSm = 4;
constexpr int kG8Grab = 16;  // C blocks per group and grab

template <int MR, int GS>
__global__ void __launch_bounds__(kG8Warps * 32, kG8DirectBlocksPerSm)
    k_numeric_fp64_g8_direct(DevMat A, DevMat B, DevOut C, DevMat Cin, double alpha, double beta,
                             DevWs ws, const DevStatus *st, const int32_t *items,
                             const int64_t *seg, unsigned long long *work) {
  if (st->overflow) return;
  const int lane = threadIdx.x & 31;
  const int grp = lane / GS, cl = lane - grp * GS;
  if (grp >= 32 / GS) return;  // lanes past the last whole group
  const unsigned gmask = ((1u << GS) - 1u) << (GS * grp);
  int64_t wb, we;
  work_range(st, seg, wb, we);

  // the group's current grab [w, wend) and C block (group-uniform state)
  int64_t w = 0, wend = 0, p = 0, p1 = 0, cbase = 0;
  int m = 0, n = 0;
  const double *cinv = nullptr;
  double acc[MR];
  auto next_block = [&]() -> bool {
    if (w >= wend) {
      unsigned long long got = 0;
      if (cl == 0) got = atomicAdd(work, (unsigned long long)kG8Grab);
      w = wb + (int64_t)__shfl_sync(gmask, got, GS * grp);
      wend = (w + kG8Grab < we) ? w + kG8Grab : we;
      if (w >= we) return false;
    }
    const int64_t g = items ? items[w] : w;
    w++;
    m = C.row_sizes[C.blk_row[g]];
    n = C.col_sizes[C.col_idx[g]];
    p = ws.prod_ptr[g];
    p1 = ws.prod_ptr[g + 1];
    const int cin = ws.c_cin[g];
    cinv = (cin >= 0) ? Cin.vals + Cin.blk_off[cin] : nullptr;
    cbase = C.blk_off[g];
#pragma unroll
    for (int r = 0; r < MR; r++) acc[r] = 0.0;
    return true;
  };
  // column cl of product q, added to acc
  auto product = [&](int64_t q) {
    const int2 pr = ws.prods[q];
    const double *Ab = A.vals + A.blk_off[pr.x];
    const int s = A.col_sizes[A.col_idx[pr.x]];
    const double *Bb = B.vals + B.blk_off[pr.y] + (int64_t)cl * s;
    for (int kk = 0; kk < s; kk++) {
      const double bv = __ldg(Bb + kk);
      const double *a = Ab + (int64_t)kk * m;
#pragma unroll
      for (int r = 0; r < MR; r++)
        if (r < m) acc[r] = fma(__ldg(a + r), bv, acc[r]);
    }
  };
  // C_ij = beta * C_in_ij + alpha * S_ij
  auto store = [&]() {
#pragma unroll
    for (int r = 0; r < MR; r++) {
      if (r < m) {
        const int64_t loc = (int64_t)cl * m + r;
        double v = alpha * acc[r];
        if (cinv) v = fma(beta, cinv[loc], v);
        C.vals[cbase + loc] = v;
      }
    }
  };

  bool have = next_block();
  while (have) {
    if (p < p1) {  // one product of the block (products in ascending k)
      if (cl < n) product(p);
      p++;
    }
    if (p >= p1) {  // the block is complete
      if (cl < n) store();
      have = next_block();
    }
  }
}

// ----------------------------------------------------------------------------
// pk
// ----------------------------------------------------------------------------
constexpr int kPkWarps = 8;          // warps per thread block (2 blocks per SM)
constexpr int kPkTile = 16;          // output tile edge
constexpr int kPkMaxSlots = 16;      // accumulator slots per lane (largest nT) of the pk16 variant
constexpr int kPkMaxG = kPkMaxGroups;  // largest number of k-groups
constexpr int kPkMaxKC = 64;         // largest chunk (k positions)
// Doubles per stage (two stages per warp; 2 blocks of 8 warps fit an SM). A
// tile of tm x tn takes chunks of KC k positions with KC * tm + tn * (KC + 1)
// within the stage.
constexpr int kPkStage = 880;
static_assert(32 * kPkMaxSlots <= kPkStage, "the slot sums must fit one stage");

size_t pk_smem_bytes() { return (size_t)kPkWarps * 2 * kPkStage * sizeof(double); }

// Slot shape of a tile of te (1..256) elements with at most `slots` slots per
// lane: the (nT, G) with nT <= slots, G <= kPkMaxG and te * G <= 32 * nT that
// maximises te * G / (32 * nT), the smallest nT among equals.
struct PkShapes {
  uint8_t nt[kPkTile * kPkTile + 1], g[kPkTile * kPkTile + 1];
};
constexpr PkShapes make_pk_shapes(int slots) {
  PkShapes tab{};
  for (int te = 1; te <= kPkTile * kPkTile; te++) {
    int bt = (te + 31) / 32, bg = 1;
    for (int t = 1; t <= slots; t++) {
      int g = (32 * t) / te;
      if (g > kPkMaxG) g = kPkMaxG;
      if (g >= 1 && g * bt > bg * t) {
        bt = t;
        bg = g;
      }
    }
    tab.nt[te] = (uint8_t)bt;
    tab.g[te] = (uint8_t)bg;
  }
  return tab;
}
__constant__ PkShapes c_pk_shapes12 = make_pk_shapes(12);
__constant__ PkShapes c_pk_shapes16 = make_pk_shapes(16);
static_assert(kPkTabEdge == kPkTile + 1, "the tuned table covers every tile shape");

void pk_formula_shape(int slots, int te, int *nt, int *g) {
  static const PkShapes s12 = make_pk_shapes(12), s16 = make_pk_shapes(16);
  const PkShapes &s = (slots == 12) ? s12 : s16;
  *nt = s.nt[te];
  *g = s.g[te];
}

// floor(x / d) as (x * r) >> 16 with r = ceil(2^16 / d): exact while
// x * (r * d - 2^16) < 2^16, i.e. for d <= 16 and x < 4096 (the error term is
// below d).
__device__ __forceinline__ uint32_t rcp16(uint32_t d) { return (65535u + d) / d; }
__device__ __forceinline__ int div16(int x, uint32_t r) { return (int)(((uint32_t)x * r) >> 16); }

__device__ __forceinline__ void cp_async8(double *sdst, const double *gsrc) {
  const uint32_t sa = (uint32_t)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void pk_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void pk_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// C blocks a warp takes from the work counter at a time.
constexpr int kPkGrab = 1;
constexpr int kPkUnits = 16;  // units of work per warp up to which C blocks are split

// `steps` steps of one chunk for a tile of NT slots per lane: slot t adds
// sA[ia_t + u * G * tm] * sB[ib_t + u * G] at step u. NT is a compile-time
// constant, so all loads of a step can be issued ahead of its FMAs; the step
// loop itself is not unrolled (with 16 instances, unrolled copies overflow the
// instruction cache on workloads with many tile shapes).
template <int NT, int SLOTS>
__device__ __forceinline__ void pk_steps(const double *__restrict__ sA,
                                         const double *__restrict__ sB,
                                         const uint32_t (&idx)[SLOTS],
                                         double (&acc)[SLOTS], int steps, int gtm, int G) {
#pragma unroll 1  // one copy of the step body per NT keeps the instruction footprint small
  for (int u = 0; u < steps; u++) {
#pragma unroll
    for (int t = 0; t < NT; t++) acc[t] = fma(sA[idx[t] & 0xFFFFu], sB[idx[t] >> 16], acc[t]);
    sA += gtm;
    sB += G;
  }
}

// C block gblk by one warp. wbuf: two stages of shared memory. hout: host copy
// of C's values or null. SLOTS: accumulator slots per lane (12 or 16). Fewer
// slots lower the lane use of some tile shapes (13 x 13: 96% instead of 99%)
// but shorten the per-tile code; which wins depends on the block mix (the
// autotuner measures it).
template <int SLOTS>
__device__ __forceinline__ void pk_block(const DevMat &A, const DevMat &B, const DevOut &C,
                                         const DevMat &Cin, double alpha, double beta,
                                         const DevWs &ws, int64_t gblk, int part, int parts, double *wbuf,
                                         double *hout, int lane) {
  constexpr int kStage = kPkStage;
  const PkShapes &shapes = (SLOTS == 12) ? c_pk_shapes12 : c_pk_shapes16;
  const int i = C.blk_row[gblk], j = C.col_idx[gblk];
  const int m = C.row_sizes[i], n = C.col_sizes[j];
  const int64_t p0 = ws.prod_ptr[gblk], p1 = ws.prod_ptr[gblk + 1];
  const int cin = ws.c_cin[gblk];
  const double *cinv = (cin >= 0) ? Cin.vals + Cin.blk_off[cin] : nullptr;
  double *out = C.vals + C.blk_off[gblk];
  double *hblk = hout ? hout + C.blk_off[gblk] : nullptr;

  int at = 0;  // the tile's number
  for (int r0 = 0; r0 < m; r0 += kPkTile) {
    for (int c0 = 0; c0 < n; c0 += kPkTile) {
      if (parts > 1 && at++ % parts != part) continue;
      const int tm = min(kPkTile, m - r0), tn = min(kPkTile, n - c0);
      const int te = tm * tn;
      int nT = shapes.nt[te], G = shapes.g[te];
      if (ws.pk_tab) {  // a tuned shape (validated by the host)
        const uint32_t e = ws.pk_tab[(SLOTS == 16 ? kPkTabSize : 0) + tm * kPkTabEdge + tn];
        nT = (int)(e >> 8);
        G = (int)(e & 0xFFu);
      }
      const int used = te * G;
      const uint32_t rtm = rcp16(tm), rg = rcp16(G);
      // chunk length: the largest multiple of G with KC * tm + tn * (KC + 1) <= kStage
      const int kfit = min(kPkMaxKC, (kStage - tn) / (tm + tn));
      const int KC = G * div16(kfit, rg);
      const int ldB = KC + 1;  // sB[c * ldB + kk]
      const int dq_tm = div16(32, rtm), dr_tm = 32 - dq_tm * tm;  // 32 = dq_tm * tm + dr_tm
      // slot t of this lane: z = lane + 32 t -> group g = z / te, element
      // e = z % te (row e % tm, column e / tm); its operands at step 0 are
      // sA[ia] and sB[ib], kept as ia | ib << 16 (both below 2^9)
      uint32_t idx[SLOTS];
      double acc[SLOTS];
      {
        int g = 0, e = lane;
        while (e >= te) {
          e -= te;
          g++;
        }
#pragma unroll
        for (int t = 0; t < SLOTS; t++) {
          idx[t] = 0;  // slots past te * G read valid operands; their sums are discarded
          if (g < G) {
            const int c = div16(e, rtm), r = e - c * tm;
            idx[t] = (uint32_t)(g * tm + r) | ((uint32_t)(c * ldB + g) << 16);
          }
          acc[t] = 0.0;
          e += 32;
          while (e >= te) {
            e -= te;
            g++;
          }
        }
      }

      // product cursor: batch [pb, pb + nb) of metadata, one product per lane
      int64_t pb = p0;
      int nb = 0, q = 0, lq = 0;
      int64_t my_a = 0, my_b = 0;
      int my_s = 1;
      auto load_batch = [&]() {
        nb = (p1 - pb < 32) ? (int)(p1 - pb) : 32;
        if (lane < nb) {
          const int2 pr = __ldcs(ws.prods + pb + lane);  // read once: evict first
          my_a = A.blk_off[pr.x];
          my_b = B.blk_off[pr.y];
          my_s = A.col_sizes[A.col_idx[pr.x]];
        }
      };
      if (pb < p1) load_batch();

      // Copies the next (up to) KC k positions of the concatenated products
      // into stage `buf`: sA[kk * tm + r] = A(r0 + r, k), sB[c * ldB + kk] =
      // B(k, c0 + c); zero-fills up to the next multiple of G. Returns the
      // number of steps (k positions / G) of the chunk.
      auto fill = [&](int buf) -> int {
        double *sA = wbuf + buf * kStage;
        double *sB = sA + KC * tm;
        int kk = 0;
        while (kk < KC && pb < p1) {
          const int s = __shfl_sync(0xffffffffu, my_s, q);
          const int64_t ao = __shfl_sync(0xffffffffu, my_a, q);
          const int64_t bo = __shfl_sync(0xffffffffu, my_b, q);
          const int nc = min(s - lq, KC - kk);
          const double *Ab = A.vals + ao + (int64_t)lq * m + r0;  // column lq, row r0
          const double *Bb = B.vals + bo + (int64_t)c0 * s + lq;  // row lq, column c0
          double *dA = sA + kk * tm;
          if (tm == m) {  // whole columns: one contiguous range
            for (int z = lane; z < nc * m; z += 32) cp_async8(dA + z, Ab + z);
          } else {  // (l, r) = divmod(z, tm), stepped by 32
            int l = div16(lane, rtm), r = lane - l * tm;
            for (int z = lane; z < nc * tm; z += 32) {
              cp_async8(dA + l * tm + r, Ab + (int64_t)l * m + r);
              l += dq_tm;
              r += dr_tm;
              if (r >= tm) {
                r -= tm;
                l++;
              }
            }
          }
          {  // (c, l) = divmod(z, nc), stepped by 32
            const uint32_t rnc = rcp16(nc);
            const int dq = div16(32, rnc), dr = 32 - dq * nc;
            int c = div16(lane, rnc), l = lane - c * nc;
            double *dB = sB + kk;
            for (int z = lane; z < nc * tn; z += 32) {
              cp_async8(dB + c * ldB + l, Bb + (int64_t)c * s + l);
              c += dq;
              l += dr;
              if (l >= nc) {
                l -= nc;
                c++;
              }
            }
          }
          kk += nc;
          lq += nc;
          if (lq == s) {
            lq = 0;
            if (++q == nb) {
              pb += nb;
              q = 0;
              if (pb < p1) load_batch();
            }
          }
        }
        const int steps = div16(kk + G - 1, rg);
        const int pad = steps * G - kk;
        if (pad) {
          for (int z = lane; z < pad * tm; z += 32) sA[kk * tm + z] = 0.0;
          for (int z = lane; z < pad * tn; z += 32) {
            const int c = div16(z, rcp16(pad)), l = z - c * pad;
            sB[c * ldB + kk + l] = 0.0;
          }
        }
        return steps;
      };

      int cur = fill(0);  // steps of the current chunk
      pk_commit();
      for (int ch = 0;; ch++) {
        const int buf = ch & 1;
        const int nxt = (pb < p1) ? fill(buf ^ 1) : 0;
        pk_commit();
        pk_wait<1>();  // the current chunk has landed
        __syncwarp();
        const double *sA = wbuf + buf * kStage;
        const double *sB = sA + KC * tm;
        const int gtm = G * tm;
        switch (nT) {
#define BSM_PK_CASE(N)                                                                 \
  case N:                                                                              \
if (N <= SLOTS) pk_steps<(N <= SLOTS ? N : 1), SLOTS>(sA, sB, idx, acc, cur, gtm, G); \
break;
          BSM_PK_CASE(1) BSM_PK_CASE(2) BSM_PK_CASE(3) BSM_PK_CASE(4)
          BSM_PK_CASE(5) BSM_PK_CASE(6) BSM_PK_CASE(7) BSM_PK_CASE(8)
          BSM_PK_CASE(9) BSM_PK_CASE(10) BSM_PK_CASE(11) BSM_PK_CASE(12)
          BSM_PK_CASE(13) BSM_PK_CASE(14) BSM_PK_CASE(15) BSM_PK_CASE(16)
#undef BSM_PK_CASE
        }
        __syncwarp();  // the stage is read before it is filled again
        if (nxt == 0) break;
        cur = nxt;
      }
      pk_wait<0>();
      __syncwarp();

      // the G partial sums of each element, added in group order
      double *red = wbuf;
#pragma unroll
      for (int t = 0; t < SLOTS; t++) {
        const int z = lane + 32 * t;
        if (t < nT && z < used) red[z] = acc[t];
      }
      __syncwarp();
      int c = div16(lane, rtm), r = lane - c * tm;
      for (int e = lane; e < te; e += 32) {
        double v = red[e];
        for (int g = 1; g < G; g++) v += red[g * te + e];
        const int64_t loc = (int64_t)(c0 + c) * m + r0 + r;
        v = alpha * v;
        if (cinv) v = fma(beta, cinv[loc], v);
        // written once, not read by this multiply: streaming stores keep the
        // operand rows, which the next C blocks read, in L2
        __stcs(out + loc, v);
        if (hblk) __stcs(hblk + loc, v);
        c += dq_tm;
        r += dr_tm;
        if (r >= tm) {
          r -= tm;
          c++;
        }
      }
      __syncwarp();
    }
  }
}

// work: a counter that is zero when the launch starts; warps take the next
// kPkGrab C blocks of the work range from it until the range is exhausted. With
// ntiles > 0 (the tiles that a C block has at most), a few C blocks are split into
// parts, every parts-th of a block's tiles each: those that another kernel leaves are
// few, and a large one that is a warp's alone takes as long as a whole multiply (2% of
// 8695 blocks of up to 33 x 33: 449 -> 115 us).
template <int SLOTS>
__global__ void __launch_bounds__(kPkWarps * 32, 2)
    k_numeric_fp64_pk(DevMat A, DevMat B, DevOut C, DevMat Cin, double alpha, double beta,
                      DevWs ws, const DevStatus *st, const int32_t *items, const int64_t *seg,
                      unsigned long long *work, int ntiles) {
  if (st->overflow) return;
  extern __shared__ double smem_pk[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double *wbuf = smem_pk + warp * 2 * kPkStage;
  int64_t wb, we;
  work_range(st, seg, wb, we);
  // the second destination (host memory) when the whole result fits it
  double *hout = (C.host_vals && st->nnz_c <= C.host_cap) ? C.host_vals : nullptr;
  int parts = 1;
  if (ntiles > 0) {
    const int64_t warps = (int64_t)gridDim.x * kPkWarps;
    parts = (int)min((int64_t)ntiles, max((int64_t)1, kPkUnits * warps / max((int64_t)1, we - wb)));
    we = wb + (we - wb) * parts;
  }

  for (;;) {
    unsigned long long got = 0;
    if (lane == 0) got = atomicAdd(work, (unsigned long long)kPkGrab);
    const int64_t w0 = wb + (int64_t)__shfl_sync(0xffffffffu, got, 0);
    if (w0 >= we) break;
    const int64_t w1 = (w0 + kPkGrab < we) ? w0 + kPkGrab : we;
    for (int64_t w = w0; w < w1; w++) {
      const int64_t b = parts > 1 ? wb + (w - wb) / parts : w;
      pk_block<SLOTS>(A, B, C, Cin, alpha, beta, ws, items ? items[b] : b,
                      parts > 1 ? (int)((w - wb) % parts) : 0, parts, wbuf, hout, lane);
    }
  }
}

// ----------------------------------------------------------------------------
// dg: the FP64 products on the tensor cores, in exact integer arithmetic. The
// operands come as eight signed base-256 digits per value, on a scale of their
// own for every scalar row of A and column of B (bsm_internal.h, digits.cuh). A
// product of two values is sum_d 256^-d v_d, v_d = sum over i + j = d of a_i b_j;
// the digit pairs of every diagonal d < kDgDiag are multiplied by mma.sync (FP16
// operands that are small integers, so every term is exact) into one FP32
// accumulator per element and diagonal. With at most 144 values of k between two
// reads its sums stay below 2^24, where FP32 numbers are exact integers. A read
// adds the diagonals up in 64-bit integers, and the whole sum (of the products of one
// class) is rounded to FP64 once. What is lost besides is half a unit of 2^-62 of each
// row's scale and the diagonals from kDgDiag on (2^-67.4 of the product of the scales for
// each value of k): dg_enough says for which C blocks that is no more than FP64 FMAs lose.
// Measured against long double, relative Frobenius error of C (and the worst of C's
// blocks): water of 128 molecules 4.5e-17 (1.4e-16), the packed kernel 4.7e-16
// (7.9e-16); amorphous of 200 atoms 4.6e-17 (7.3e-17), packed 1.0e-15 (1.7e-15); rows of
// unlike scales in blocks of 1 to 33 5.9e-17 (4.4e-16), packed 4.0e-16 (9.6e-15). Largest
// error of an element against the sum of its absolute products: ragged blocks 2.7e-16, sign
// iterates of 64 water molecules 0.4, 2.4 and 0.8e-15, water 1.0e-16, amorphous 1.0e-16;
// packed 5.1e-16; 2.4, 3.0 and 4.4e-15; 2.0e-15; 3.1e-15.
//
// Why: the FP64 pipe does 2 FMA per clock and SM, mma.sync on FP16 1024, and 43
// digit pairs stand for one product. (FP8 and INT8 mma.sync are emulated or slow on
// this part: 3.8 and 16 clocks per m16n8k32 and SM, FP16 m16n8k16 2.0.) Numeric
// phase, packed kernel -> this one: water of 2048 molecules 47.7 -> 23.3 ms (21.3 without
// dg_enough; 0.8 is the packed kernel's on the 8% of the C blocks that it leaves),
// amorphous of 1024 atoms 67.9 -> 22.7 (22.0), 64 x 64 full blocks of 32 15.7 -> 2.0. What
// bounds it: the MMA pipe (0.49 of the clocks of the first) and the instructions beside
// it, which do not hide behind the MMAs whatever the number of warps (with 16, 20 and 24
// per SM 21.4, 21.9 and 22.2 ms): left out one at a time, the digits' conversion is
// 1.5 ms, the search for an octet's product and the loads' misses 4, the 64-bit sums 0.8,
// the epilogue nothing (L2 and L1 are at 10 and 20%).
//
// A warp takes whole C blocks while there are kDgUnits per warp, else parts of their
// tiles (dense matrices of 8 x 8, 16 x 16, 32 x 32 and 64 x 64 blocks of 32: 0.144,
// 0.326, 0.628 and 2.40 ms with whole blocks, 0.041, 0.061, 0.281 and 2.04 with parts; up
// to 16 and 32 units a warp gain nothing more and cost up to 5% on blocks of one tile).
//
// The products of a C block are concatenated along k in octets (8 of k), two to an
// MMA step; a warp takes a tile of up to 16 x 8 (the MMA's shape):
//   WIDE: more than 8 rows;
//   else: MMA rows 0-7 take the even, rows 8-15 the odd digits of the left side,
//         so one MMA adds to two diagonals (23 instead of 43 MMAs per 16 k).
// A lane's part of an operand octet is one 16-byte load, all digits of two values
// (a warp's load is whole 128-byte lines), straight into registers, where two
// instructions make an MMA register of each digit. (Measured and left: staging in
// shared memory, where each cp.async costs three more instructions on this part and
// the register groups of the MMAs a move per register, 31 ms; FP16 words in memory,
// without conversions but four times the bytes, 24-26 ms; registers loaded a step
// ahead in 12 warps, 24.6 ms.)
// ----------------------------------------------------------------------------
constexpr int kDgWarps = 8;             // warps per thread block
constexpr int kDgBlocksPerSm = 2;
constexpr int kDgDiag = 9;              // diagonals kept
constexpr int kDgFold = 18;             // octets between two reads of the accumulators
constexpr int kDgGrab = 8;              // C blocks a warp takes at a time, at most
constexpr int kDgUnits = 8;              // units of work per warp up to which C blocks are split

__device__ __forceinline__ void dg_mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                       uint32_t a3, uint32_t b0, uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// The exact sum of an element: h * 2^40 + l, in units of 2^(Ea + Eb - 76), 0 <= l < 2^40.
struct __align__(16) DgSum {
  int64_t h, l;
};
static_assert(kDgDiag == 9, "the sum below is written for nine diagonals");
// the diagonals' sums f (|f_d| <= 2^24) added to o
__device__ __forceinline__ DgSum dg_sum(const float (&f)[kDgDiag], const DgSum &o) {
  int v[kDgDiag];
#pragma unroll
  for (int d = 0; d < kDgDiag; d++) v[d] = __float2int_rn(f[d]);
  // |v_0| <= 64^2 * 144, |v_2| <= (2 * 64 * 128 + 128^2) * 144: these pairs fit 32 bits
  const int64_t h = ((int64_t)((v[0] << 8) + v[1]) << 16) + ((v[2] << 8) + v[3]);
  const int64_t l = ((int64_t)v[4] << 32) + ((int64_t)v[5] << 24) + ((int64_t)v[6] << 16) +
                    ((int64_t)v[7] << 8) + v[8] + o.l;
  return {o.h + h + (l >> 40), l & ((1ll << 40) - 1)};
}
__device__ __forceinline__ double dg_value(const DgSum &s) {
  return fma((double)s.h, 0x1p40, (double)s.l);
}
// v * 2^e for v = 0 or 2^-100 <= |v| <= 2^200 (no FP64 instruction while the result
// is a normal number)
__device__ __forceinline__ double dg_scaled(double v, int e) {
  const int hi = __double2hiint(v), x = ((hi >> 20) & 0x7FF) + e;
  if (v == 0.0) return v;
  if (x > 0 && x < 2047) return __hiloint2double(hi + (e << 20), __double2loint(v));
  const int half = max(e, -800);
  return v * __hiloint2double((1023 + half) << 20, 0) * __hiloint2double((1023 + e - half) << 20, 0);
}

// Fields of a block's metadata: octets, values of k, class, sum of a row.
__device__ __forceinline__ int dg_octets(uint2 x) { return (int)(x.y & kDigitMaxOctets); }
__device__ __forceinline__ int dg_length(uint2 x) {
  return 8 * dg_octets(x) - (int)(x.y >> kDigitPadAt & 7);
}
__device__ __forceinline__ int dg_class(uint2 x) { return (int)(x.y >> kDigitClassAt & 0x3F); }
__device__ __forceinline__ uint32_t dg_sum_code(uint2 x) { return x.y >> kDigitSumAt & 0x7F; }

// A word of a unit (digits 2 i and 2 i + 1 of two values) as the two MMA registers.
__device__ __forceinline__ uint32_t dg_even(uint32_t w) { return digit_half2(w, 0x4140); }
__device__ __forceinline__ uint32_t dg_odd(uint32_t w) { return digit_half2(w, 0x4342); }

// One tile of a C block that has no operand block outside: rows from 16 mt of A,
// columns from 8 nt of B, tm x tn; out (column-major) receives the tile's sums of
// the products of one class, which is returned (their weight is 2^(-8 class)); the
// sums of the classes before it are added up in part, if there are any (*parts).
// m, n: the block's sizes; prods: its np products, ma and mb the metadata of the
// first 32 (one per lane).
template <bool WIDE>
__device__ __forceinline__ int dg_tile(const Digits &dg, const int2 *__restrict__ prods, int np,
                                        uint2 ma, uint2 mb, int m, int n, int mt, int nt, int tm,
                                        int tn, DgSum *out, double *part, bool *parts, int lane) {
  const int g = lane >> 2, t = lane & 3;
  // the lane's units of an octet (rows past the last one: the last one again)
  const uint4 *__restrict__ ua = dg.a.units + min(g, tm - 1) * 4 + t;
  const uint4 *__restrict__ ub = dg.b.units + min(g, tn - 1) * 4 + t;
  const int low = (min(g + 8, tm - 1) - min(g, tm - 1)) * 4;  // to MMA row g + 8's
  struct Raw {  // an MMA step: two octets
    uint4 a[2], a8[2], b[2];
  };
  float acc[kDgDiag][4];
  auto mma = [&](const Raw &f) {
    uint32_t b[2][kDigits];
#pragma unroll
    for (int h = 0; h < 2; h++) {
      b[h][0] = dg_even(f.b[h].x), b[h][1] = dg_odd(f.b[h].x);
      b[h][2] = dg_even(f.b[h].y), b[h][3] = dg_odd(f.b[h].y);
      b[h][4] = dg_even(f.b[h].z), b[h][5] = dg_odd(f.b[h].z);
      b[h][6] = dg_even(f.b[h].w), b[h][7] = dg_odd(f.b[h].w);
    }
#pragma unroll
    for (int i = 0; i < kDigits; i += 2) {
      auto word = [&](const uint4 &u) { return i == 0 ? u.x : i == 2 ? u.y : i == 4 ? u.z : u.w; };
      if (WIDE) {
        uint32_t a0 = dg_even(word(f.a[0])), a1 = dg_even(word(f.a8[0]));
        uint32_t a2 = dg_even(word(f.a[1])), a3 = dg_even(word(f.a8[1]));
#pragma unroll
        for (int j = 0; j < kDigits; j++)
          if (i + j < kDgDiag) dg_mma(acc[i + j], a0, a1, a2, a3, b[0][j], b[1][j]);
        a0 = dg_odd(word(f.a[0])), a1 = dg_odd(word(f.a8[0]));
        a2 = dg_odd(word(f.a[1])), a3 = dg_odd(word(f.a8[1]));
#pragma unroll
        for (int j = 0; j < kDigits; j++)
          if (i + 1 + j < kDgDiag) dg_mma(acc[i + 1 + j], a0, a1, a2, a3, b[0][j], b[1][j]);
      } else {
        const uint32_t a0 = dg_even(word(f.a[0])), a1 = dg_odd(word(f.a[0]));
        const uint32_t a2 = dg_even(word(f.a[1])), a3 = dg_odd(word(f.a[1]));
#pragma unroll
        for (int j = 0; j < kDigits; j++)
          if (i + j < kDgDiag) dg_mma(acc[i + j], a0, a1, a2, a3, b[0][j], b[1][j]);
      }
    }
  };
  int held = -1;  // the class of the sums in out
  *parts = false;
  for (int pb = 0;;) {
    const uint2 xa = ma, xb = mb;  // lane p: product p of the batch
    const bool in = pb + lane < np;
    const int cls = dg_class(xa) + dg_class(xb);
    pb += 32;
    if (pb < np) {  // the next batch's metadata, on its way during this one
      ma = mb = make_uint2(0, 0);
      if (pb + lane < np) {
        const int2 pr = __ldg(prods + pb + lane);
        ma = __ldg(dg.a.meta + pr.x);
        mb = __ldg(dg.b.meta + pr.y);
      }
    }
    // the products of one class (the weight 2^(-8 class)) after the other: mostly
    // all have the same
    uint32_t todo = __ballot_sync(0xffffffffu, in);
#pragma unroll 1
    while (todo) {
      const int now = __shfl_sync(0xffffffffu, cls, __ffs(todo) - 1);
      const bool mine = in && cls == now;
      todo &= ~__ballot_sync(0xffffffffu, mine);
      // its octets' end, and its units less its first slot's
      const int octets = mine ? dg_octets(xa) : 0;
      int incl = octets;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
      }
      const int slots = __shfl_sync(0xffffffffu, incl, 31);
      const uint32_t am = xa.x + (uint32_t)(64 * mt - (incl - octets) * 4 * m);
      const uint32_t bm = xb.x + (uint32_t)(32 * nt - (incl - octets) * 4 * n);
      if (held >= 0 && held != now) {
        __syncwarp();
        for (int e = lane; e < tm * tn; e += 32) {
          const double v = dg_scaled(dg_value(out[e]), -8 * held);
          part[e] = *parts ? part[e] + v : v;
        }
        __syncwarp();
        *parts = true;
        held = -1;
      }
#pragma unroll 1
      for (int s0 = 0; s0 < slots; s0 += kDgFold) {
        // lane l: where the units of slot s0 + l start (zeros past the end)
        const int s = s0 + lane;
        int p = 0;  // products that end at or before slot s
#pragma unroll
        for (int step = 16; step; step >>= 1)
          if (__shfl_sync(0xffffffffu, incl, p + step - 1) <= s) p += step;
        uint32_t fa = __shfl_sync(0xffffffffu, am, p) + (uint32_t)(s * 4 * m);
        uint32_t fb = __shfl_sync(0xffffffffu, bm, p) + (uint32_t)(s * 4 * n);
        if (s >= slots) fa = fb = 0;
        auto load = [&](Raw &f, int o) {
#pragma unroll
          for (int h = 0; h < 2; h++) {
            const uint4 *xa = ua + __shfl_sync(0xffffffffu, fa, o + h);
            f.a[h] = __ldg(xa);
            if (WIDE) f.a8[h] = __ldg(xa + low);
            f.b[h] = __ldg(ub + __shfl_sync(0xffffffffu, fb, o + h));
          }
        };
#pragma unroll
        for (int d = 0; d < kDgDiag; d++)
#pragma unroll
          for (int e = 0; e < 4; e++) acc[d][e] = 0.0f;
        const int end = min(kDgFold, slots - s0);
#pragma unroll 1
        for (int o = 0; o < end; o += 2) {
          Raw f0;
          load(f0, o);
          mma(f0);
        }
#pragma unroll
        for (int e = 0; e < (WIDE ? 4 : 2); e++) {
          float f[kDgDiag];
#pragma unroll
          for (int d = 0; d < kDgDiag; d++)
            f[d] = (WIDE || d == 0) ? acc[d][e] : __fadd_rn(acc[d][e], acc[d - 1][e + 2]);
          const int x = g + (e >> 1) * 8, y = 2 * t + (e & 1);
          if (x < tm && y < tn) {
            DgSum *to = out + (y * tm + x);
            *to = dg_sum(f, held < 0 ? DgSum{0, 0} : *to);
          }
        }
        held = now;
      }
    }
    if (pb >= np) return held;
  }
}

// Whether the digits hold enough of a C block. A product of s values of k loses at most
// 2^-63 (sa + sb) + 2^-67.4 s in units of W, the product of the row's and the column's scale
// less the classes: half a unit of X for each value of one side beside the other side's
// values, whose absolute sum over k is at most sa (sb) of the scale, and the digit pairs
// beyond kDgDiag. Over the C block, N values of k in all, the first may come to sqrt(N) 2^-53
// of the element's sum of absolute products, the second to 3 sqrt(N) 2^-53 (of both, the
// fractions of their limits to 1). FP64 FMAs lose up to N 2^-53 of that sum. What they lose of
// ordinary elements is 0.4 2^-53 of it where terms are alike, as the second, being a sum of
// many independent parts, at its limit; and 0.3 sqrt(N) 2^-53 where one term is most of the sum,
// as where the first comes near its limit.
// The sum of absolute products is bounded from below by the two top digits t of both
// values (2^14 of the scale): t_a t_b less the digits' rounding, added up by one MMA for
// every 16 k. Any part of the products will do, so those of the largest scales go first and
// it ends when every element has enough, mostly after the first one or two. C blocks that
// have not enough with all of theirs are left to the packed kernel.
// sa + sb
__device__ __forceinline__ float dg_sums(uint2 a, uint2 b) {
  return digit_sum_of(dg_sum_code(a)) + digit_sum_of(dg_sum_code(b));
}
// the weight of products whose classes add up to d more than the least (2 and more: at most this)
__device__ __forceinline__ float dg_weight(int d) {
  return d == 0 ? 1.0f : d == 1 ? 0x1p-8f : 0x1p-16f;
}

// What the sums of t_a t_b have to reach; infinity where an operand block is outside.
// least: the least sum of two classes.
__device__ __forceinline__ float dg_need(const Digits &dg, const int2 *__restrict__ prods, int np,
                                         uint2 ma, uint2 mb, int &least, int lane) {
  auto loss = [&](uint2 a, uint2 b) {
    return 3 * 0x1p18f * dg_sums(a, b) + 12400.0f * (float)dg_length(a);
  };
  // the lane's products: their least class and their loss at its weight
  int cls = 1 << 10, n = 0;
  float sum = 0.0f;
  uint32_t flags = ma.y | mb.y;
  if (lane < np) {
    cls = dg_class(ma) + dg_class(mb);
    n = dg_length(ma);
    sum = loss(ma, mb);
  }
  for (int p = lane + 32; p < np; p += 32) {
    const int2 q = __ldg(prods + p);
    const uint2 a = __ldg(dg.a.meta + q.x), b = __ldg(dg.b.meta + q.y);
    const int c = dg_class(a) + dg_class(b), now = min(c, cls);
    sum = sum * dg_weight(cls - now) + loss(a, b) * dg_weight(c - now);
    cls = now;
    n += dg_length(a);
    flags |= a.y | b.y;
  }
  if (__any_sync(0xffffffffu, flags & kDigitOutside)) return INFINITY;
  least = __reduce_min_sync(0xffffffffu, cls);
  n = __reduce_add_sync(0xffffffffu, n);
  sum *= dg_weight(cls - least);
#pragma unroll
  for (int d = 16; d; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
  // t carries 11 bits, the sums 24, the root and the quotient 20: 1% covers them
  return 1.01f / 3.0f * sum * rsqrtf((float)n);
}

__device__ __forceinline__ uint32_t dg_top(uint32_t w) {  // |256 d_0 + d_1| of two values
  uint32_t h = dg_even(w);
  asm("fma.rn.f16x2 %0, %0, %1, %2;\n" : "+r"(h) : "r"(0x5C005C00u), "r"(dg_odd(w)));
  return h & 0x7FFF7FFFu;
}

// Products that are looked at before a tile may be given up: operands whose values cancel
// along k by 2^-10 to 2^10 (water of 512 molecules, every C block left to the packed kernel)
// 14.2 ms with all products looked at, 13.1 so, 12.2 for the packed kernel alone.
constexpr int kDgLook = 3;

// Whether each element of a tile reaches `need`: rows from r0 of A and columns from c0 of
// B, tm x tn of up to 16 x 16 (the left side's registers serve both halves of the columns).
__device__ __forceinline__ bool dg_enough(const Digits &dg, const int2 *__restrict__ prods, int np,
                                          uint2 ma, uint2 mb, int m, int n, int r0, int c0, int tm,
                                          int tn, float need, int least, int lane) {
  const int g = lane >> 2, t = lane & 3;
  // rows and columns past the last one: the last one again, so that every sum is an element's
  const uint4 *__restrict__ ua = dg.a.units + min(g, tm - 1) * 4 + t;
  const uint4 *__restrict__ ub = dg.b.units + min(g, tn - 1) * 4 + t;
  const int low = (min(g + 8, tm - 1) - min(g, tm - 1)) * 4;
  const int right = (min(g + 8, tn - 1) - min(g, tn - 1)) * 4;
  float sum[2][4] = {};
  int seen = 0;
  for (int pb = 0;;) {
    const int above = dg_class(ma) + dg_class(mb) - least;
    uint32_t key = pb + lane < np && above <= 1
                       ? (32 * above + 254 - dg_sum_code(ma) - dg_sum_code(mb)) << 5 | lane
                       : ~0u;
#pragma unroll 1
    for (;;) {
      const uint32_t best = __reduce_min_sync(0xffffffffu, key);
      if (best == ~0u) break;
      const int p = best & 31;
      if (lane == p) key = ~0u;
      const uint2 xa = make_uint2(__shfl_sync(0xffffffffu, ma.x, p), __shfl_sync(0xffffffffu, ma.y, p));
      const uint2 xb = make_uint2(__shfl_sync(0xffffffffu, mb.x, p), __shfl_sync(0xffffffffu, mb.y, p));
      const int octets = dg_octets(xa);
      float acc[2][4] = {};
#pragma unroll 1
      for (int o = 0; o < octets; o += 2) {
        uint32_t a[2], a8[2], b[2], b8[2];
#pragma unroll
        for (int h = 0; h < 2; h++) {
          const bool in = o + h < octets;  // else zeros
          const uint4 *pa = ua + (in ? xa.x + (uint32_t)(4 * r0 + (o + h) * 4 * m) : 0u);
          const uint4 *pb = ub + (in ? xb.x + (uint32_t)(4 * c0 + (o + h) * 4 * n) : 0u);
          a[h] = __ldg(&pa->x);
          a8[h] = __ldg(&pa[low].x);
          b[h] = __ldg(&pb->x);
          if (tn > 8) b8[h] = __ldg(&pb[right].x);
        }
        const uint32_t x0 = dg_top(a[0]), x1 = dg_top(a8[0]), x2 = dg_top(a[1]), x3 = dg_top(a8[1]);
        dg_mma(acc[0], x0, x1, x2, x3, dg_top(b[0]), dg_top(b[1]));
        if (tn > 8) dg_mma(acc[1], x0, x1, x2, x3, dg_top(b8[0]), dg_top(b8[1]));
      }
      const float w = dg_weight(dg_class(xa) + dg_class(xb) - least);
      // t may be 0.503 above the value: what that adds at most
      need += w * (8260.0f * dg_sums(xa, xb) + 0.3f * (float)dg_length(xa));
      float some = INFINITY;  // the least sum of the lane's elements
#pragma unroll
      for (int e = 0; e < 4; e++) {
        sum[0][e] += w * acc[0][e];
        sum[1][e] += w * acc[1][e];
        some = fminf(some, tn <= 8 ? sum[0][e] : fminf(sum[0][e], sum[1][e]));
      }
      if (__all_sync(0xffffffffu, some >= need)) return true;
      // not with four times as much from each of the others, which are smaller: no use going on
      if (++seen >= kDgLook &&
          __any_sync(0xffffffffu, some * (float)(4 * np) < need * (float)seen)) return false;
    }
    pb += 32;
    if (pb >= np) return false;
    ma = mb = make_uint2(0, 0);
    if (pb + lane < np) {
      const int2 pr = __ldg(prods + pb + lane);
      ma = __ldg(dg.a.meta + pr.x);
      mb = __ldg(dg.b.meta + pr.y);
    }
  }
}

struct DgItem {  // a C block of a warp's run
  const int2 *prods;
  int64_t coff;
  int32_t gblk, np, m, n, cin, fa, fb;
  int32_t part, nparts;  // the part of its tiles that is to be done
  int32_t at;            // its number in the work range
};
// words of the bits in dg.marks: a bit for each C block that is split into parts
constexpr int dg_mark_words(int warps) { return (kDgUnits * warps / 2 + 31) / 32; }
int64_t digit_state_bytes(int nsm) {
  return 2 * sizeof(int64_t) + 4 * (int64_t)dg_mark_words(nsm * kDgBlocksPerSm * kDgWarps);
}

// C blocks without products (C_in only), with an operand block outside or with too little
// of the digits go to dg.list, for the packed kernel (whose values replace those that other
// parts of such a block have stored).
__global__ void __launch_bounds__(kDgWarps * 32, kDgBlocksPerSm)
    k_numeric_fp64_dg(DevMat A, DevMat B, DevOut C, DevMat Cin, double alpha, double beta,
                      DevWs ws, const DevStatus *st, const int32_t *items, const int64_t *seg,
                      unsigned long long *work, Digits dg, int ntiles) {
  if (st->overflow) return;
  __shared__ DgSum tiles[kDgWarps][16 * 8];
  __shared__ double parts[kDgWarps][16 * 8];
  __shared__ DgItem s_items[kDgWarps][kDgGrab];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  DgSum *tile = tiles[warp];
  double *part = parts[warp];
  DgItem *item = s_items[warp];
  int64_t wb, we;
  work_range(st, seg, wb, we);
  double *hout = (C.host_vals && st->nnz_c <= C.host_cap) ? C.host_vals : nullptr;
  // fewer at a time where that would leave warps without work
  const int64_t warps = (int64_t)gridDim.x * kDgWarps;
  // the parts of a C block (every nparts-th of its tiles), a unit of work each
  const int nparts =
      (int)min((int64_t)ntiles, max((int64_t)1, kDgUnits * warps / max((int64_t)1, we - wb)));
  we = wb + (we - wb) * nparts;
  // Towards the end shorter runs, a quarter to an eighth of what is left for each warp,
  // so that the warps end together (a fixed length: water of 64 molecules 0.66 ms, of 512
  // 5.45, blocks of 1 to 33 in 200 rows 1.25; this 0.61, 5.34 and 1.02).
  const int shift = 34 - __clz((int)warps);
  int64_t base = wb;
  for (;;) {
    const int grab = (int)max((int64_t)1, min((int64_t)kDgGrab, (we - base) >> shift));
    unsigned long long got = 0;
    if (lane == 0) got = atomicAdd(work, (unsigned long long)grab);
    base = wb + (int64_t)__shfl_sync(0xffffffffu, got, 0);
    if (base >= we) break;
    const int count = we - base < grab ? (int)(we - base) : grab;
    // what the C blocks of the run need, a lane each: the next block is then found
    // without a chain of loads
    if (lane < count) {
      DgItem it;
      const int64_t unit = base + lane - wb, blk = nparts > 1 ? wb + unit / nparts : base + lane;
      it.part = nparts > 1 ? (int)(unit % nparts) : 0;
      it.nparts = nparts;
      it.gblk = items ? items[blk] : (int)blk;
      it.at = (int)(blk - wb);
      const int64_t pp = ws.prod_ptr[it.gblk];
      it.prods = ws.prods + pp;
      it.np = (int)(ws.prod_ptr[it.gblk + 1] - pp);
      const int i = C.blk_row[it.gblk], j = C.col_idx[it.gblk];
      it.m = C.row_sizes[i];
      it.n = C.col_sizes[j];
      it.coff = C.blk_off[it.gblk];
      it.cin = ws.c_cin[it.gblk];
      it.fa = dg.a.first[i];
      it.fb = dg.b.first[j];
      item[lane] = it;
    }
    __syncwarp();
    // a block's products and their metadata are loaded while the block before is
    // computed
    int2 pr = make_int2(-1, -1);
    auto products = [&](int at) {
      pr = make_int2(-1, -1);
      if (at < count && lane < item[at].np) pr = __ldg(item[at].prods + lane);
    };
    uint2 ma, mb;
    auto metadata = [&]() {
      ma = mb = make_uint2(0, 0);
      if (pr.x >= 0) {
        ma = __ldg(dg.a.meta + pr.x);
        mb = __ldg(dg.b.meta + pr.y);
      }
    };
    products(0);
    metadata();
    for (int x = 0; x < count; x++) {
      const DgItem &it = item[x];
      products(x + 1);
      const int np = it.np;
      const int m = it.m, n = it.n;
      const uint2 ka = ma, kb = mb;
      int at = 0;  // the tile's number
      int least;
      const float need = np > 0 ? dg_need(dg, it.prods, np, ka, kb, least, lane) : INFINITY;
      bool held = need < INFINITY;
      bool first = it.part == 0;  // that finds out
      if (held) {
        for (int r0 = 0; r0 < m && held; r0 += 16)
          for (int c0 = 0; c0 < n && held; c0 += 16) {
            if (it.nparts > 1 && at++ % it.nparts != it.part) continue;
            held = dg_enough(dg, it.prods, np, ka, kb, m, n, r0, c0, min(16, m - r0),
                             min(16, n - c0), need, least, lane);
          }
        at = 0;
        if (!held && it.nparts > 1 && lane == 0) {
          const uint32_t bit = 1u << (it.at & 31);
          first = !(atomicOr(dg.marks + (it.at >> 5), bit) & bit);
        }
      }
      if (!held) {
        if (lane == 0 && first)
          dg.list[atomicAdd(reinterpret_cast<unsigned long long *>(dg.range + 1), 1ull)] = it.gblk;
        metadata();
        continue;
      }
      for (int r0 = 0; r0 < m; r0 += 16) {
        for (int c0 = 0; c0 < n; c0 += 8) {
          if (it.nparts > 1 && at++ % it.nparts != it.part) continue;
          const int tm = min(16, m - r0), tn = min(8, n - c0);
          // the exponents of the tile's scales: lane r row r's, lane c column c's
          const int xa = dg.a.expo[it.fa + r0 + min(lane, tm - 1)];
          const int xb = dg.b.expo[it.fb + c0 + min(lane, tn - 1)];
          bool more;
          const int cls = tm > 8 ? dg_tile<true>(dg, it.prods, np, ka, kb, m, n, r0 >> 4, c0 >> 3,
                                                 tm, tn, tile, part, &more, lane)
                                 : dg_tile<false>(dg, it.prods, np, ka, kb, m, n, r0 >> 4, c0 >> 3,
                                                  tm, tn, tile, part, &more, lane);
          __syncwarp();
          const double *cinv = (it.cin >= 0) ? Cin.vals + Cin.blk_off[it.cin] : nullptr;
          const uint32_t rtm = rcp16(tm);
          for (int e0 = 0; e0 < tm * tn; e0 += 32) {
            const int e = e0 + lane, c = div16(e, rtm), r = e - c * tm;
            // 2^(Ea + Eb - 76), E = field - 1022; a row without a scale holds only zeros
            const int fa = __shfl_sync(0xffffffffu, xa, r), fb = __shfl_sync(0xffffffffu, xb, c & 31);
            if (e >= tm * tn) continue;
            const int f = (fa >= kDigitExpLo && fb >= kDigitExpLo) ? fa + fb - 2044 - 76 : 0;
            const int64_t loc = it.coff + (int64_t)(c0 + c) * m + r0 + r;
            double v = dg_value(tile[e]);
            if (more) v = part[e] + dg_scaled(v, -8 * cls);
            v = dg_scaled(v, more ? f : f - 8 * cls);
            if (alpha != 1.0) v *= alpha;
            if (cinv) v = fma(beta, cinv[loc - it.coff], v);
            // written once, not read by this multiply
            __stcs(C.vals + loc, v);
            if (hout) __stcs(hout + loc, v);
          }
          __syncwarp();
        }
      }
      metadata();
    }
    __syncwarp();  // the items are read before the next ones are written
  }
}

// The tiles of a C block of m x n, at most (block sizes may be anything below 2^31).
static int tiles_of(int m, int n, int tm, int tn) {
  const int64_t t = (((int64_t)m + tm - 1) / tm) * (((int64_t)n + tn - 1) / tn);
  return (int)std::min<int64_t>(t, INT32_MAX);
}

cudaError_t launch_numeric_fp64(int variant, DevMat A, DevMat B, DevOut C, DevMat Cin,
                                double alpha, double beta, DevWs ws, const DevStatus *st,
                                const int32_t *items, const int64_t *seg, int grid,
                                unsigned long long *work, int max_m, int max_n, const Digits *digits,
                                cudaStream_t stream) {
  switch (variant) {
    case kFp64Dg:
      k_numeric_fp64_dg<<<grid, kDgWarps * 32, 0, stream>>>(
          A, B, C, Cin, alpha, beta, ws, st, items, seg, work, *digits, tiles_of(max_m, max_n, 16, 8));
      break;
    case kFp64G8: {
      const int mr = max_m <= 4 ? 4 : max_m <= 6 ? 6 : 8;
      const int gs = max_n <= 4 ? 4 : max_n <= 6 ? 6 : 8;
      const bool direct = !C.host_vals && max_m <= 8 && max_n <= 8 &&
                          (alpha != 1.0 || beta != 0.0 || (mr == 4 && gs == 4));
// the shared memory is opted into here, for the one instance (it loads its code)
#define BSM_G8(R, G)                                                                             \
  do {                                                                                           \
    if (direct) {                                                                                \
      k_numeric_fp64_g8_direct<R, G>                                                             \
          <<<grid / kG8BlocksPerSm * kG8DirectBlocksPerSm, kG8Warps * 32, 0, stream>>>(          \
              A, B, C, Cin, alpha, beta, ws, st, items, seg, work);                              \
      break;                                                                                     \
    }                                                                                            \
    const cudaError_t e = cudaFuncSetAttribute(                                                  \
        k_numeric_fp64_g8<R, G>, cudaFuncAttributeMaxDynamicSharedMemorySize,                    \
        (int)g8_smem_bytes());                                                                   \
    if (e != cudaSuccess) return e;                                                              \
    k_numeric_fp64_g8<R, G><<<grid, kG8Warps * 32, g8_smem_bytes(), stream>>>(                   \
        A, B, C, Cin, alpha, beta, ws, st, items, seg, work);                                    \
  } while (0)
      if (mr == 4) {
        if (gs == 4) BSM_G8(4, 4); else if (gs == 6) BSM_G8(4, 6); else BSM_G8(4, 8);
      } else if (mr == 6) {
        if (gs == 4) BSM_G8(6, 4); else if (gs == 6) BSM_G8(6, 6); else BSM_G8(6, 8);
      } else {
        if (gs == 4) BSM_G8(8, 4); else if (gs == 6) BSM_G8(8, 6); else BSM_G8(8, 8);
      }
#undef BSM_G8
      break;
    }
    case kFp64T16B3:
      k_numeric_fp64_t16<3><<<grid, kSWarps * 32, 0, stream>>>(A, B, C, Cin, alpha, beta, ws, st,
                                                               items, seg, work);
      break;
    case kFp64T32: {
      // the shared-memory attribute is set once per device by numeric_fp64_init
      const size_t smem = (size_t)kNumWarps * kWarpSmem * sizeof(double);
      k_numeric_fp64_t32<<<grid, kNumWarps * 32, smem, stream>>>(A, B, C, Cin, alpha, beta, ws,
                                                                 st, items, seg);
      break;
    }
    case kFp64Pk12:
      // digits: the blocks that the digit kernel left, tile by tile
      k_numeric_fp64_pk<12><<<grid, kPkWarps * 32, pk_smem_bytes(), stream>>>(
          A, B, C, Cin, alpha, beta, ws, st, items, seg, work,
          digits ? tiles_of(max_m, max_n, kPkTile, kPkTile) : 0);
      break;
    case kFp64Pk16:
      k_numeric_fp64_pk<16><<<grid, kPkWarps * 32, pk_smem_bytes(), stream>>>(
          A, B, C, Cin, alpha, beta, ws, st, items, seg, work, 0);
      break;
    default:
      k_numeric_fp64_t16<2><<<grid, kSWarps * 32, 0, stream>>>(A, B, C, Cin, alpha, beta, ws, st,
                                                               items, seg, work);
  }
  return cudaGetLastError();
}

int fp64_variant_blocks_per_sm(int variant) {
  if (variant == kFp64Dg) return kDgBlocksPerSm;
  if (variant == kFp64G8) return kG8BlocksPerSm;
  return (variant == kFp64T16B3 || variant == kFp64T32) ? 3 : 2;
}

cudaError_t numeric_fp64_init() {
  const size_t smem = (size_t)kNumWarps * kWarpSmem * sizeof(double);
  cudaError_t e = cudaFuncSetAttribute(k_numeric_fp64_t32,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // its operands come through L1: no more shared memory than its own
  e = cudaFuncSetAttribute(k_numeric_fp64_dg, cudaFuncAttributePreferredSharedMemoryCarveout, 50);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_numeric_fp64_pk<12>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)pk_smem_bytes());
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_numeric_fp64_pk<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)pk_smem_bytes());
}

}  // namespace bsm
