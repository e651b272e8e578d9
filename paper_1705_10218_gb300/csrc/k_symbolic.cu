// k_symbolic.cu -- block norms, symbolic phase with the on-the-fly filter,
// and the per-C-block grouping of the kept products.
//
// Sec. 2 of the paper: the result pattern is determined by the multiplication
// itself, and a block product is only performed when the product of the two
// block norms passes the threshold. Here that becomes three device passes:
//   count: per C block row, the set of columns reached by a kept product
//          (a bitmap in shared memory), the number of kept products, FLOPs;
//   scan:  exclusive sums over block rows -> C's row pointers, product and
//          value offsets, and the capacity check of the output buffers;
//   fill:  per C block row, the sorted column list of C, every C block's
//          value offset, and the kept products written grouped by C block in
//          ascending k (a per-row counting sort), so that the numeric phase
//          accumulates each C block in one place, without atomics.
#include <type_traits>

#include "bsm_internal.h"
#include "digits.cuh"

namespace bsm {

// The filter of Sec. 2: drop iff nrm(A_ik)*nrm(B_kj) < eps (a tie and NaN are kept),
// decided exactly as FP64 decides it.
__device__ __forceinline__ bool keep_product(double na, double nb, double eps) {
  return !(__dmul_rn(na, nb) < eps);
}

// The same decision with FP32 arithmetic for all but the near-ties. The FP32
// copies of the norms are within 2^-24 (relative) of the FP64 norms and lie in
// [2^-60, 2^60] (else NaN), so their FP32 product is within 3*2^-24 of the
// exact product; it is compared with eps widened by 2^-20 either way (lo, hi),
// and only a product inside that band (or a NaN) takes the FP64 test.
struct EpsBand {
  float lo, hi;
};

__device__ __forceinline__ EpsBand eps_band(double eps) {
  EpsBand b;
  if (!(eps > 0.0)) {  // eps <= 0 (or NaN eps): every non-NaN product is kept
    b.lo = -INFINITY;
    b.hi = -INFINITY;
  } else if (eps >= 0x1p-100 && eps <= 0x1p100) {
    b.lo = __double2float_rd(eps * (1.0 - 0x1p-20));
    b.hi = __double2float_ru(eps * (1.0 + 0x1p-20));
  } else {  // out of the fast test's range: always the FP64 test
    b.lo = -INFINITY;
    b.hi = INFINITY;
  }
  if (eps != eps) {
    b.lo = -INFINITY;
    b.hi = INFINITY;
  }
  return b;
}

__device__ __forceinline__ bool keep_fast(float fa, float fb, double na, double nb, double eps,
                                          const EpsBand &band) {
  const float x = fa * fb;
  if (x >= band.hi) return true;
  if (x < band.lo) return false;
  return keep_product(na, nb, eps);
}

__device__ __forceinline__ int lower_bound_i32(const int32_t *a, int lo, int hi, int key) {
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (a[mid] < key) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// ----------------------------------------------------------------------------
// Block norms: canonical Frobenius norm, column-major, no fused multiply-add; the
// block count is read on the device so that a matrix produced by an earlier multiply
// needs no host round trip. And the scales of the digit representation in the same
// launch (rexp, cexp: where they are wanted): the first thread blocks take the norms,
// the others the scales, a warp per block: each lane's elements go to their row's and
// column's maximum in shared memory, and a maximum that the array does not hold yet there.
//
// A norm's additions have a fixed order, so a block's chain of them is one lane's. The
// FP64 pipe takes a warp's instruction in 64 clocks of a quarter SM, whatever its
// active lanes: many blocks are a lane each (its loads eight ahead). Where that would
// leave quarters idle, LANES lanes share a block: each loads and squares every
// LANES-th value, and all follow the additions, so that the chain is an addition per
// value instead of an addition and a multiplication, with loads of whole sectors; and
// consecutive warps' blocks go to different SMs. 2795 + 2487 blocks of up to 33 x 33:
// 140 + 138 -> 74 + 74 us, of which 17 + 17 are the scales.
// ----------------------------------------------------------------------------
constexpr int kScaleWarps = 8;
constexpr int kNormAhead = 8;   // loads of a lane in flight
constexpr int kNormBlocksPerSm = 8;
constexpr int kScaleRows = 64;  // rows and columns kept in shared memory

// The sum of squares of the n values at x, in order; LANES lanes of a warp have the
// same x and n, sub is the lane's number among them. All lanes of the warp take part.
template <int LANES>
__device__ __forceinline__ double sum_of_squares(const double *__restrict__ x, int64_t n, int sub) {
  double s = 0.0;
  if (LANES == 1) {
    double v[kNormAhead];
    int64_t e = 0;
    for (; e + kNormAhead <= n; e += kNormAhead) {
#pragma unroll
      for (int u = 0; u < kNormAhead; u++) v[u] = __ldg(x + e + u);
#pragma unroll
      for (int u = 0; u < kNormAhead; u++) s = __dadd_rn(s, __dmul_rn(v[u], v[u]));
    }
    for (; e < n; e++) {
      const double y = __ldg(x + e);
      s = __dadd_rn(s, __dmul_rn(y, y));
    }
    return s;
  }
  constexpr int kAhead = kNormAhead / 2, kStep = LANES * kAhead;
  double v[kAhead];
  auto load = [&](int64_t e) {
#pragma unroll
    for (int u = 0; u < kAhead; u++)
      v[u] = e + u * LANES + sub < n ? __ldg(x + e + u * LANES + sub) : 0.0;
  };
  load(0);
  int64_t most = n;
  for (int d = LANES; d < 32; d <<= 1)
    most = max(most, __shfl_xor_sync(0xffffffffu, most, d));
  for (int64_t e = 0; e < most; e += kStep) {
    double q[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; u++) q[u] = __dmul_rn(v[u], v[u]);
    load(e + kStep);
#pragma unroll
    for (int u = 0; u < kAhead; u++)
#pragma unroll
      for (int l = 0; l < LANES; l++) {
        const double y = __shfl_sync(0xffffffffu, q[u], l, LANES);
        if (e + u * LANES + l < n) s = __dadd_rn(s, y);
      }
  }
  return s;
}

template <int LANES>
__device__ __forceinline__ void block_norms(const int32_t *__restrict__ row_sizes,
                                            const int32_t *__restrict__ col_sizes,
                                            const int32_t *__restrict__ blk_row,
                                            const int32_t *__restrict__ col_idx,
                                            const int64_t *__restrict__ blk_off,
                                            const double *__restrict__ vals, int64_t nblk,
                                            double *__restrict__ norms, float *__restrict__ normsf,
                                            int norm_blocks, int nsm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kPerWarp = 32 / LANES;
  // the thread blocks of an SM start with warps of different quarters of it
  const int turn = (warp + blockIdx.x / nsm) % kScaleWarps;
  for (int64_t w = (int64_t)turn * norm_blocks + blockIdx.x; w * kPerWarp < nblk;
       w += (int64_t)norm_blocks * kScaleWarps) {
    const int64_t b = w * kPerWarp + lane / LANES;
    const bool in = b < nblk;
    const int64_t n = in ? (int64_t)row_sizes[blk_row[b]] * col_sizes[col_idx[b]] : 0;
    const double s = sum_of_squares<LANES>(vals + (in ? blk_off[b] : 0), n, lane % LANES);
    if (!in || lane % LANES) continue;
    const double nrm = __dsqrt_rn(s);
    norms[b] = nrm;
    normsf[b] = (nrm >= 0x1p-60 && nrm <= 0x1p60) ? __double2float_rn(nrm) : NAN;
  }
}

__global__ void __launch_bounds__(kScaleWarps * 32, 5)
    k_block_norms_scales(const int32_t *__restrict__ row_sizes,
                         const int32_t *__restrict__ col_sizes,
                         const int32_t *__restrict__ blk_row, const int32_t *__restrict__ col_idx,
                         const int64_t *__restrict__ blk_off, const double *__restrict__ vals,
                         const int64_t *__restrict__ hdr, double *__restrict__ norms,
                         float *__restrict__ normsf, const int32_t *__restrict__ rfirst,
                         const int32_t *__restrict__ cfirst, int32_t *rexp, int32_t *cexp,
                         int norm_blocks) {
  const int64_t nblk = hdr[0];
  if ((int)blockIdx.x < norm_blocks) {
    auto norms_by = [&](auto lanes) {
      block_norms<decltype(lanes)::value>(row_sizes, col_sizes, blk_row, col_idx, blk_off, vals,
                                          nblk, norms, normsf, norm_blocks, norm_blocks / kNormBlocksPerSm);
    };
    // the most lanes that need no more warps than there are quarters of SMs
    const int64_t quarters = norm_blocks / kNormBlocksPerSm * 4;
    if (nblk <= 2 * quarters)
      norms_by(std::integral_constant<int, 16>{});
    else if (nblk <= 8 * quarters)
      norms_by(std::integral_constant<int, 4>{});
    else
      norms_by(std::integral_constant<int, 1>{});
    return;
  }
  __shared__ int32_t smax[kScaleWarps][2 * kScaleRows];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t *rmax = smax[warp], *cmax = rmax + kScaleRows;
  const int64_t w0 = (int64_t)(blockIdx.x - norm_blocks) * kScaleWarps + warp;
  const int64_t nw = (int64_t)(gridDim.x - norm_blocks) * kScaleWarps;
  for (int64_t b = w0; b < nblk; b += nw) {
    const int i = blk_row[b], j = col_idx[b];
    const int m = row_sizes[i], n = col_sizes[j];
    const double *x = vals + blk_off[b];
    int32_t *re = rexp ? rexp + rfirst[i] : nullptr, *ce = cexp ? cexp + cfirst[j] : nullptr;
    const bool shared = m <= kScaleRows && n <= kScaleRows;
    if (shared) {
      for (int r = lane; r < 2 * kScaleRows; r += 32) rmax[r] = 0;
      __syncwarp();
    }
    // element e: column c, row r; 32 elements on, four loads ahead
    const int64_t len = (int64_t)m * n;
    const int dc = 32 / m, dr = 32 - dc * m;
    int c = lane / m, r = lane - c * m;
    double v[4];
#pragma unroll
    for (int u = 0; u < 4; u++) v[u] = lane + 32 * u < len ? __ldg(x + lane + 32 * u) : 0.0;
    for (int64_t e = lane; e < len; e += 32) {
      const int f = digit_field(v[0]);
      v[0] = v[1], v[1] = v[2], v[2] = v[3];
      v[3] = e + 128 < len ? __ldg(x + e + 128) : 0.0;
      if (shared) {
        if (re) atomicMax(&rmax[r], f);
        if (ce) atomicMax(&cmax[c], f);
      } else {
        if (re && re[r] < f) atomicMax(re + r, f);
        if (ce && ce[c] < f) atomicMax(ce + c, f);
      }
      r += dr, c += dc;
      if (r >= m) r -= m, c++;
    }
    if (!shared) continue;
    __syncwarp();
    for (int r = lane; r < m; r += 32)  // a stale smaller value only costs an atomic
      if (re && re[r] < rmax[r]) atomicMax(re + r, rmax[r]);
    for (int c = lane; c < n; c += 32)
      if (ce && ce[c] < cmax[c]) atomicMax(ce + c, cmax[c]);
    __syncwarp();
  }
}

cudaError_t launch_block_norms_scales(const int32_t *row_sizes, const int32_t *col_sizes,
                                      const int32_t *blk_row, const int32_t *col_idx,
                                      const int64_t *blk_off, const double *vals,
                                      const int64_t *hdr, double *norms, float *normsf,
                                      const int32_t *rfirst, const int32_t *cfirst, int32_t *rexp,
                                      int32_t *cexp, int nsm, cudaStream_t stream) {
  const int norm_blocks = nsm * kNormBlocksPerSm, scale_blocks = (rexp || cexp) ? nsm * 4 : 0;
  k_block_norms_scales<<<norm_blocks + scale_blocks, kScaleWarps * 32, 0, stream>>>(
      row_sizes, col_sizes, blk_row, col_idx, blk_off, vals, hdr, norms, normsf, rfirst, cfirst,
      rexp, cexp, norm_blocks);
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// Block-wide exclusive scan of one int64 per thread (blockDim a multiple of 32,
// at most 1024). Returns the exclusive prefix; *total gets the block sum.
// ----------------------------------------------------------------------------
__device__ int64_t block_exclusive_scan(int64_t v, int64_t *total) {
  __shared__ int64_t warp_sums[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  int64_t x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    int64_t y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int64_t w = (lane < nwarps) ? warp_sums[lane] : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      int64_t y = __shfl_up_sync(0xffffffffu, w, d);
      if (lane >= d) w += y;
    }
    if (lane < nwarps) warp_sums[lane] = w;
  }
  __syncthreads();
  const int64_t before = (warp > 0) ? warp_sums[warp - 1] : 0;
  *total = warp_sums[nwarps - 1];
  __syncthreads();
  return before + x - v;
}

__device__ int64_t block_sum(int64_t v) {
  int64_t t;
  block_exclusive_scan(v, &t);
  return t;
}

// ----------------------------------------------------------------------------
// The kept-column bitmap of C block row i over the window [w0, w0+wn):
// bit (j-w0) is set iff some kept product (i,k,j) exists, or (when use_cin)
// C_in holds block (i,j). Warps walk A's row i, lanes walk B's row k.
// With COUNT, also counts candidates, kept products and their 2mnk.
// ----------------------------------------------------------------------------
template <bool COUNT>
__device__ void row_bitmap(const DevMat &A, const DevMat &B, const DevMat &Cin, int use_cin,
                           double eps, int i, int w0, int wn, bool whole, uint32_t *bitmap,
                           int nwords, int64_t &cand, int64_t &kept, int64_t &flops) {
  for (int t = threadIdx.x; t < nwords; t += blockDim.x) bitmap[t] = 0u;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int m = A.row_sizes[i];
  const int p0 = A.row_ptr[i], p1 = A.row_ptr[i + 1];
  const EpsBand band = eps_band(eps);
  for (int p = p0 + warp; p < p1; p += nwarps) {
    const int k = A.col_idx[p];
    const double na = A.norms[p];
    const float fa = A.normsf[p];
    int q0 = B.row_ptr[k], q1 = B.row_ptr[k + 1];
    if (!whole) {
      q0 = lower_bound_i32(B.col_idx, q0, q1, w0);
      q1 = lower_bound_i32(B.col_idx, q0, q1, w0 + wn);
    }
    const int64_t ms = (int64_t)m * B.row_sizes[k];
    for (int q = q0 + lane; q < q1; q += 32) {
      const int j = B.col_idx[q];
      if (COUNT) cand++;
      if (keep_fast(fa, B.normsf[q], na, B.norms[q], eps, band)) {
        const int jj = j - w0;
        atomicOr(&bitmap[jj >> 5], 1u << (jj & 31));
        if (COUNT) {
          kept++;
          flops += 2 * ms * B.col_sizes[j];
        }
      }
    }
  }
  if (use_cin) {
    int c0 = Cin.row_ptr[i], c1 = Cin.row_ptr[i + 1];
    if (!whole) {
      c0 = lower_bound_i32(Cin.col_idx, c0, c1, w0);
      c1 = lower_bound_i32(Cin.col_idx, c0, c1, w0 + wn);
    }
    for (int c = c0 + threadIdx.x; c < c1; c += blockDim.x) {
      const int jj = Cin.col_idx[c] - w0;
      atomicOr(&bitmap[jj >> 5], 1u << (jj & 31));
    }
  }
  __syncthreads();
}

// ----------------------------------------------------------------------------
// Scan: one thread block. Exclusive sums over block rows, totals, capacity check,
// C's header and the sentinel of the product ranges.
// ----------------------------------------------------------------------------
__device__ void symbolic_scan(int32_t nbr, const DevWs &ws, const DevOut &C, DevStatus *st) {
  // rows in tiles of blockDim.x, a row per thread (coalesced loads), the
  // running totals carried from tile to tile
  int64_t tb = 0, tp = 0, tn = 0, sc = 0, sf = 0;
  for (int base = 0; base < nbr; base += blockDim.x) {
    const int r = base + (int)threadIdx.x;
    const bool in = r < nbr;
    const int64_t b = in ? ws.row_cblk[r] : 0, p = in ? ws.row_prod[r] : 0;
    const int64_t n = in ? ws.row_nnz[r] : 0;
    if (in) {
      sc += ws.row_cand[r];
      sf += ws.row_flops[r];
    }
    int64_t sb, sp, sn;
    const int64_t eb = block_exclusive_scan(b, &sb);
    const int64_t ep = block_exclusive_scan(p, &sp);
    const int64_t en = block_exclusive_scan(n, &sn);
    if (in) {
      C.row_ptr[r] = (int32_t)(tb + eb);
      ws.prod_off[r] = tp + ep;
      ws.nnz_off[r] = tn + en;
    }
    tb += sb;
    tp += sp;
    tn += sn;
  }
  const int64_t tc = block_sum(sc);
  const int64_t tf = block_sum(sf);
  if (threadIdx.x == 0) {
    C.row_ptr[nbr] = (int32_t)tb;
    ws.prod_off[nbr] = tp;
    ws.nnz_off[nbr] = tn;
    const int overflow = (tb > C.cap_blk) || (tn > C.cap_nnz) || (tp > ws.cap_prod) ||
                         (tb >= (int64_t)INT32_MAX);
    st->nblk_c = tb;
    st->nnz_c = tn;
    st->nprod = tp;
    st->candidates = tc;
    st->kept = tp;
    st->flops = tf;
    st->overflow = overflow;
    st->error = 0;
    if (!overflow) {
      C.hdr[0] = tb;
      C.hdr[1] = tn;
      ws.prod_ptr[tb] = tp;
    }
  }
}

// ----------------------------------------------------------------------------
// Count pass: one thread block per C block row (grid-stride).
// ----------------------------------------------------------------------------
template <int THREADS>
__global__ void __launch_bounds__(THREADS)
    k_symbolic_count(DevMat A, DevMat B, DevMat Cin, int use_cin, double eps, DevWs ws, DevOut C,
                     DevStatus *st, int32_t *ticket) {
  extern __shared__ uint32_t smem_bits[];
  const int nbc = B.nbc;
  const bool whole = nbc <= kWindowCols;
  for (int i = blockIdx.x; i < A.nbr; i += gridDim.x) {
    int64_t cand = 0, kept = 0, flops = 0, colsum = 0, nblk = 0;
    for (int w0 = 0; w0 < nbc; w0 += kWindowCols) {
      const int wn = min(kWindowCols, nbc - w0);
      const int nwords = (wn + 31) >> 5;
      row_bitmap<true>(A, B, Cin, use_cin, eps, i, w0, wn, whole, smem_bits, nwords, cand, kept,
                       flops);
      for (int t = threadIdx.x; t < nwords; t += blockDim.x) {
        uint32_t bits = smem_bits[t];
        nblk += __popc(bits);
        while (bits) {
          const int b = __ffs(bits) - 1;
          bits &= bits - 1;
          colsum += B.col_sizes[w0 + 32 * t + b];
        }
      }
      __syncthreads();
    }
    cand = block_sum(cand);
    kept = block_sum(kept);
    flops = block_sum(flops);
    colsum = block_sum(colsum);
    nblk = block_sum(nblk);
    if (threadIdx.x == 0) {
      ws.row_cblk[i] = (int32_t)nblk;
      ws.row_prod[i] = kept;
      ws.row_nnz[i] = (int64_t)A.row_sizes[i] * colsum;
      ws.row_cand[i] = cand;
      ws.row_flops[i] = flops;
    }
  }
  if (ticket) {  // the last thread block to get here has every row's counts
    __shared__ int last;
    if (threadIdx.x == 0) {
      __threadfence();
      last = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    symbolic_scan(A.nbr, ws, C, st);
    if (threadIdx.x == 0) *ticket = 0;
  }
}

// Threads of a thread block, which takes a row at a time: a row is a chain of loads for
// every warp, so few rows (up to three per SM) get 16 warps each, more rows 8 and twice the
// thread blocks per SM. Count and fill with digits, 96 rows 78 -> 60 us, 192 rows 113 -> 91,
// 64 rows of 64 blocks of 32 106 -> 85; 32 warps a row 93 and 89 for the last two.
static int sym_threads(int nbr, int nsm) { return nbr <= 3 * nsm ? 512 : 256; }

cudaError_t launch_symbolic_count(DevMat A, DevMat B, DevMat Cin, int use_cin, double eps,
                                  DevWs ws, DevOut C, DevStatus *st, int32_t *ticket, int nsm,
                                  cudaStream_t stream) {
  const int nwords = (min(B.nbc, kWindowCols) + 31) / 32;
  const size_t smem = (size_t)max(nwords, 1) * sizeof(uint32_t);
  const int threads = sym_threads(A.nbr, nsm);
  int grid = nsm * 6;
  if (ticket) grid = min(grid, max(A.nbr, 1));  // fewer to wait for
  if (threads == 512)
    k_symbolic_count<512><<<grid, 512, smem, stream>>>(A, B, Cin, use_cin, eps, ws, C, st, ticket);
  else
    k_symbolic_count<256><<<grid, 256, smem, stream>>>(A, B, Cin, use_cin, eps, ws, C, st, ticket);
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// Scan pass of its own: one thread block of 1024 threads.
// ----------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_symbolic_scan(int32_t nbr, DevWs ws, DevOut C,
                                                        DevStatus *st) {
  symbolic_scan(nbr, ws, C, st);
}

cudaError_t launch_symbolic_scan(int32_t nbr, DevWs ws, DevOut C, DevStatus *st,
                                 cudaStream_t stream) {
  k_symbolic_scan<<<1, 1024, 0, stream>>>(nbr, ws, C, st);
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// Fill pass helpers.
// ----------------------------------------------------------------------------
// wpre[t] = number of set bits in bitmap[0..t); returns the total.
__device__ int word_prefix(const uint32_t *bitmap, int32_t *wpre, int nwords) {
  const int per = (nwords + blockDim.x - 1) / blockDim.x;
  const int beg = min(nwords, (int)threadIdx.x * per), end = min(nwords, beg + per);
  int64_t s = 0;
  for (int t = beg; t < end; t++) s += __popc(bitmap[t]);
  int64_t total;
  int64_t run = block_exclusive_scan(s, &total);
  for (int t = beg; t < end; t++) {
    wpre[t] = (int32_t)run;
    run += __popc(bitmap[t]);
  }
  __syncthreads();
  return (int)total;
}

// Words of the per-row (C block x A block) bit matrix of the fill pass, at
// most (the launch may ask for fewer, for more resident blocks).
constexpr int kMaskWords = 8192;

// Rank of column offset jj inside the window among the set bits.
__device__ __forceinline__ int bit_rank(const uint32_t *bitmap, const int32_t *wpre, int jj) {
  return wpre[jj >> 5] + __popc(bitmap[jj >> 5] & ((1u << (jj & 31)) - 1u));
}

// ----------------------------------------------------------------------------
// Fill pass: one thread block per C block row (grid-stride).
// ----------------------------------------------------------------------------
template <int THREADS>
__global__ void __launch_bounds__(THREADS)
    k_symbolic_fill(DevMat A, DevMat B, DevMat Cin, int use_cin, double eps, DevWs ws, DevOut C,
                    const DevStatus *st, int mask_words, Digits dg) {
  if (st->overflow) return;
  extern __shared__ uint32_t smem_bits[];
  const int nbc = B.nbc;
  const bool whole = nbc <= kWindowCols;
  const int nwords_max = (min(nbc, kWindowCols) + 31) >> 5;
  uint32_t *bitmap = smem_bits;
  int32_t *wpre = reinterpret_cast<int32_t *>(smem_bits + nwords_max);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  int64_t dummy0 = 0, dummy1 = 0, dummy2 = 0;

  uint32_t *mask = smem_bits + 2 * nwords_max;  // mask_words words, see below
  const EpsBand band = eps_band(eps);

  for (int i = blockIdx.x; i < A.nbr; i += gridDim.x) {
    const int g0 = C.row_ptr[i], g1 = C.row_ptr[i + 1];
    if (g0 == g1) continue;
    const int m = A.row_sizes[i];
    const int p0 = A.row_ptr[i], p1 = A.row_ptr[i + 1];

    // Fast path (one column window, small enough row): a bit matrix in shared
    // memory with one bit per (C block of the row, A block of the row) says
    // which kept products exist; a product's place in its C block's list
    // (ascending k) is then the popcount of the bits before it, so every
    // product is placed at once, without a pass per A block.
    const int wps = (p1 - p0 + 31) >> 5;  // mask words per C block
    if (whole && (int64_t)(g1 - g0) * wps <= mask_words) {
      const int nwords = (nbc + 31) >> 5;
      row_bitmap<false>(A, B, Cin, use_cin, eps, i, 0, nbc, true, bitmap, nwords, dummy0, dummy1,
                        dummy2);
      word_prefix(bitmap, wpre, nwords);
      for (int t = threadIdx.x; t < nwords; t += blockDim.x) {
        uint32_t bits = bitmap[t];
        int g = g0 + wpre[t];
        while (bits) {
          const int b = __ffs(bits) - 1;
          bits &= bits - 1;
          C.col_idx[g] = 32 * t + b;
          C.blk_row[g] = i;
          ws.c_cin[g] = -1;
          g++;
        }
      }
      for (int t = threadIdx.x; t < (g1 - g0) * wps; t += blockDim.x) mask[t] = 0u;
      __syncthreads();
      for (int p = p0 + warp; p < p1; p += nwarps) {
        const int k = A.col_idx[p];
        const double na = A.norms[p];
        const float fa = A.normsf[p];
        const uint32_t bit = 1u << ((p - p0) & 31);
        const int wofs = (p - p0) >> 5;
        for (int q = B.row_ptr[k] + lane; q < B.row_ptr[k + 1]; q += 32) {
          if (keep_fast(fa, B.normsf[q], na, B.norms[q], eps, band)) {
            const int sl = bit_rank(bitmap, wpre, B.col_idx[q]);
            atomicOr(&mask[sl * wps + wofs], bit);
          }
        }
      }
      if (use_cin) {
        for (int c = Cin.row_ptr[i] + threadIdx.x; c < Cin.row_ptr[i + 1]; c += blockDim.x)
          ws.c_cin[g0 + bit_rank(bitmap, wpre, Cin.col_idx[c])] = c;
      }
      __syncthreads();
      // product ranges and value offsets of the row's C blocks
      int64_t carry_p = ws.prod_off[i], carry_v = ws.nnz_off[i];
      for (int base = g0; base < g1; base += blockDim.x) {
        const int g = base + threadIdx.x;
        const bool in = g < g1;
        int64_t cp = 0;
        if (in)
          for (int w = 0; w < wps; w++) cp += __popc(mask[(g - g0) * wps + w]);
        const int64_t cv = in ? (int64_t)m * C.col_sizes[C.col_idx[g]] : 0;
        int64_t tp, tv;
        const int64_t ep = block_exclusive_scan(cp, &tp);
        const int64_t ev = block_exclusive_scan(cv, &tv);
        if (in) {
          ws.prod_ptr[g] = carry_p + ep;
          C.blk_off[g] = carry_v + ev;
        }
        carry_p += tp;
        carry_v += tv;
      }
      __syncthreads();
      // every kept product straight to its place
      for (int p = p0 + warp; p < p1; p += nwarps) {
        const int k = A.col_idx[p];
        const double na = A.norms[p];
        const float fa = A.normsf[p];
        const int pi = p - p0;
        const uint32_t below = (1u << (pi & 31)) - 1u;
        for (int q = B.row_ptr[k] + lane; q < B.row_ptr[k + 1]; q += 32) {
          if (keep_fast(fa, B.normsf[q], na, B.norms[q], eps, band)) {
            const int sl = bit_rank(bitmap, wpre, B.col_idx[q]);
            const uint32_t *mk = mask + sl * wps;
            int pos = __popc(mk[pi >> 5] & below);
            for (int w = 0; w < (pi >> 5); w++) pos += __popc(mk[w]);
            ws.prods[ws.prod_ptr[g0 + sl] + pos] = make_int2(p, q);
          }
        }
      }
      __syncthreads();
      continue;
    }

    // pass 1: C blocks of the row, per-block product counts, C_in map
    int slot_base = 0;
    for (int w0 = 0; w0 < nbc; w0 += kWindowCols) {
      const int wn = min(kWindowCols, nbc - w0);
      const int nwords = (wn + 31) >> 5;
      row_bitmap<false>(A, B, Cin, use_cin, eps, i, w0, wn, whole, bitmap, nwords, dummy0, dummy1,
                        dummy2);
      const int nw = word_prefix(bitmap, wpre, nwords);
      for (int t = threadIdx.x; t < nwords; t += blockDim.x) {
        uint32_t bits = bitmap[t];
        int g = g0 + slot_base + wpre[t];
        while (bits) {
          const int b = __ffs(bits) - 1;
          bits &= bits - 1;
          C.col_idx[g] = w0 + 32 * t + b;
          C.blk_row[g] = i;
          ws.cnt[g] = 0;
          ws.c_cin[g] = -1;
          g++;
        }
      }
      __syncthreads();
      for (int p = p0 + warp; p < p1; p += nwarps) {
        const int k = A.col_idx[p];
        const double na = A.norms[p];
        const float fa = A.normsf[p];
        int q0 = B.row_ptr[k], q1 = B.row_ptr[k + 1];
        if (!whole) {
          q0 = lower_bound_i32(B.col_idx, q0, q1, w0);
          q1 = lower_bound_i32(B.col_idx, q0, q1, w0 + wn);
        }
        for (int q = q0 + lane; q < q1; q += 32) {
          if (keep_fast(fa, B.normsf[q], na, B.norms[q], eps, band)) {
            const int g = g0 + slot_base + bit_rank(bitmap, wpre, B.col_idx[q] - w0);
            atomicAdd(&ws.cnt[g], 1);
          }
        }
      }
      if (use_cin) {
        int c0 = Cin.row_ptr[i], c1 = Cin.row_ptr[i + 1];
        if (!whole) {
          c0 = lower_bound_i32(Cin.col_idx, c0, c1, w0);
          c1 = lower_bound_i32(Cin.col_idx, c0, c1, w0 + wn);
        }
        for (int c = c0 + threadIdx.x; c < c1; c += blockDim.x) {
          const int g = g0 + slot_base + bit_rank(bitmap, wpre, Cin.col_idx[c] - w0);
          ws.c_cin[g] = c;
        }
      }
      __syncthreads();
      slot_base += nw;
    }

    // pass 2: product ranges and value offsets of the row's C blocks
    {
      int64_t carry_p = ws.prod_off[i], carry_v = ws.nnz_off[i];
      for (int base = g0; base < g1; base += blockDim.x) {
        const int g = base + threadIdx.x;
        const bool in = g < g1;
        const int64_t cp = in ? ws.cnt[g] : 0;
        const int64_t cv = in ? (int64_t)m * C.col_sizes[C.col_idx[g]] : 0;
        int64_t tp, tv;
        const int64_t ep = block_exclusive_scan(cp, &tp);
        const int64_t ev = block_exclusive_scan(cv, &tv);
        if (in) {
          ws.prod_ptr[g] = carry_p + ep;
          C.blk_off[g] = carry_v + ev;
          ws.cnt[g] = 0;
        }
        carry_p += tp;
        carry_v += tv;
      }
      __syncthreads();
    }

    // pass 3: kept products grouped by C block, ascending k inside a block
    slot_base = 0;
    for (int w0 = 0; w0 < nbc; w0 += kWindowCols) {
      const int wn = min(kWindowCols, nbc - w0);
      const int nwords = (wn + 31) >> 5;
      int nw;
      if (!whole) {
        row_bitmap<false>(A, B, Cin, use_cin, eps, i, w0, wn, whole, bitmap, nwords, dummy0,
                          dummy1, dummy2);
        nw = word_prefix(bitmap, wpre, nwords);
      } else {
        nw = g1 - g0;
      }
      for (int p = p0; p < p1; p++) {
        const int k = A.col_idx[p];
        const double na = A.norms[p];
        const float fa = A.normsf[p];
        int q0 = B.row_ptr[k], q1 = B.row_ptr[k + 1];
        if (!whole) {
          q0 = lower_bound_i32(B.col_idx, q0, q1, w0);
          q1 = lower_bound_i32(B.col_idx, q0, q1, w0 + wn);
        }
        for (int q = q0 + threadIdx.x; q < q1; q += blockDim.x) {
          if (keep_fast(fa, B.normsf[q], na, B.norms[q], eps, band)) {
            const int g = g0 + slot_base + bit_rank(bitmap, wpre, B.col_idx[q] - w0);
            const int c = ws.cnt[g];
            ws.cnt[g] = c + 1;
            ws.prods[ws.prod_ptr[g] + c] = make_int2(p, q);
          }
        }
        __syncthreads();
      }
      slot_base += nw;
    }
  }

  // the operands' digits, where the numeric phase takes them: bandwidth-bound
  // work that fits between the latency-bound rows of other thread blocks
  if (dg.a.units) {
    __syncthreads();
    int32_t *seg = reinterpret_cast<int32_t *>(smem_bits) + warp * 2 * kDigitMaxRows;
    const bool same = A.vals == B.vals;
    // few rows: from the last thread block on, which has none, and one block of each, so
    // that few blocks are on as many SMs; else consecutive blocks in a thread block
    const int64_t w0 = THREADS == 512 ? (int64_t)warp * gridDim.x + (gridDim.x - 1 - blockIdx.x)
                                      : (int64_t)blockIdx.x * nwarps + warp;
    const int64_t nw = (int64_t)gridDim.x * nwarps;
    digits_of(A, &dg.a, same ? &dg.b : nullptr, seg, w0, nw, lane);
    if (!same) digits_of(B, nullptr, &dg.b, seg, w0, nw, lane);
  }
}

cudaError_t launch_symbolic_fill(DevMat A, DevMat B, DevMat Cin, int use_cin, double eps,
                                 DevWs ws, DevOut C, const DevStatus *st, int nsm, int mask_words,
                                 const Digits *digits, cudaStream_t stream) {
  const int nwords = (min(B.nbc, kWindowCols) + 31) / 32;
  const int mw = (mask_words > 0 && mask_words < kMaskWords) ? mask_words : kMaskWords;
  size_t smem = ((size_t)max(nwords, 1) * 2 + mw) * sizeof(uint32_t);
  const int threads = sym_threads(A.nbr, nsm);
  if (digits) smem = max(smem, sizeof(int32_t) * 2 * kDigitMaxRows * (threads / 32));
  // one wave of resident blocks (rows taken in a grid stride): more resident
  // blocks hide more of each row's load latency, a second wave only adds a tail
  int per_sm = 0;
  const auto fill = threads == 512 ? k_symbolic_fill<512> : k_symbolic_fill<256>;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fill, threads, smem);
  if (e != cudaSuccess) return e;
  const int grid = nsm * (per_sm > 0 ? per_sm : 1);
  fill<<<grid, threads, smem, stream>>>(A, B, Cin, use_cin, eps, ws, C, st, mw,
                                        digits ? *digits : Digits{});
  return cudaGetLastError();
}

}  // namespace bsm
