// Numeric pass: columns (ascending) and values of every row of C, per path
// of the row bins; templated on the value type and on the semiring (Sec. 2.2's
// sum and product, or min-plus, max-plus, or-and: those skip the rank path,
// register sorts above 128 products and the non-default window sizes).
#pragma once

#include <cstddef>

#include "launch_util.cuh"
#include "numband.cuh"
#include "numblock.cuh"
#include "numonce.cuh"
#include "numrank.cuh"
#include "numwarp.cuh"
#include "rowhash.cuh"
#include "rowlane.cuh"
#include "rowpass.cuh"

namespace sg {

constexpr int NUM_WARPS_CTA = 4;  // warps per block on the window path
// k_num_warp1's warps per block: 9 warps of 1024-column FP64 windows
// (74.9 KB) let 3 blocks, 27 warps, share an SM's 228 KB of shared memory
// (4-warp blocks fit 24); wider windows take fewer warps per block.
template <int W>
constexpr int num_warps_cta1() {
  return W <= 1024 ? 9 : (W <= 2048 ? 4 : 2);
}

static long long rows_in(const int* path_rows, int p) { return path_rows ? path_rows[p] : -1; }

template <typename T, int G, int E, int SR>
static cudaError_t tiny_num(const LaunchCtx& c, const Csr& A, const Csr& B, const T* av, const T* bv,
                            const RowInfo& ri, int lo, int hi, const int32_t* c_rp, int32_t* c_ci, T* c_v,
                            long long rows) {
  auto k = k_tiny<G, E, true, T, SR>;
  const int occ = kernel_blocks_per_sm(k, 256, 0);
  const int grid = persistent_grid(rows, 8 * (32 / G), c.nsm, occ);
  k<<<grid, 256, 0, c.stream>>>(A, B, av, bv, ri, c.st, lo, hi, nullptr, c_rp, c_ci, c_v, c.err);
  count_launch(c);
  return cudaGetLastError();
}

// Whether bins lo..hi hold no row (hist: rows per bin on the host, as the
// symbolic pass read them; null: unknown, never empty).
static bool empty_bins(const int* hist, int lo, int hi) {
  if (!hist) return false;
  for (int b = lo; b <= hi; ++b)
    if (hist[b]) return false;
  return true;
}

// Small rows in one launch, each warp taking its share of every kind: a warp
// and its table for 17 to 128 products, register sorts below.  (Five launches
// of kernels that each fill a few SMs, one after the other, cost a product of
// 12,345 vertices 31 us of 570.)
constexpr int SMALL_WARPS = 4;

struct SmallBins {  // inclusive; lo > hi: none
  int tiny_lo, tiny_hi;  // at most bin 5
  int hash_lo, hash_hi;  // bins 6..8
};

template <typename T, int SR>
__global__ void __launch_bounds__(SMALL_WARPS * 32)
k_num_small(Csr A, Csr B, const T* __restrict__ av, const T* __restrict__ bv, RowInfo ri, const DevStats* st,
            SmallBins b, const int32_t* __restrict__ c_rp, int32_t* __restrict__ c_ci, T* __restrict__ c_v,
            uint32_t* err) {
  __shared__ __align__(16) HashWarp<T> s_hash[SMALL_WARPS];
  __shared__ int s_r[5][2];
  const int warp = threadIdx.x >> 5, lane = lane_id();
  auto range = [&](int i, int lo, int hi) { block_bin_range(st, lo, hi, &s_r[i][0], &s_r[i][1]); };
  range(0, max(b.hash_lo, 8), min(b.hash_hi, 8));
  range(1, max(b.hash_lo, 7), min(b.hash_hi, 7));
  range(2, max(b.hash_lo, 6), min(b.hash_hi, 6));
  range(3, max(b.tiny_lo, 5), min(b.tiny_hi, 5));
  range(4, b.tiny_lo, min(b.tiny_hi, 4));
  HashWarp<T>& sm = s_hash[warp];
  if (b.hash_hi >= b.hash_lo)
    for (int t = lane; t < 256; t += 32) sm.key[t] = HASH_EMPTY;
  if (block_skip(st)) return;
  const long long w = (long long)blockIdx.x * SMALL_WARPS + warp, nw = (long long)gridDim.x * SMALL_WARPS;
  hash_num_rows<4, T, SR>(A, B, av, bv, ri, s_r[0][0], s_r[0][1], w, nw, sm, c_rp, c_ci, c_v, err);
  hash_num_rows<2, T, SR>(A, B, av, bv, ri, s_r[1][0], s_r[1][1], w, nw, sm, c_rp, c_ci, c_v, err);
  hash_num_rows<1, T, SR>(A, B, av, bv, ri, s_r[2][0], s_r[2][1], w, nw, sm, c_rp, c_ci, c_v, err);
  tiny_rows<16, 1, true, T, SR>(A, B, av, bv, ri, s_r[3][0], s_r[3][1], w, nw, nullptr, c_rp, c_ci, c_v, err);
  tiny_rows<8, 1, true, T, SR>(A, B, av, bv, ri, s_r[4][0], s_r[4][1], w, nw, nullptr, c_rp, c_ci, c_v, err);
}

template <typename T, int SR>
static cudaError_t small_num(const LaunchCtx& c, const Csr& A, const Csr& B, const T* av, const T* bv,
                             const RowInfo& ri, const SmallBins& b, const int32_t* c_rp, int32_t* c_ci, T* c_v,
                             const int* hist) {
  long long warps = 0;  // hash rows take a warp each, the others a part of one
  for (int k = b.hash_lo; hist && k <= b.hash_hi; ++k) warps += hist[k];
  for (int k = b.tiny_lo; hist && k <= b.tiny_hi; ++k) warps += (hist[k] + 1) / 2;
  if (hist && warps == 0) return cudaSuccess;
  auto k = k_num_small<T, SR>;
  const int occ = kernel_blocks_per_sm(k, SMALL_WARPS * 32, 0);
  if (occ <= 0) return cudaErrorInvalidConfiguration;
  k<<<persistent_grid(hist ? warps : -1, SMALL_WARPS, c.nsm, occ), SMALL_WARPS * 32, 0, c.stream>>>(
      A, B, av, bv, ri, c.st, b, c_rp, c_ci, c_v, c.err);
  count_launch(c);
  return cudaGetLastError();
}

template <typename T, int NT, int SR>
static cudaError_t once_num(const LaunchCtx& c, const Csr& A, const Csr& B, const T* av, const T* bv,
                            const RowInfo& ri, int lo, int hi, const int32_t* c_rp, int32_t* c_ci, T* c_v,
                            const int* hist) {
  auto k = k_num_once<NT, T, SR>;
  int wlog = 10;  // the narrowest bitmap that holds a row of B, up to the widest
  while (wlog < once_wlog_max<NT>() && (1ll << wlog) < B.ncols) ++wlog;
  const size_t smem = once_smem_bytes<NT, T>(wlog);
  const int occ = kernel_blocks_per_sm(k, NT, smem);
  if (occ <= 0) return cudaErrorInvalidConfiguration;
  long long rows = hist ? 0 : -1;
  for (int b = lo; hist && b <= hi; ++b) rows += hist[b];
  const int grid = persistent_grid(rows, 1, c.nsm, occ);
  k<<<grid, NT, smem, c.stream>>>(A, B, av, bv, ri, c.st, lo, hi, wlog, c_rp, c_ci, c_v, c.err);
  count_launch(c);
  return cudaGetLastError();
}

// Bins lo..hi (at most 8192 products) by the threads whose registers hold a
// row: 64 threads up to 512 products, then twice the threads per bin.
template <typename T, int SR>
static cudaError_t once_dispatch(const LaunchCtx& c, const Csr& A, const Csr& B, const T* av, const T* bv,
                                 const RowInfo& ri, int lo, int hi, const int32_t* c_rp, int32_t* c_ci, T* c_v,
                                 const int* hist) {
  cudaError_t e = cudaSuccess;
  auto clip = [&](int a, int b, auto f) {
    const int l = lo > a ? lo : a, h = hi < b ? hi : b;
    if (e == cudaSuccess && l <= h && !empty_bins(hist, l, h)) e = f(c, A, B, av, bv, ri, l, h, c_rp, c_ci, c_v, hist);
  };
  clip(14, 14, once_num<T, 1024, SR>);  // longest rows first
  clip(13, 13, once_num<T, 512, SR>);
  clip(12, 12, once_num<T, 256, SR>);
  clip(11, 11, once_num<T, 128, SR>);
  clip(1, 10, once_num<T, 64, SR>);
  return e;
}

template <typename T, int W, int SR>
static cudaError_t warp_num(const LaunchCtx& c, const Csr& A, const Csr& B, const T* av, const T* bv,
                            const RowInfo& ri, int lo, int hi, const SplitInfo& sp, int32_t* cur, int32_t* nxt,
                            const int32_t* c_rp, int32_t* c_ci, T* c_v, long long rows_wide) {
  auto k = k_num_warp<W, NUM_WARPS_CTA, T, SR>;
  const size_t smem = (size_t)NUM_WARPS_CTA * ((size_t)W * sizeof(T) + W / 8);
  const int occ = kernel_blocks_per_sm(k, NUM_WARPS_CTA * 32, smem);
  if (occ <= 0) return cudaErrorInvalidConfiguration;
  NumSplit ns;
  ns.heavy_bin = sp.heavy_bin;
  ns.hi_bin = sp.hi_bin;
  ns.hcap = sp.hcap;
  ns.ntf = sp.ntf;
  ns.rr = sp.rr;
  ns.runs = sp.runs;
  ns.hcnt = sp.hcnt;
  ns.counter = &c.st->work[0];
  // rows of at most 32 nonzeros first (one cursor per lane, next window's
  // loads overlapped with this window's emission), then the others
  constexpr int NW1 = num_warps_cta1<W>();
  auto k1 = k_num_warp1<W, NW1, T, SR>;
  const size_t smem1 = (size_t)NW1 * ((size_t)W * sizeof(T) + W / 8);
  const int occ1 = kernel_blocks_per_sm(k1, NW1 * 32, smem1);
  if (occ1 <= 0) return cudaErrorInvalidConfiguration;
  unsigned* counter1 = &c.st->work[3];
  // the general kernel has work only for split rows and rows of more than
  // 32 nonzeros (a stencil or Galerkin product has neither)
  const bool general = rows_wide != 0 || (sp.heavy_bin < NBINS && sp.hcap > 0);
  cudaError_t e = cudaMemsetAsync(counter1, 0, sizeof(unsigned), c.stream);
  if (e == cudaSuccess && general) e = cudaMemsetAsync(ns.counter, 0, sizeof(unsigned), c.stream);
  if (e != cudaSuccess) return e;
  k1<<<c.nsm * occ1, NW1 * 32, smem1, c.stream>>>(A, B, av, bv, ri, c.st, lo, hi, ns, c_rp, c_ci, c_v,
                                                           counter1, c.err);
  count_launch(c);
  if ((e = cudaGetLastError()) != cudaSuccess || !general) return e;
  const int grid = c.nsm * occ;
  k<<<grid, NUM_WARPS_CTA * 32, smem, c.stream>>>(A, B, av, bv, ri, c.st, lo, hi, ns, cur, nxt, c_rp, c_ci, c_v,
                                                  c.err, 1);
  count_launch(c);
  return cudaGetLastError();
}

template <typename T, int W, int NUM_BLOCK_WARPS, int SR>
static cudaError_t block_num(const LaunchCtx& c, const Csr& A, const Csr& B, const T* av, const T* bv,
                             const RowInfo& ri, int lo, int hi, const SplitInfo& sp, int32_t* cur, int32_t* nxt,
                             const int32_t* c_rp, int32_t* c_ci, T* c_v) {
  auto k = k_num_block<W, NUM_BLOCK_WARPS, T, SR>;
  const size_t smem = numblock_smem_bytes<W, NUM_BLOCK_WARPS, T>();
  const int occ = kernel_blocks_per_sm(k, NUM_BLOCK_WARPS * 32, smem);
  if (occ <= 0) return cudaErrorInvalidConfiguration;
  unsigned* counter = &c.st->work[1];
  cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned), c.stream);
  if (e != cudaSuccess) return e;
  if (!sp.rrb || !sp.runsb || (1 << sp.wb_shift) != W) return cudaErrorInvalidValue;  // block-granular runs
  k<<<c.nsm * occ, NUM_BLOCK_WARPS * 32, smem, c.stream>>>(A, B, av, bv, ri, c.st, lo, hi, sp.rrb, sp.runsb, cur,
                                                          c_rp, c_ci, c_v, counter, c.err);
  count_launch(c);
  return cudaGetLastError();
}

template <typename T, int SR>
static cudaError_t band_num(const LaunchCtx& c, const Csr& A, const Csr& B, const T* av, const T* bv,
                            const RowInfo& ri, int lo, int hi, int32_t* cur, int32_t* nxt, const int32_t* c_rp,
                            int32_t* c_ci, T* c_v) {
  auto k = k_num_band<T, SR>;
  int wlog = 10;  // the narrowest bitmap that holds a row of B, up to the widest
  while (wlog < BAND_WLOG && (1ll << wlog) < B.ncols) ++wlog;
  const size_t smem = band_smem_bytes<T>(wlog);
  const int occ = kernel_blocks_per_sm(k, BAND_THREADS, smem);
  if (occ <= 0) return cudaErrorInvalidConfiguration;
  unsigned* counter = &c.st->work[1];
  cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned), c.stream);
  if (e != cudaSuccess) return e;
  k<<<c.nsm * occ, BAND_THREADS, smem, c.stream>>>(A, B, av, bv, ri, c.st, lo, hi, wlog, cur, nxt, c_rp, c_ci, c_v,
                                                   counter, c.err);
  count_launch(c);
  return cudaGetLastError();
}

// Rank-compacted accumulator: 8 warps per block; values either reduced into
// C in global memory (the default, 56 KB of shared memory per block, four
// blocks per SM) or summed in shared memory 6144 ranks at a time (104 KB in
// FP64, two blocks per SM).
constexpr int RANK_WARPS = 8;
constexpr int RANK_CAP = 6144;

template <typename T, int CAP>
static cudaError_t rank_num(const LaunchCtx& c, const Csr& A, const Csr& B, const T* av, const T* bv,
                            const RowInfo& ri, int lo, int hi, const int32_t* c_rp, int32_t* c_ci, T* c_v) {
  auto k = k_num_rank<RANK_WARPS, CAP, T>;
  const size_t smem = numrank_smem_bytes<RANK_WARPS, CAP, T>();
  const int occ = kernel_blocks_per_sm(k, RANK_WARPS * 32, smem);
  if (occ <= 0) return cudaErrorInvalidConfiguration;
  unsigned* counter = &c.st->work[2];
  cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned), c.stream);
  if (e != cudaSuccess) return e;
  k<<<c.nsm * occ, RANK_WARPS * 32, smem, c.stream>>>(A, B, av, bv, ri, c.st, lo, hi, c_rp, c_ci, c_v, counter,
                                                      c.err);
  count_launch(c);
  return cudaGetLastError();
}

// The rank-compacted path and register sorts of more than 128 products
// exist for the ordinary sum and product only; other semirings never route
// rows to them.
template <typename T, int G, int E, int SR>
static cudaError_t tiny_num_wide(const LaunchCtx& c, const Csr& A, const Csr& B, const T* av, const T* bv,
                                 const RowInfo& ri, int lo, int hi, const int32_t* c_rp, int32_t* c_ci, T* c_v,
                                 long long rows) {
  if constexpr (SR == SPGEMM_PLUS_TIMES) return tiny_num<T, G, E, SR>(c, A, B, av, bv, ri, lo, hi, c_rp, c_ci, c_v, rows);
  else return cudaErrorInvalidValue;
}
template <typename T, int CAP, int SR>
static cudaError_t rank_num_plus(const LaunchCtx& c, const Csr& A, const Csr& B, const T* av, const T* bv,
                                 const RowInfo& ri, int lo, int hi, const int32_t* c_rp, int32_t* c_ci, T* c_v) {
  if constexpr (SR == SPGEMM_PLUS_TIMES) return rank_num<T, CAP>(c, A, B, av, bv, ri, lo, hi, c_rp, c_ci, c_v);
  else return cudaErrorInvalidValue;
}

template <typename F8, typename F16, typename F32, typename F64, typename F128, typename F256, typename F512>
static cudaError_t tiny_dispatch(const int* hist, int lo, int hi, F8 f8, F16 f16, F32 f32, F64 f64, F128 f128,
                                 F256 f256, F512 f512) {
  cudaError_t e = cudaSuccess;
  auto clip = [&](int a, int b, auto f) -> cudaError_t {
    const int l = lo > a ? lo : a, h = hi < b ? hi : b;
    return (l <= h && !empty_bins(hist, l, h)) ? f(l, h) : cudaSuccess;
  };
  if ((e = clip(1, 4, f8))) return e;
  if ((e = clip(5, 5, f16))) return e;
  if ((e = clip(6, 6, f32))) return e;
  if ((e = clip(7, 7, f64))) return e;
  if ((e = clip(8, 8, f128))) return e;
  if ((e = clip(9, 9, f256))) return e;
  if ((e = clip(10, 10, f512))) return e;
  return cudaSuccess;
}

// With the banded accumulator as the default, the block window takes over (on
// narrow FP32 products, see numeric_block_bin) when fewer than 40 rows per SM
// are in its bins: the longest row then sets the time, and two dense windows
// with adds that need no compare-and-swap finish it sooner than bands do
// (12,345 columns: 0.22 ms against 0.26; 20,000 columns and 2 M nonzeros:
// 3.5 against 3.3).
static int block_lo(const Tuning& tu, const int* hist, int nsm) {
  if (tu.num_lo_band >= NBINS || tu.num_lo_block >= NBINS) return tu.num_lo_block;
  long long rows = 0;
  for (int b = tu.num_lo_block; hist && b < NBINS; ++b) rows += hist[b];
  return hist && rows < 40ll * nsm ? tu.num_lo_block : NBINS;
}

template <typename T, int SR>
static cudaError_t numeric_t(const LaunchCtx& c, const Csr& A, const Csr& B, const RowInfo& ri,
                             const PathBins& pb, const Tuning& tu, const SplitInfo& sp, const T* av,
                             const T* bv, int32_t* cur, int32_t* nxt, const int32_t* c_rp, int32_t* c_ci,
                             T* c_v, const int* path_rows, long long rows_wide, long long rows_wide8, const int* hist) {
  cudaError_t e = cudaSuccess;
  if (pb.hi[PATH_HASH] >= pb.lo[PATH_HASH]) {  // with it, register sorts stop at 16 products
    timer_mark(c, T_NUM_HASH, 0);
    SmallBins b{pb.lo[PATH_TINY], pb.hi[PATH_TINY], pb.lo[PATH_HASH], pb.hi[PATH_HASH]};
    // Rows of up to 64 products by one lane each when they are most of the
    // product's rows and enough to give every SM several warps (stencil and
    // Galerkin products): throughput over many similar rows.  When no row has
    // more than LANE_MERGE_K nonzeros (they are merged), the smallest ones
    // too: the register sort exchanges every product of a row with its
    // neighbours log2(P)^2 / 2 times (96^3 Galerkin, A*P with 7 products a
    // row: 107 us).  Fewer rows keep a warp each, whose latency per row is
    // lower.
    long long all_rows = 0, lane_rows_n = 0;
    const bool merge = rows_wide8 == 0 && b.tiny_hi + 1 == b.hash_lo;
    if (path_rows && hist) {
      for (int q = 0; q < NPATHS; ++q) all_rows += path_rows[q];
      for (int k = merge ? b.tiny_lo : b.hash_lo; k <= b.hash_hi && k <= 7; ++k) lane_rows_n += hist[k];
    }
    if (lane_rows_n >= lane_rows_from(rows_wide8, c.nsm) && (merge || 2 * (long long)path_rows[PATH_HASH] >= all_rows)) {
      const int llo = merge ? b.tiny_lo : b.hash_lo, lhi = b.hash_hi < 7 ? b.hash_hi : 7;
      e = lane_rows<T, SR>(c, A, B, av, bv, ri, llo, lhi, c_rp, c_ci, c_v, lane_rows_n, rows_wide8);
      b.hash_lo = lhi + 1;
      if (merge) b.tiny_hi = b.tiny_lo - 1;
    }
    if (!e) e = small_num<T, SR>(c, A, B, av, bv, ri, b, c_rp, c_ci, c_v, hist);
    timer_mark(c, T_NUM_HASH, 1);
    if (e) return e;
  } else if (pb.hi[PATH_TINY] >= pb.lo[PATH_TINY]) {
    const long long rows = rows_in(path_rows, PATH_TINY);
    timer_mark(c, T_NUM_TINY, 0);
    e = tiny_dispatch(hist, pb.lo[PATH_TINY], pb.hi[PATH_TINY],
        [&](int l, int h) { return tiny_num<T, 8, 1, SR>(c, A, B, av, bv, ri, l, h, c_rp, c_ci, c_v, rows); },
        [&](int l, int h) { return tiny_num<T, 16, 1, SR>(c, A, B, av, bv, ri, l, h, c_rp, c_ci, c_v, rows); },
        [&](int l, int h) { return tiny_num<T, 32, 1, SR>(c, A, B, av, bv, ri, l, h, c_rp, c_ci, c_v, rows); },
        [&](int l, int h) { return tiny_num<T, 32, 2, SR>(c, A, B, av, bv, ri, l, h, c_rp, c_ci, c_v, rows); },
        [&](int l, int h) { return tiny_num<T, 32, 4, SR>(c, A, B, av, bv, ri, l, h, c_rp, c_ci, c_v, rows); },
        [&](int l, int h) { return tiny_num_wide<T, 32, 8, SR>(c, A, B, av, bv, ri, l, h, c_rp, c_ci, c_v, rows); },
        [&](int l, int h) { return tiny_num_wide<T, 32, 16, SR>(c, A, B, av, bv, ri, l, h, c_rp, c_ci, c_v, rows); });
    timer_mark(c, T_NUM_TINY, 1);
    if (e) return e;
  }
  // every other row (rows of the symbolic warp and block paths both land
  // here): the warp-owned dense window for all but the longest when most are
  // dense (tu.windows); the block-wide window from block_lo on, the banded accumulator from
  // num_lo_band on, below them the register path and, where an option asks
  // for it, the warp-owned dense window
  int lo = NBINS, hi = 0;
  for (int p : {PATH_WARP, PATH_BLOCK})
    if (pb.hi[p] >= pb.lo[p]) {
      lo = pb.lo[p] < lo ? pb.lo[p] : lo;
      hi = pb.hi[p] > hi ? pb.hi[p] : hi;
    }
  if (tu.windows && hi >= lo) {
    const int whi = hi < bin_of(65536) ? hi : bin_of(65536);
    if (whi >= lo && !empty_bins(hist, lo, whi)) {
      timer_mark(c, T_NUM_WARP, 0);
      e = warp_num<T, 1024, SR>(c, A, B, av, bv, ri, lo, whi, sp, cur, nxt, c_rp, c_ci, c_v, rows_wide);
      timer_mark(c, T_NUM_WARP, 1);
      if (e) return e;
    }
    if (whi >= lo) lo = whi + 1;
  }
  const int nlo = block_lo(tu, hist, c.nsm);
  const int blo = nlo > lo ? nlo : lo;
  if (hi >= blo && !empty_bins(hist, blo, hi)) {
    timer_mark(c, T_NUM_BLOCK, 0);
#define SG_BLOCK_NUM(WW, NWW) e = block_num<T, WW, NWW, SR>(c, A, B, av, bv, ri, blo, hi, sp, cur, nxt, c_rp, c_ci, c_v)
    // supported geometries (window columns, warps); others fall back to 8192 x 8
    const int wbk = tu.window_block, nwk = tu.block_warps;
    if (wbk == 16384 && nwk == 16) SG_BLOCK_NUM(16384, 16);
    else if (SR != SPGEMM_PLUS_TIMES) SG_BLOCK_NUM(8192, 8);
    else if (wbk == 2048 && nwk == 4) SG_BLOCK_NUM(2048, 4);
    else if (wbk == 2048 && nwk == 8) SG_BLOCK_NUM(2048, 8);
    else if (wbk == 4096 && nwk == 4) SG_BLOCK_NUM(4096, 4);
    else if (wbk == 4096 && nwk == 8) SG_BLOCK_NUM(4096, 8);
    else if (wbk == 4096 && nwk == 16) SG_BLOCK_NUM(4096, 16);
    else if (wbk == 8192 && nwk == 16) SG_BLOCK_NUM(8192, 16);
    else SG_BLOCK_NUM(8192, 8);
#undef SG_BLOCK_NUM
    timer_mark(c, T_NUM_BLOCK, 1);
    if (e) return e;
  }
  if (hi >= blo) hi = blo - 1;
  // with many rows of 2,049 to 4,096 products the register path keeps them
  // (64 products of 1,024 to 50,000 rows: 0.55 ms, 0.83 in bands)
  int band = tu.num_lo_band > lo ? tu.num_lo_band : lo;
  if (hist && band == bin_of(2048) + 1 && hist[band] >= 40 * c.nsm) ++band;
  if (blo >= NBINS && hi >= band) {
    if (!empty_bins(hist, band, hi)) {
      timer_mark(c, T_NUM_BLOCK, 0);
      e = band_num<T, SR>(c, A, B, av, bv, ri, band, hi, cur, nxt, c_rp, c_ci, c_v);
      timer_mark(c, T_NUM_BLOCK, 1);
      if (e) return e;
    }
    hi = band - 1;
  }
  // rows of the rank bins (below the block window) take the rank-compacted
  // accumulator, unless heavy rows are split (the warp kernel owns those)
  const bool split = sp.heavy_bin < NBINS && sp.hcap > 0;
  const int rlo = tu.num_lo_rank > lo ? tu.num_lo_rank : lo;
  if (SR == SPGEMM_PLUS_TIMES && !split && hi >= rlo) {
    if (!empty_bins(hist, rlo, hi)) {
      timer_mark(c, T_NUM_RANK, 0);
      e = tu.rank_accum == 1 ? rank_num_plus<T, RANK_CAP, SR>(c, A, B, av, bv, ri, rlo, hi, c_rp, c_ci, c_v)
                             : rank_num_plus<T, 0, SR>(c, A, B, av, bv, ri, rlo, hi, c_rp, c_ci, c_v);
      timer_mark(c, T_NUM_RANK, 1);
      if (e) return e;
    }
    hi = rlo - 1;
  }
  if (hi >= lo && !empty_bins(hist, lo, hi)) {
    timer_mark(c, T_NUM_WARP, 0);
    if (tu.num_hi_once >= lo) {  // rows whose products fit a block's registers
      const int ohi = hi < tu.num_hi_once ? hi : tu.num_hi_once;
      e = once_dispatch<T, SR>(c, A, B, av, bv, ri, lo, ohi, c_rp, c_ci, c_v, hist);
      lo = ohi + 1;
    }
    if (!e && hi >= lo && !empty_bins(hist, lo, hi))
      switch (SR == SPGEMM_PLUS_TIMES ? tu.window_warp : 1024) {
        case 2048: e = warp_num<T, 2048, SR>(c, A, B, av, bv, ri, lo, hi, sp, cur, nxt, c_rp, c_ci, c_v, rows_wide); break;
        case 4096: e = warp_num<T, 4096, SR>(c, A, B, av, bv, ri, lo, hi, sp, cur, nxt, c_rp, c_ci, c_v, rows_wide); break;
        default: e = warp_num<T, 1024, SR>(c, A, B, av, bv, ri, lo, hi, sp, cur, nxt, c_rp, c_ci, c_v, rows_wide); break;
      }
    timer_mark(c, T_NUM_WARP, 1);
    if (e) return e;
  }
  return cudaSuccess;
}


// Entry of the numeric pass for one semiring, both value types.
template <int SR>
static cudaError_t launch_numeric_sr(const LaunchCtx& c, const Csr& A, const Csr& B, const RowInfo& ri,
                                     const PathBins& pb, const Tuning& tu, const SplitInfo& sp, int dtype,
                                     const void* av, const void* bv, int32_t* cur, int32_t* nxt,
                                     const int32_t* c_rp, int32_t* c_ci, void* c_v, const int* path_rows,
                                     long long rows_wide, long long rows_wide8, const int* hist) {
  if (dtype == SPGEMM_F32)
    return numeric_t<float, SR>(c, A, B, ri, pb, tu, sp, (const float*)av, (const float*)bv, cur, nxt, c_rp, c_ci,
                                (float*)c_v, path_rows, rows_wide, rows_wide8, hist);
  return numeric_t<double, SR>(c, A, B, ri, pb, tu, sp, (const double*)av, (const double*)bv, cur, nxt, c_rp, c_ci,
                               (double*)c_v, path_rows, rows_wide, rows_wide8, hist);
}

}  // namespace sg
