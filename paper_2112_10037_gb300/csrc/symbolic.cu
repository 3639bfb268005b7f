// Symbolic pass: the number of distinct columns of every row of C
// (Sec. 2.2: the union of the columns of the B rows a row of A touches).
#include "launch_util.cuh"
#include "rowhash.cuh"
#include "rowlane.cuh"
#include "rowpass.cuh"
#include "symblock.cuh"

namespace sg {

// Symbolic windows hold only a presence bitmap, so they are wide.
constexpr int SYM_WARP_W = 32768;    // 4 KB of bits per warp
constexpr int SYM_BLOCK_W = 262144;  // 32 KB of bits per block
constexpr int SYM_BLOCK_WARPS = 8;

template <int G, int E>
static cudaError_t tiny_sym(const LaunchCtx& c, const Csr& A, const Csr& B, const RowInfo& ri, int lo, int hi,
                            int32_t* c_cnt, long long rows) {
  const double* nv = nullptr;
  double* nvo = nullptr;
  auto k = k_tiny<G, E, false, double>;
  const int occ = kernel_blocks_per_sm(k, 256, 0);
  const int grid = persistent_grid(rows, 8 * (32 / G), c.nsm, occ);
  k<<<grid, 256, 0, c.stream>>>(A, B, nv, nv, ri, c.st, lo, hi, c_cnt, nullptr, nullptr, nvo, c.err);
  count_launch(c);
  return cudaGetLastError();
}

// Register-sort bins: 1..4 -> 8 lanes, 5 -> 16 lanes, 6 -> 32 lanes,
// 7 -> 32 lanes x 2 slots, 8 -> x 4, 9 -> x 8, 10 -> x 16 slots (P <= 512).
template <typename F8, typename F16, typename F32, typename F64, typename F128, typename F256, typename F512>
static cudaError_t tiny_dispatch(int lo, int hi, F8 f8, F16 f16, F32 f32, F64 f64, F128 f128, F256 f256,
                                 F512 f512) {
  cudaError_t e = cudaSuccess;
  auto clip = [&](int a, int b, auto f) -> cudaError_t {
    const int l = lo > a ? lo : a, h = hi < b ? hi : b;
    return l <= h ? f(l, h) : cudaSuccess;
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

// Rows of at most 128 products in one launch: one lane and its table per row
// of 17 to 64 products, and of fewer when no row has more than LANE_MERGE_K
// nonzeros (a lane walks its nonzeros one by one; otherwise register sorts), a
// warp and its table above and where the rows are too few for lanes.  The host does not know yet which bins have rows,
// so separate kernels would cost a small product four launches that find
// nothing to do.  (Counting by the numeric pass's merge instead of the lane's
// table: 98 us against 73 on the 96^3 stencil's square.)
constexpr int SYM_SMALL_WARPS = 4;

struct SymBins {
  int tiny_lo, tiny_hi;  // register sort (hi at most 5)
  int lane_hi;           // one lane per row: bins tiny_hi + 1 .. lane_hi
  int hash_hi;           // a warp per row: bins lane_hi + 1 .. hash_hi
};

__global__ void __launch_bounds__(SYM_SMALL_WARPS * 32)
k_sym_small(Csr A, Csr B, RowInfo ri, const DevStats* st, SymBins b, int nsm, int32_t* __restrict__ c_cnt,
            uint32_t* err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_t8[2], s_t16[2], s_lane[2], s_hash[2], s_wide8;
  const int warp = threadIdx.x >> 5, lane = lane_id();
  block_bin_range(st, b.tiny_lo, b.tiny_hi < 4 ? b.tiny_hi : 4, &s_t8[0], &s_t8[1]);
  block_bin_range(st, 5, b.tiny_hi, &s_t16[0], &s_t16[1]);
  block_bin_range(st, b.tiny_hi + 1, b.lane_hi, &s_lane[0], &s_lane[1]);
  block_bin_range(st, b.lane_hi + 1, b.hash_hi, &s_hash[0], &s_hash[1]);
  if (threadIdx.x == 0) s_wide8 = (int)st->rows_wide8;
  if (block_skip(st)) return;
  const long long gw = (long long)blockIdx.x * SYM_SMALL_WARPS + warp;
  const long long nw = (long long)gridDim.x * SYM_SMALL_WARPS;
  const long long from = lane_rows_from(s_wide8, nsm);
  const bool many = s_lane[1] - s_lane[0] >= from;
  const bool lanes = s_wide8 == 0 && s_t8[1] - s_t16[0] >= from;
  int* const keys = reinterpret_cast<int*>(smem_raw) + (size_t)warp * LANE_SLOTS * 32;
  if (s_hash[1] > s_hash[0] || s_lane[1] > s_lane[0] || lanes) {
    for (int h = 0; h < LANE_SLOTS; ++h) keys[h * 32 + lane] = LANE_EMPTY;
    __syncwarp();
  }
  // the warp tables first: their rows are the longest
  hash_sym_rows<4>(A, B, ri, s_hash[0], s_hash[1], gw, nw, keys, c_cnt, err);
  if (!many) {  // too few rows to give every SM several warps of lanes
    hash_sym_rows<2>(A, B, ri, s_lane[0], s_lane[1], gw, nw, keys, c_cnt, err);
  } else {
    lane_hash_rows<false, float>(A, B, nullptr, nullptr, ri, s_lane[0], s_lane[1], gw, nw, keys, nullptr, c_cnt,
                                 nullptr, nullptr, nullptr, err, -1);
  }
  if (lanes) {
    lane_hash_rows<false, float, SPGEMM_PLUS_TIMES, 32>(A, B, nullptr, nullptr, ri, s_t16[0], s_t8[1], gw, nw, keys,
                                                        nullptr, c_cnt, nullptr, nullptr, nullptr, err, -1);
    return;
  }
  tiny_rows<16, 1, false, float>(A, B, nullptr, nullptr, ri, s_t16[0], s_t16[1], gw, nw, c_cnt, nullptr, nullptr,
                                 nullptr, err);
  tiny_rows<8, 1, false, float>(A, B, nullptr, nullptr, ri, s_t8[0], s_t8[1], gw, nw, c_cnt, nullptr, nullptr,
                                nullptr, err);
}

static cudaError_t small_sym(const LaunchCtx& c, const Csr& A, const Csr& B, const RowInfo& ri, const PathBins& pb,
                             int32_t* c_cnt) {
  SymBins b;
  b.tiny_lo = pb.lo[PATH_TINY];
  b.tiny_hi = pb.hi[PATH_TINY];
  b.hash_hi = pb.hi[PATH_HASH];
  b.lane_hi = b.hash_hi < 7 ? b.hash_hi : 7;
  const size_t smem = (size_t)SYM_SMALL_WARPS * LANE_SLOTS * 32 * sizeof(int);
  const int occ = kernel_blocks_per_sm(k_sym_small, SYM_SMALL_WARPS * 32, smem);
  if (occ <= 0) return cudaErrorInvalidConfiguration;
  k_sym_small<<<persistent_grid(ri.mloc, SYM_SMALL_WARPS, c.nsm, occ), SYM_SMALL_WARPS * 32, smem, c.stream>>>(
      A, B, ri, c.st, b, c.nsm, c_cnt, c.err);
  count_launch(c);
  return cudaGetLastError();
}

// Rows above the small ones in one launch: blocks take the longest rows one at
// a time, then their warps the others.  work[4], work[5] hand them out; the
// scan that follows sets them back to zero.
__global__ void __launch_bounds__(SYM_BLOCK_WARPS * 32)
k_sym_large(Csr A, Csr B, RowInfo ri, DevStats* st, int warp_lo, int warp_hi, int block_lo, int block_hi,
            SplitInfo sp, int32_t* __restrict__ cursor, int32_t* __restrict__ c_cnt, uint32_t* err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_b[2], s_w[2], s_nh, s_hs;
  block_bin_range(st, block_lo, block_hi, &s_b[0], &s_b[1]);
  block_bin_range(st, warp_lo, warp_hi, &s_w[0], &s_w[1]);
  if (threadIdx.x == 0) s_nh = split_rows(st, sp, &s_hs);
  if (block_skip(st)) return;
  if (s_b[1] > s_b[0]) {
    sym_block_rows<SYM_BLOCK_W, SYM_BLOCK_WARPS>(A, B, ri, s_b[0], s_b[1], s_hs, s_nh, sp, cursor, c_cnt,
                                                 &st->work[4], smem_raw, err);
    __syncthreads();  // the block's bitmap becomes its warps'
  }
  if (s_w[1] > s_w[0])
    sym_window_rows<SYM_WARP_W>(A, B, ri, s_w[0], s_w[1], s_hs, s_nh, sp, cursor, c_cnt, &st->work[5],
                                smem_raw + (threadIdx.x >> 5) * sym_window_bytes<SYM_WARP_W>(), err);
}

static cudaError_t large_sym(const LaunchCtx& c, const Csr& A, const Csr& B, const RowInfo& ri, const PathBins& pb,
                             const SplitInfo& sp, int32_t* cursor, int32_t* c_cnt) {
  size_t smem = symblock_smem_bytes<SYM_BLOCK_W, SYM_BLOCK_WARPS>();
  const size_t win = SYM_BLOCK_WARPS * sym_window_bytes<SYM_WARP_W>();
  if (win > smem) smem = win;
  const int occ = kernel_blocks_per_sm(k_sym_large, SYM_BLOCK_WARPS * 32, smem);
  if (occ <= 0) return cudaErrorInvalidConfiguration;
  k_sym_large<<<persistent_grid(ri.mloc, 1, c.nsm, occ), SYM_BLOCK_WARPS * 32, smem, c.stream>>>(
      A, B, ri, c.st, pb.lo[PATH_WARP], pb.hi[PATH_WARP], pb.lo[PATH_BLOCK], pb.hi[PATH_BLOCK], sp, cursor, c_cnt,
      c.err);
  count_launch(c);
  return cudaGetLastError();
}

cudaError_t launch_symbolic(const LaunchCtx& c, const Csr& A, const Csr& B, const RowInfo& ri,
                            const PathBins& pb, const SplitInfo& sp, int32_t* cursor, int32_t* c_cnt) {
  cudaError_t e = cudaSuccess;
  if (pb.hi[PATH_HASH] >= pb.lo[PATH_HASH]) {  // with it, register sorts stop at 16 products
    timer_mark(c, T_SYM_HASH, 0);
    e = small_sym(c, A, B, ri, pb, c_cnt);
    timer_mark(c, T_SYM_HASH, 1);
  } else if (pb.hi[PATH_TINY] >= pb.lo[PATH_TINY]) {
    timer_mark(c, T_SYM_TINY, 0);
    e = tiny_dispatch(pb.lo[PATH_TINY], pb.hi[PATH_TINY],
        [&](int l, int h) { return tiny_sym<8, 1>(c, A, B, ri, l, h, c_cnt, -1); },
        [&](int l, int h) { return tiny_sym<16, 1>(c, A, B, ri, l, h, c_cnt, -1); },
        [&](int l, int h) { return tiny_sym<32, 1>(c, A, B, ri, l, h, c_cnt, -1); },
        [&](int l, int h) { return tiny_sym<32, 2>(c, A, B, ri, l, h, c_cnt, -1); },
        [&](int l, int h) { return tiny_sym<32, 4>(c, A, B, ri, l, h, c_cnt, -1); },
        [&](int l, int h) { return tiny_sym<32, 8>(c, A, B, ri, l, h, c_cnt, -1); },
        [&](int l, int h) { return tiny_sym<32, 16>(c, A, B, ri, l, h, c_cnt, -1); });
    timer_mark(c, T_SYM_TINY, 1);
  }
  if (e != cudaSuccess) return e;
  if (pb.hi[PATH_WARP] >= pb.lo[PATH_WARP] || pb.hi[PATH_BLOCK] >= pb.lo[PATH_BLOCK]) {
    timer_mark(c, T_SYM_BLOCK, 0);
    e = large_sym(c, A, B, ri, pb, sp, cursor, c_cnt);
    timer_mark(c, T_SYM_BLOCK, 1);
  }
  return e;
}

}  // namespace sg
