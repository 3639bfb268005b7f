// Lane-per-row hash accumulator for rows of 17..64 products (bins 6..7):
// every row of a 3D 7-point stencil product (49 products, 25 columns) and of
// the Galerkin coarse product lands here.
//
// Row-wise Gustavson (Sec. 2.2): row i of C is the sum of the scaled rows
// A(i,k) * B(k,:), equal columns merged by adding their values (Algorithm
// 1), the row emitted with ascending columns.
//
// A warp takes 32 rows at once, one per lane.  Each lane owns a private
// open-addressing table of 64 slots in shared memory, laid out slot-major
// ([slot][lane]), so whatever slots the 32 lanes touch, each lane stays in
// its own bank: no bank conflicts and no atomics.  A lane walks its row's
// products one by one -- the first product of a column stores A(i,k)*B(k,j),
// later ones add with one fused multiply-add -- then compacts its occupied
// slots into a list (clearing the table for its next row) and writes each
// listed column at the position given by the number of smaller listed
// columns.  A warp-per-row table instead pays a shared-memory atomic per
// product, an FP64 reduction per repeated column (the FP64 pipe runs one
// such instruction per conflicting lane), and warp-wide gather and ranking
// work per row; here the FP64 pipe does one operation per product with all
// 32 lanes busy.
//
// A row of P <= 64 products has at most 64 distinct columns, so its table
// never overflows (the probe loop is bounded by the table size).
//
// Rows with at most 8 nonzeros of A (the 7-point stencil's) skip the table:
// their B rows are merged in column order from registers (lane_merge_rows).
#pragma once

#include "launch_util.cuh"
#include "semiring.cuh"

namespace sg {

constexpr int LANE_SLOTS = 64;     // table slots per lane (rows of at most 64 products)
constexpr int LANE_WARPS = 4;      // warps per block
constexpr int LANE_EMPTY = -1;
// Fewest rows per SM that take a lane each; with rows of more than
// LANE_MERGE_K nonzeros among them (wide8) many more, since their tables walk
// one entry at a time.  A warp and its table per row otherwise: 24,013 rows of
// 49 products on random columns 69 us by lanes, 31 by warps; 85,184 rows of a
// 44^3 stencil 25 and 74; 50,000 rows of 2 to 12 nonzeros 246 and 71.
constexpr int LANE_ROWS_PER_SM = 160;
constexpr int LANE_ROWS_PER_SM_WIDE = 1024;

__host__ __device__ inline long long lane_rows_from(long long wide8, int nsm) {
  return (long long)nsm * (wide8 ? LANE_ROWS_PER_SM_WIDE : LANE_ROWS_PER_SM);
}

template <int SLOTS>
__device__ __forceinline__ unsigned lane_hash(int c) {
  return ((unsigned)c * 0x9E3779B1u) >> (SLOTS == 64 ? 26 : 27);
}

// Slot of column j in the lane's table (claimed if absent; *fresh tells).
// keys: this warp's table base, slot-major.  -1 if the table is full of
// other columns (ruled out by the row's product count).
template <int SLOTS>
__device__ __forceinline__ int lane_probe(int* keys, int lane, int j, bool* fresh) {
  static_assert(SLOTS == 64 || SLOTS == 32, "slots per lane");
  unsigned h = lane_hash<SLOTS>(j);
  *fresh = false;
  for (int it = 0; it < SLOTS; ++it) {
    int* kp = &keys[h * 32 + lane];
    const int k = *kp;
    if (k == j) return (int)h;
    if (k == LANE_EMPTY) {
      *kp = j;
      *fresh = true;
      return (int)h;
    }
    h = (h + 1u) & (SLOTS - 1);
  }
  return -1;
}

// NUM = false: c_cnt[r] = distinct columns of row r.  NUM = true: C's
// columns and values at [c_rp[r], c_rp[r+1]).  Rows at list positions
// [lb, le), warp gw of nw takes its share; rows of at most skip_upto nonzeros
// are left out.  keys (all LANE_EMPTY) and vals: this warp's.  SLOTS: 64, or
// 32 for rows of at most 16 products.
template <bool NUM, typename T, int SR = SPGEMM_PLUS_TIMES, int SLOTS = LANE_SLOTS>
__device__ __forceinline__ void lane_hash_rows(const Csr& A, const Csr& B, const T* __restrict__ av,
                                               const T* __restrict__ bv, const RowInfo& ri, long long lb,
                                               long long le, long long gw, long long nw, int* keys, T* vals,
                                               int32_t* __restrict__ c_cnt, const int32_t* __restrict__ c_rp,
                                               int32_t* __restrict__ c_ci, T* __restrict__ c_v, uint32_t* err,
                                               int skip_upto) {
  const int lane = lane_id();
  for (long long base = lb + gw * 32; base < le; base += nw * 32) {
    const long long idx = base + lane;
    if (idx < le) {
      const int r = ri.rows[idx];
      const long long i = ri.row_begin + r;
      const int a0 = A.rp[i], a1 = A.rp[i + 1];
      if (a1 - a0 <= skip_upto) continue;  // k_lane_merge took the row
      int nd = 0;     // distinct columns so far
      int np = 0;     // products so far
      bool over = false;
      for (int e = a0; e < a1; ++e) {
        const int k = A.ci[e];
        const T a = NUM ? av[e] : T(0);
        const int q0 = B.rp[k], q1 = B.rp[k + 1];
        // B(k,:) in groups of 8 entries whose loads are all issued before
        // the group's table updates (the updates depend on each other
        // through the table, the loads do not)
        for (int g = q0; g < q1; g += 8) {
          int jj[8];
          T bb[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            jj[u] = g + u < q1 ? B.ci[g + u] : -1;
            if (NUM) bb[u] = g + u < q1 ? bv[g + u] : T(0);
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            if (jj[u] < 0) continue;
            bool fresh;
            const int h = lane_probe<SLOTS>(keys, lane, jj[u], &fresh);
            ++np;
            if (h < 0) {
              over = true;
              continue;
            }
            if (fresh) ++nd;
            if (NUM) {
              T* vp = &vals[h * 32 + lane];
              *vp = fresh ? SrOps<T, SR>::first(SrOps<T, SR>::mul(a, bb[u])) : SrOps<T, SR>::madd(a, bb[u], *vp);
            }
          }
        }
      }
      if (over || np > SLOTS) atomicOr(err, EB_INTERNAL);  // the row's bin rules this out
      if (!NUM) {
        c_cnt[r] = nd;
        for (int h = 0; h < SLOTS; ++h) keys[h * 32 + lane] = LANE_EMPTY;
      } else {
        // compact the occupied slots into slots [0, nd) of a list kept in
        // the same columns (read slot h before writing entry d <= h), and
        // clear the rest of the table
        int d = 0;
        for (int h = 0; h < SLOTS; ++h) {
          const int k = keys[h * 32 + lane];
          if (k != LANE_EMPTY) {
            const T v = vals[h * 32 + lane];
            keys[h * 32 + lane] = LANE_EMPTY;
            keys[d * 32 + lane] = k;  // d <= h
            vals[d * 32 + lane] = v;
            ++d;
          }
        }
        const int ob = c_rp[r], oe = c_rp[r + 1];
        if (ob + d != oe) atomicOr(err, EB_INTERNAL);
        // output position of a column: the listed columns smaller than it
        for (int x = 0; x < d; ++x) {
          const int kx = keys[x * 32 + lane];
          int r0 = 0, r1 = 0, r2 = 0, r3 = 0;  // four independent counts, so the loads overlap
          int y = 0;
          for (; y + 4 <= d; y += 4) {
            r0 += keys[y * 32 + lane] < kx;
            r1 += keys[(y + 1) * 32 + lane] < kx;
            r2 += keys[(y + 2) * 32 + lane] < kx;
            r3 += keys[(y + 3) * 32 + lane] < kx;
          }
          for (; y < d; ++y) r0 += keys[y * 32 + lane] < kx;
          const int rank = r0 + r1 + r2 + r3;
          const int o = ob + rank;
          if (o < oe) {
            c_ci[o] = kx;
            c_v[o] = vals[x * 32 + lane];
          }
        }
        for (int x = 0; x < d; ++x) keys[x * 32 + lane] = LANE_EMPTY;
      }
    }
  }
}

template <typename T, int SR = SPGEMM_PLUS_TIMES>
__global__ void __launch_bounds__(LANE_WARPS * 32)
k_lane_rows(Csr A, Csr B, const T* __restrict__ av, const T* __restrict__ bv, RowInfo ri, const DevStats* st,
            int bin_lo, int bin_hi, const int32_t* __restrict__ c_rp, int32_t* __restrict__ c_ci,
            T* __restrict__ c_v, uint32_t* err, int skip_upto) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_lb, s_le;
  const int warp = threadIdx.x >> 5, lane = lane_id();
  // per warp: keys [64][32] int32, then values [64][32] T
  const size_t per_warp = (size_t)LANE_SLOTS * 32 * (sizeof(int) + sizeof(T));
  int* keys = reinterpret_cast<int*>(smem_raw + warp * per_warp);
  T* vals = reinterpret_cast<T*>(smem_raw + warp * per_warp + (size_t)LANE_SLOTS * 32 * sizeof(int));
  for (int h = 0; h < LANE_SLOTS; ++h) keys[h * 32 + lane] = LANE_EMPTY;
  block_bin_range(st, bin_lo, bin_hi, &s_lb, &s_le);
  if (block_skip(st)) return;
  lane_hash_rows<true, T, SR>(A, B, av, bv, ri, s_lb, s_le, (long long)blockIdx.x * LANE_WARPS + warp,
                              (long long)gridDim.x * LANE_WARPS, keys, vals, nullptr, c_rp, c_ci, c_v, err, skip_upto);
}

// Rows with at most LANE_MERGE_K nonzeros of A (every row of a 7-point
// stencil product and of a stencil times an aggregation): one lane per row
// merges its B rows -- the next output column is the smallest head column,
// its value the products of the heads that hold it, each head advanced past
// it -- so the row comes out in column order with no table and no ranking.
// The sums run in A's order, every product fused into the running sum from
// the semiring's identity (for plus-times the first product is a*b rounded,
// +0 where that product is exactly -0).
//
// A head's column, the column after it and its value are in registers, read
// one step before they are needed, so no shared memory holds B rows and an SM
// keeps as many warps as the registers allow.  Outputs are collected 8 per
// row and written by 8 lanes per row: lanes that wrote their own rows would
// touch 32 sectors with every store.  96^3 stencil squared in FP64: 0.37 ms
// with the B rows staged in shared memory (8 warps per SM, lanes storing their
// own rows), 0.20 ms here (20 warps at 96 registers); the floor of one FP64
// operation per product and full warps is 0.07 ms, that of the bytes 0.04 ms.
// A heads' test issues its FP64 instruction when any lane of the warp matches.
constexpr int LANE_MERGE_K = 8;
constexpr int LANE_OUT = 8;          // outputs collected per row
constexpr int LANE_OUT_CI = 36;      // strides of the collecting arrays that keep both
constexpr int LANE_OUT_V = 34;       // sides of the exchange free of bank conflicts

template <typename T>
struct LaneOut {
  T val[LANE_OUT * LANE_OUT_V];
  int col[LANE_OUT * LANE_OUT_CI];
};

// The 8 outputs from `first` on of every lane's row (n: the row's outputs so
// far, its entries go to [ob, oe)).  Every lane must call it.
template <typename T>
__device__ __forceinline__ void lane_flush(const LaneOut<T>& so, int first, int n, int ob, int oe,
                                           int32_t* __restrict__ c_ci, T* __restrict__ c_v) {
  const int lane = lane_id(), t = lane & 7;
  __syncwarp();
#pragma unroll
  for (int g = 0; g < 8; ++g) {
    const int j = g * 4 + (lane >> 3);
    const int nj = __shfl_sync(FULL, n, j), oj = __shfl_sync(FULL, ob, j), ej = __shfl_sync(FULL, oe, j);
    const int o = oj + first + t;
    if (first + t < nj && o < ej) {
      c_ci[o] = so.col[t * LANE_OUT_CI + j];
      c_v[o] = so.val[t * LANE_OUT_V + j];
    }
  }
  __syncwarp();
}

// One warp's 32 rows (a0 == a1: none): columns and values to [ob, oe);
// returns the lane's distinct columns.
template <typename T, int SR>
__device__ __forceinline__ int lane_merge_rows(const Csr& A, const Csr& B, const T* __restrict__ av,
                                               const T* __restrict__ bv, int a0, int a1, LaneOut<T>* so, int ob,
                                               int oe, int32_t* __restrict__ c_ci, T* __restrict__ c_v) {
  using Ops = SrOps<T, SR>;
  constexpr int K = LANE_MERGE_K;
  const int lane = lane_id();
  int hs[K], he[K], hc[K], hn[K];  // head position, end, head column, the column after it
  T a[K], v[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    hs[k] = he[k] = 0;
    a[k] = v[k] = T(0);
    if (a0 + k < a1) {
      const int kk = A.ci[a0 + k];
      hs[k] = B.rp[kk];
      he[k] = B.rp[kk + 1];
      a[k] = av[a0 + k];
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    hc[k] = hs[k] < he[k] ? B.ci[hs[k]] : INT_MAX;
    hn[k] = hs[k] + 1 < he[k] ? B.ci[hs[k] + 1] : INT_MAX;
    if (hs[k] < he[k]) v[k] = bv[hs[k]];
  }
  int n = 0;
  for (int step = 0;; ++step) {
    int m = hc[0];
#pragma unroll
    for (int k = 1; k < K; ++k) m = min(m, hc[k]);
    const bool act = m != INT_MAX;
    if (step > 0 && (step & (LANE_OUT - 1)) == 0) lane_flush(*so, step - LANE_OUT, n, ob, oe, c_ci, c_v);
    if (!__any_sync(FULL, act)) {
      if ((step & (LANE_OUT - 1)) != 0) lane_flush(*so, step & ~(LANE_OUT - 1), n, ob, oe, c_ci, c_v);
      break;
    }
    if (act) {
      T acc = Ops::zero();
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (hc[k] == m) {
          acc = Ops::madd(a[k], v[k], acc);  // one FP64 instruction per head test
          ++hs[k];
          hc[k] = hn[k];
          hn[k] = hs[k] + 1 < he[k] ? B.ci[hs[k] + 1] : INT_MAX;
          if (hs[k] < he[k]) v[k] = bv[hs[k]];
        }
      }
      so->col[(step & (LANE_OUT - 1)) * LANE_OUT_CI + lane] = m;
      so->val[(step & (LANE_OUT - 1)) * LANE_OUT_V + lane] = acc;
      ++n;
    }
  }
  return n;
}

template <typename T, int SR>
__global__ void __launch_bounds__(LANE_WARPS * 32)
k_lane_merge(Csr A, Csr B, const T* __restrict__ av, const T* __restrict__ bv, RowInfo ri, const DevStats* st,
             int bin_lo, int bin_hi, const int32_t* __restrict__ c_rp, int32_t* __restrict__ c_ci,
             T* __restrict__ c_v, uint32_t* err) {
  __shared__ LaneOut<T> s_out[LANE_WARPS];
  __shared__ int s_lb, s_le;
  const int warp = threadIdx.x >> 5, lane = lane_id();
  block_bin_range(st, bin_lo, bin_hi, &s_lb, &s_le);
  if (block_skip(st)) return;
  const long long lb = s_lb, le = s_le;
  const long long gw = (long long)blockIdx.x * LANE_WARPS + warp;
  const long long nw = (long long)gridDim.x * LANE_WARPS;
  for (long long base = lb + gw * 32; base < le; base += nw * 32) {
    const long long idx = base + lane;
    int a0 = 0, a1 = 0, ob = 0, oe = 0;
    if (idx < le) {
      const int r = ri.rows[idx];
      a0 = A.rp[ri.row_begin + r];
      a1 = A.rp[ri.row_begin + r + 1];
      if (a1 - a0 > LANE_MERGE_K) a0 = a1;  // k_lane_rows takes the row
      if (a1 > a0) {
        ob = c_rp[r];
        oe = c_rp[r + 1];
      }
    }
    const int n = lane_merge_rows<T, SR>(A, B, av, bv, a0, a1, &s_out[warp], ob, oe, c_ci, c_v);
    if (a1 > a0 && ob + n != oe) atomicOr(err, EB_INTERNAL);  // the symbolic count rules this out
  }
}

template <typename T>
constexpr size_t lane_rows_smem() {
  return (size_t)LANE_WARPS * LANE_SLOTS * 32 * (sizeof(int) + sizeof(T));
}

// Numeric launch over the rows of bins [lo, hi] (rows: their number, -1
// unknown): rows of at most LANE_MERGE_K nonzeros of A are merged, the others
// (wide8: rows of the plan with more, -1 unknown) go through the tables.
template <typename T, int SR = SPGEMM_PLUS_TIMES>
static cudaError_t lane_rows(const LaunchCtx& c, const Csr& A, const Csr& B, const T* av, const T* bv,
                             const RowInfo& ri, int lo, int hi, const int32_t* c_rp, int32_t* c_ci, T* c_v,
                             long long rows, long long wide8) {
  auto km = k_lane_merge<T, SR>;
  const int occm = kernel_blocks_per_sm(km, LANE_WARPS * 32, 0);
  if (occm <= 0) return cudaErrorInvalidConfiguration;
  km<<<persistent_grid(rows, LANE_WARPS * 32, c.nsm, occm), LANE_WARPS * 32, 0, c.stream>>>(
      A, B, av, bv, ri, c.st, lo, hi, c_rp, c_ci, c_v, c.err);
  count_launch(c);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || wide8 == 0) return e;
  auto k = k_lane_rows<T, SR>;
  const size_t smem = lane_rows_smem<T>();
  const int occ = kernel_blocks_per_sm(k, LANE_WARPS * 32, smem);
  if (occ <= 0) return cudaErrorInvalidConfiguration;
  k<<<persistent_grid(rows, LANE_WARPS * 32, c.nsm, occ), LANE_WARPS * 32, smem, c.stream>>>(
      A, B, av, bv, ri, c.st, lo, hi, c_rp, c_ci, c_v, c.err, LANE_MERGE_K);
  count_launch(c);
  return cudaGetLastError();
}

}  // namespace sg
