// Adjoint of C = A*B for a scalar loss L with dL/dC = dC given on C's
// pattern (the loss L = sum W .* C has dC = W):
//   dA(i,k) = sum_j dC(i,j) * B(k,j)   on the pattern of A   (dC * B^T sampled)
//   dB(k,j) = sum_i A(i,k) * dC(i,j)   on the pattern of B   (A^T * dC sampled)
// Every (i,k,j) with A(i,k), B(k,j) nonzero has C(i,j) in C's pattern, so
// each lookup of dC(i,j) succeeds.  Both gradients need the same lookup, one
// per scalar product of the forward pass; everything else is streaming.
//
// The lookups run once, in the order of A's rows, where row i of C is at
// hand: k_grad_rows stages its values with a presence bitmap of its columns
// in shared memory, finds dC(i,j) as a rank (one bitmap word and its prefix),
// sums dA(i,k) on the spot and writes the values dC(i,j) to a buffer in
// product order -- B(k,:) long and contiguous for every nonzero (i,k).
// k_grad_cols then sums dB(k,:) over the nonzeros of A^T(k,:), each a
// contiguous read of the buffer.  The buffer holds a chunk of the products at
// a time (64 MB, so that it stays in the L2 cache between the two kernels);
// the chunks follow each other in product order and add to dB in that order.
// Rows of C that are too short to be worth a block or too long or too wide
// for its shared memory are searched in global memory by k_grad_slabs.
//
// Orders are fixed (a lane's own chain, fixed trees, chunks in order), nothing
// is accumulated atomically: the same bits on every run, and for dB whether it
// passes through the buffer or not (grad_route says when it does).
//
// 65,536 rows of 32 x 32 products, FP32: a binary search in C's row per
// product and gradient (k_grad_a, k_grad_b) took 0.82 ms for dA and 1.88 ms for
// dB, bound by the memory latency and the 32-byte sectors of scattered searches
// in C (533 MB).  Here k_grad_rows takes 0.44 ms for four chunks (bound by the
// latency of a row's loads, 7.3 of 14 stalled warps per issue, 8 of 16 warps per
// scheduler resident at 64 registers), k_grad_cols 0.18 ms (load latency; L1 50 %
// and DRAM 31 % busy).
#include <cmath>

#include "launch_util.cuh"

namespace sg {

// Sums of at most this many terms stay in one lane: with lanes of a slab
// summing up to this many terms each, their chains run side by side; a sum
// far longer than its neighbours' (a hub row) would hold the warp alone.
constexpr int GRAD_LANE_MAX = 128;

constexpr long long GRAD_BUFFER_BYTES = 64ll << 20;  // a chunk of the products' dC values: half the L2 cache
constexpr int GRAD_ROW_CAP = 4096;                   // entries of a row of C staged in shared memory

__device__ __forceinline__ int find_col(const int32_t* __restrict__ ci, int lo, int hi, int c) {
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (ci[mid] < c) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// out[q] = the row holding entry q (one warp per row), so the gradient
// kernels find an output's row with one load.
__global__ void __launch_bounds__(256) k_row_index(const int32_t* __restrict__ rp, long long nrows,
                                                   int32_t* __restrict__ out) {
  const long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nw = (gridDim.x * (long long)blockDim.x) >> 5;
  const int lane = lane_id();
  for (long long r = w; r < nrows; r += nw)
    for (int q = rp[r] + lane; q < rp[r + 1]; q += 32) out[q] = (int32_t)r;
}

// Sum of the 32 lanes' partial sums in a fixed order (a butterfly tree).
template <typename T>
__device__ __forceinline__ T warp_sum_fixed(T v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(FULL, v, d);
  return v;
}

// dA over the plan's rows [row_begin, row_begin + mloc): output e = (i,k) is
// the dot product of B(k,:) with dC(i,:).
template <typename T>
__global__ void __launch_bounds__(256) k_grad_a(Csr A, Csr B, const T* __restrict__ bv, long long row_begin,
                                                long long mloc, const int32_t* __restrict__ a_row,
                                                const int32_t* __restrict__ c_rp,
                                                const int32_t* __restrict__ c_ci, const T* __restrict__ dc,
                                                T* __restrict__ da, uint32_t* err) {
  const int lane = lane_id();
  const long long e_lo = A.rp[row_begin], e_hi = A.rp[row_begin + mloc];
  const long long nslab = (e_hi - e_lo + 31) >> 5;
  const long long w0 = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nw = (gridDim.x * (long long)blockDim.x) >> 5;
  for (long long s = w0; s < nslab; s += nw) {
    const long long e = e_lo + (s << 5) + lane;
    const bool have = e < e_hi;
    int k = 0, b0 = 0, b1 = 0, c0 = 0, c1 = 0;
    if (have) {
      const long long r = (long long)a_row[e] - row_begin;
      k = A.ci[e];
      b0 = B.rp[k];
      b1 = B.rp[k + 1];
      c0 = c_rp[r];
      c1 = c_rp[r + 1];
    }
    const bool wide = have && b1 - b0 > GRAD_LANE_MAX;
    // short sums: the lane's own chain, walking B(k,:) (ascending, so the
    // search range narrows)
    T acc = T(0);
    if (have && !wide) {
      int lo = c0;
      for (int q = b0; q < b1; ++q) {
        const int j = B.ci[q];
        const int pos = find_col(c_ci, lo, c1, j);
        if (pos < c1 && c_ci[pos] == j) {
          acc = fma(dc[pos], bv[q], acc);
          lo = pos + 1;
        } else {
          atomicOr(err, EB_INTERNAL);
        }
      }
    }
    // long sums: the whole warp on one output at a time
    unsigned wm = __ballot_sync(FULL, wide);
    while (wm) {
      const int L = __ffs(wm) - 1;
      wm &= wm - 1;
      const int lb0 = __shfl_sync(FULL, b0, L), lb1 = __shfl_sync(FULL, b1, L);
      const int lc0 = __shfl_sync(FULL, c0, L), lc1 = __shfl_sync(FULL, c1, L);
      T part = T(0);
      for (int q = lb0 + lane; q < lb1; q += 32) {
        const int j = B.ci[q];
        const int pos = find_col(c_ci, lc0, lc1, j);
        if (pos < lc1 && c_ci[pos] == j) part = fma(dc[pos], bv[q], part);
        else atomicOr(err, EB_INTERNAL);
      }
      const T tot = warp_sum_fixed(part);
      if (lane == L) acc = tot;
    }
    if (have) da[e] = acc;
  }
}

// dB: output q = (k,j) of B sums A(i,k) * dC(i,j) over the rows i of A (in
// the plan's range) with a nonzero in column k, i.e. over A^T(k,:), whose
// entries (t_ci: row i, t_src: position of A(i,k)) the plan keeps.
template <typename T>
__global__ void __launch_bounds__(256) k_grad_b(Csr B, const T* __restrict__ av, const int32_t* __restrict__ b_row,
                                                const int32_t* __restrict__ t_rp,
                                                const int32_t* __restrict__ t_ci, const int32_t* __restrict__ t_src,
                                                long long row_begin, long long row_end,
                                                const int32_t* __restrict__ c_rp, const int32_t* __restrict__ c_ci,
                                                const T* __restrict__ dc, T* __restrict__ db, uint32_t* err) {
  const int lane = lane_id();
  const long long nslab = (B.nnz + 31) >> 5;
  const long long w0 = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nw = (gridDim.x * (long long)blockDim.x) >> 5;
  for (long long s = w0; s < nslab; s += nw) {
    const long long q = (s << 5) + lane;
    const bool have = q < B.nnz;
    int j = 0, t0 = 0, t1 = 0;
    if (have) {
      const int k = b_row[q];
      j = B.ci[q];
      t0 = t_rp[k];
      t1 = t_rp[k + 1];
    }
    const bool wide = have && t1 - t0 > GRAD_LANE_MAX;
    T acc = T(0);
    if (have && !wide) {
      for (int t = t0; t < t1; ++t) {
        const long long i = t_ci[t];
        if (i < row_begin || i >= row_end) continue;  // rows outside the plan's range
        const int r = (int)(i - row_begin);
        const int c0 = c_rp[r], c1 = c_rp[r + 1];
        const int pos = find_col(c_ci, c0, c1, j);
        if (pos < c1 && c_ci[pos] == j) acc = fma(av[t_src[t]], dc[pos], acc);
        else atomicOr(err, EB_INTERNAL);
      }
    }
    unsigned wm = __ballot_sync(FULL, wide);
    while (wm) {
      const int L = __ffs(wm) - 1;
      wm &= wm - 1;
      const int lj = __shfl_sync(FULL, j, L);
      const int lt0 = __shfl_sync(FULL, t0, L), lt1 = __shfl_sync(FULL, t1, L);
      T part = T(0);
      for (int t = lt0 + lane; t < lt1; t += 32) {
        const long long i = t_ci[t];
        if (i < row_begin || i >= row_end) continue;
        const int r = (int)(i - row_begin);
        const int c0 = c_rp[r], c1 = c_rp[r + 1];
        const int pos = find_col(c_ci, c0, c1, lj);
        if (pos < c1 && c_ci[pos] == lj) part = fma(av[t_src[t]], dc[pos], part);
        else atomicOr(err, EB_INTERNAL);
      }
      const T tot = warp_sum_fixed(part);
      if (lane == L) acc = tot;
    }
    if (have) db[q] = acc;
  }
}

// ------------------------------------------------- product offsets (plan)
// off[r] = exclusive prefix sum of cnt (64 bits), off[n] the total: tile sums,
// one block over the tile sums, tiles again.
constexpr int OFF_THREADS = 256;
constexpr int OFF_TILE = OFF_THREADS * 16;

__device__ __forceinline__ long long off_block_scan(long long v, long long* total) {
  __shared__ long long s_w[OFF_THREADS / 32];
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  const long long incl = warp_incl_scan(v);
  __syncthreads();
  if (lane == 31) s_w[warp] = incl;
  __syncthreads();
  long long before = 0, all = 0;
  for (int w = 0; w < OFF_THREADS / 32; ++w) {
    if (w < warp) before += s_w[w];
    all += s_w[w];
  }
  *total = all;
  return before + incl - v;
}

__global__ void __launch_bounds__(OFF_THREADS) k_off_tiles(const long long* __restrict__ cnt, long long n,
                                                          long long* __restrict__ part) {
  const long long base = (long long)blockIdx.x * OFF_TILE;
  long long v = 0, total;
  for (int u = 0; u < 16; ++u) {
    const long long r = base + u * OFF_THREADS + threadIdx.x;
    if (r < n) v += cnt[r];
  }
  off_block_scan(v, &total);
  if (threadIdx.x == 0) part[blockIdx.x] = total;
}

__global__ void __launch_bounds__(OFF_THREADS) k_off_partials(long long* __restrict__ part, long long tiles) {
  long long carry = 0;
  for (long long b = 0; b < tiles; b += OFF_THREADS) {
    const long long i = b + threadIdx.x;
    long long total;
    const long long ex = off_block_scan(i < tiles ? part[i] : 0, &total);
    if (i < tiles) part[i] = carry + ex;
    carry += total;
  }
}

__global__ void __launch_bounds__(OFF_THREADS) k_off_down(const long long* __restrict__ cnt, long long n,
                                                         const long long* __restrict__ part,
                                                         long long* __restrict__ off) {
  const long long base = (long long)blockIdx.x * OFF_TILE;
  long long carry = part[blockIdx.x];
  for (int u = 0; u < 16; ++u) {
    const long long r = base + u * OFF_THREADS + threadIdx.x;
    const long long v = r < n ? cnt[r] : 0;
    long long total;
    const long long ex = off_block_scan(v, &total);
    if (r < n) off[r] = carry + ex;
    if (r == n - 1) off[n] = carry + ex + v;
    carry += total;
  }
}

// p_off[e] = products before nonzero e of A (rows of the plan's range): the
// row's offset plus the lengths of the row's earlier rows of B.  A warp per row.
__global__ void __launch_bounds__(256) k_product_offsets(Csr A, Csr B, long long row_begin, long long mloc,
                                                         const long long* __restrict__ row_off,
                                                         long long* __restrict__ p_off, const DevStats* st) {
  if (block_skip(st)) return;
  const int lane = lane_id();
  const long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nw = (gridDim.x * (long long)blockDim.x) >> 5;
  for (long long r = w; r < mloc; r += nw) {
    const int a0 = A.rp[row_begin + r], a1 = A.rp[row_begin + r + 1];
    long long before = row_off[r];
    for (int e0 = a0; e0 < a1; e0 += 32) {
      const int e = e0 + lane;
      int len = 0;
      if (e < a1) {
        const int k = A.ci[e];
        if (k >= 0 && (long long)k < B.nrows) len = B.rp[k + 1] - B.rp[k];
      }
      const long long incl = warp_incl_scan((long long)len);
      if (e < a1) p_off[e] = before + incl - len;
      before += __shfl_sync(FULL, incl, 31);
    }
  }
}

// The same offsets in the order of A^T; rows before and after the plan's
// range lie below and above every product.  Also the lengths of A's longest
// column and B's longest row, into the plan's statistics.
__global__ void __launch_bounds__(256) k_transposed_offsets(long long nnz, const int32_t* __restrict__ t_ci,
                                                            const int32_t* __restrict__ t_src, long long row_begin,
                                                            long long row_end, const long long* __restrict__ p_off,
                                                            long long* __restrict__ t_off,
                                                            const int32_t* __restrict__ t_rp,
                                                            const int32_t* __restrict__ b_rp, long long nrows_b,
                                                            DevStats* st) {
  if (block_skip(st)) return;
  int col = 0, row = 0;
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < nrows_b;
       k += (long long)gridDim.x * blockDim.x) {
    col = max(col, t_rp[k + 1] - t_rp[k]);
    row = max(row, b_rp[k + 1] - b_rp[k]);
  }
  col = warp_max(col);
  row = warp_max(row);
  if (lane_id() == 0 && col > 0) atomicMax(&st->max_col, col);
  if (lane_id() == 0 && row > 0) atomicMax(&st->max_row_b, row);
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < nnz; t += (long long)gridDim.x * blockDim.x) {
    const long long i = t_ci[t];
    t_off[t] = i < row_begin ? -1ll : (i >= row_end ? LLONG_MAX : p_off[t_src[t]]);
  }
}

// First index of the non-decreasing v[lo, hi) with v[index] >= x (hi if none).
template <typename I>
__device__ __forceinline__ I first_at_least(const long long* __restrict__ v, I lo, I hi, long long x) {
  while (lo < hi) {
    const I mid = lo + (hi - lo) / 2;
    if (v[mid] < x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// The same for a whole warp with one x: 32 probes a step (a block's single
// search over millions of offsets would otherwise be 20 dependent loads).
__device__ __forceinline__ long long warp_first_at_least(const long long* __restrict__ v, long long lo, long long hi,
                                                         long long x) {
  while (lo < hi) {
    const long long step = (hi - lo + 31) / 32;
    const long long q = lo + (long long)lane_id() * step;
    const unsigned below = __ballot_sync(FULL, q < hi && v[q < hi ? q : lo] < x);
    if (!below) return lo;
    const int last = 31 - __clz(below);  // v is non-decreasing: lanes 0..last are below x
    lo += last * step + 1;
    hi = min(hi, lo + step - 1);
  }
  return lo;
}

// ---------------------------------------------------- both gradients' lookups
// Which rows of C k_grad_rows takes: more than GRAD_ROW_MIN entries, at most
// `cap`, and a column span inside one bitmap of 2^wlog columns.
constexpr int GRAD_ROW_MIN = 128;

__device__ __forceinline__ bool grad_row_staged(int n, int cmin, int cmax, int cap, int wlog) {
  return n > GRAD_ROW_MIN && n <= cap && (long long)cmax - (cmin & ~31) < (1ll << wlog);
}

// One chunk [c0, c1) of the products, rows of C staged in shared memory, one
// block per row.  G lanes take a nonzero (i,k) and walk B(k,:) together; a
// warp keeps 8 nonzeros per lane group in flight and folds their 8 partial
// sums with one exchange tree (FP64 additions cost a warp the same with any
// number of lanes: 8 separate trees would take 8 * log2(G) of them, the folded
// one 7 + log2(G) - 3).  buf may be null (dB not wanted), da as well.
//
// A row is a chain of loads (its extents, its part of C, its nonzeros, their
// rows of B) with three barriers, so latency bounds it: the next row's extents
// are loaded a row ahead and its part of C and dC prefetched into the L2 cache,
// and the first 4 * NT entries of C are in flight beside the nonzeros.  65,536
// rows of 32 x 32 products, FP32: 624 us without that, 444 with it (67 M
// products: 12 bytes each from the caches or to the buffer).
template <int NT, int G, typename T>
__global__ void __launch_bounds__(NT)
k_grad_rows(Csr A, Csr B, const T* __restrict__ bv, RowInfo ri, const long long* __restrict__ row_off,
            const long long* __restrict__ p_off, const int32_t* __restrict__ c_rp, const int32_t* __restrict__ c_ci,
            const T* __restrict__ dc, T* __restrict__ da, T* __restrict__ buf, long long c0, long long c1, int cap,
            int wlog, uint32_t* err) {
  constexpr int NW = NT / 32, GPW = 32 / G, S = 8;
  constexpr int LG = G == 32 ? 5 : (G == 16 ? 4 : 3);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* const sdc = reinterpret_cast<T*>(smem_raw);
  uint32_t* const bits = reinterpret_cast<uint32_t*>(sdc + cap);
  uint16_t* const pre = reinterpret_cast<uint16_t*>(bits + ((1 << wlog) >> 5));
  __shared__ long long s_first;
  const int tid = threadIdx.x, warp = tid >> 5, lane = lane_id(), gl = lane & (G - 1), g = lane / G;
  for (int t = tid; t < (1 << wlog) / 32; t += NT) bits[t] = 0u;
  // first row with a product or an empty nonzero at or past c0
  if (warp == 0) {
    const long long f = c0 <= 0 ? 0 : warp_first_at_least(row_off, 1, ri.mloc + 1, c0) - 1;
    if (lane == 0) s_first = f;
  }
  __syncthreads();
  // a row's extents are read one row ahead, and its part of C and dC is asked
  // into the L2 cache then
  struct Row {
    long long off;
    int p0, n, cmn, cmx, a0, a1;
  };
  auto extents = [&](long long r) {
    Row x{LLONG_MAX, 0, 0, 0, 0, 0, 0};
    if (r < ri.mloc) {
      x.off = row_off[r];
      x.p0 = c_rp[r];
      x.n = c_rp[r + 1] - x.p0;
      x.cmn = ri.cmin[r];
      x.cmx = ri.cmax[r];
      x.a0 = A.rp[ri.row_begin + r];
      x.a1 = A.rp[ri.row_begin + r + 1];
    }
    return x;
  };
  Row row = extents(s_first + blockIdx.x);
  for (long long r = s_first + blockIdx.x; r < ri.mloc; r += gridDim.x) {
    const Row cur = row;
    row = extents(r + gridDim.x);
    if (cur.off >= c1) break;
    const int p0 = cur.p0, n = cur.n, cmn = cur.cmn, cmx = cur.cmx;
    if (!grad_row_staged(n, cmn, cmx, cap, wlog)) continue;
    const int base = cmn & ~31;
    const int a0 = cur.a0, a1 = cur.a1;
    // the first of C's entries, in flight while the nonzeros are read
    constexpr int F = 4;
    int sc[F];
    T sd[F];
#pragma unroll
    for (int u = 0; u < F; ++u) {
      const int p = tid + u * NT;
      sc[u] = 0;
      sd[u] = T(0);
      if (p < n) {
        sc[u] = c_ci[p0 + p] - base;
        sd[u] = dc[p0 + p];
      }
    }
    // this lane group's nonzeros of a round: e0 + s * (NW * GPW).  The first
    // round's are read before C's row is staged, both in flight together
    int b0[S], len[S], at[S];  // at: position in the buffer, -1 outside the chunk
    auto fetch = [&](int e0) {
      int k[S];
#pragma unroll
      for (int s = 0; s < S; ++s) {
        const int e = e0 + s * (NW * GPW);
        b0[s] = len[s] = 0;
        at[s] = -1;
        k[s] = -1;
        if (e < a1) {
          const long long po = p_off[e];
          k[s] = A.ci[e];
          if (po >= c0 && po < c1) at[s] = buf ? (int)(po - c0) : 0;  // without dB the chunk is every product
        }
      }
#pragma unroll
      for (int s = 0; s < S; ++s)
        if (at[s] >= 0) {
          b0[s] = B.rp[k[s]];
          len[s] = B.rp[k[s] + 1] - b0[s];
        }
    };
    fetch(a0 + warp * GPW + g);
    // stages C's entry p (column c); the first entry of a bitmap word leaves
    // the word's rank.  A column's predecessor is the lane below's.
    auto stage = [&](int p, int c, T v) {
      int before = __shfl_up_sync(FULL, c, 1);
      if (p < n) {
        if (lane == 0) before = p > 0 ? c_ci[p0 + p - 1] - base : -32;
        sdc[p] = v;
        if ((unsigned)c < (1u << wlog)) {
          atomicOr(&bits[c >> 5], 1u << (c & 31));
          if ((before >> 5) != (c >> 5)) pre[c >> 5] = (uint16_t)p;
        }
      }
    };
#pragma unroll
    for (int u = 0; u < F; ++u)
      if (u * NT < n) stage(tid + u * NT, sc[u], sd[u]);  // block-uniform
    for (int q = F * NT; q < n; q += NT) {
      const int p = q + tid;
      stage(p, p < n ? c_ci[p0 + p] - base : 0, p < n ? dc[p0 + p] : T(0));
    }
    // the next row's part of C, a line per thread
    for (int t = tid; t * 32 < row.n; t += NT)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(c_ci + row.p0 + t * 32));
    for (int t = tid; t * (int)(128 / sizeof(T)) < row.n; t += NT)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(dc + row.p0 + t * (int)(128 / sizeof(T))));
    __syncthreads();
    for (int e0 = a0 + warp * GPW + g; e0 - g < a1; e0 += S * NW * GPW) {  // warp-uniform
      if (e0 - g - warp * GPW != a0) fetch(e0);
      T part[S];
#pragma unroll
      for (int s = 0; s < S; ++s) part[s] = T(0);
      int most = 0;
#pragma unroll
      for (int s = 0; s < S; ++s) most = max(most, len[s]);
      for (int l = gl; l < most; l += G) {
        int col[S];
        T b[S];
#pragma unroll
        for (int s = 0; s < S; ++s) {
          col[s] = 0;
          b[s] = T(0);
          if (l < len[s]) {
            col[s] = B.ci[b0[s] + l];
            b[s] = bv[b0[s] + l];
          }
        }
#pragma unroll
        for (int s = 0; s < S; ++s) {
          if (l < len[s]) {
            const int j = col[s] - base;
            const unsigned m = 1u << (j & 31);
            T d = T(0);
            const uint32_t word = (unsigned)j < (1u << wlog) ? bits[j >> 5] : 0u;
            if (word & m) d = sdc[pre[j >> 5] + __popc(word & (m - 1u))];
            else atomicOr(err, EB_INTERNAL);  // C's pattern holds every product
            part[s] = fma(d, b[s], part[s]);
            if (buf) buf[at[s] + l] = d;
          }
        }
      }
      if (da) {
        // fold 8 sums per lane into one: lane bits LG-1, LG-2, LG-3 choose the
        // nonzero, then the remaining lanes add up
#pragma unroll
        for (int h = S / 2, d = G / 2; h >= 1; h >>= 1, d >>= 1) {
          const bool up = (gl & d) != 0;
#pragma unroll
          for (int x = 0; x < h; ++x) {
            const T send = up ? part[x] : part[x + h];
            const T keep = up ? part[x + h] : part[x];
            part[x] = keep + __shfl_xor_sync(FULL, send, d);
          }
        }
#pragma unroll
        for (int d = G / 16; d >= 1; d >>= 1) part[0] += __shfl_xor_sync(FULL, part[0], d);
        const int s = gl >> (LG - 3);
        int mine = -1;
#pragma unroll
        for (int x = 0; x < S; ++x)
          if (x == s) mine = at[x];
        if (mine >= 0 && (gl & ((1 << (LG - 3)) - 1)) == 0) da[e0 + s * (NW * GPW)] = part[0];
      }
    }
    __syncthreads();
    const int nwords = ((cmx - base) >> 5) + 1;
    for (int t = tid * 4; t < nwords; t += NT * 4) *reinterpret_cast<uint4*>(bits + t) = make_uint4(0, 0, 0, 0);
    __syncthreads();
  }
}

// The other rows: slabs of 32 nonzeros of A, dC(i,j) by a binary search in
// C's row in global memory.
template <typename T>
__global__ void __launch_bounds__(256)
k_grad_slabs(Csr A, Csr B, const T* __restrict__ bv, RowInfo ri, const int32_t* __restrict__ a_row,
             const long long* __restrict__ p_off, const int32_t* __restrict__ c_rp, const int32_t* __restrict__ c_ci,
             const T* __restrict__ dc, T* __restrict__ da, T* __restrict__ buf, long long c0, long long c1, int cap,
             int wlog, uint32_t* err) {
  __shared__ long long s_lo, s_hi;
  if (threadIdx.x < 32) {
    const long long lo = A.rp[ri.row_begin], hi = A.rp[ri.row_begin + ri.mloc];
    const long long f = c0 <= 0 ? lo : warp_first_at_least(p_off, lo, hi, c0);
    const long long l = c1 >= LLONG_MAX - 1 ? hi : warp_first_at_least(p_off, lo, hi, c1);
    if (threadIdx.x == 0) {
      s_lo = f;
      s_hi = l;
    }
  }
  __syncthreads();
  const int lane = lane_id();
  const long long e_lo = s_lo, e_hi = s_hi;
  const long long nslab = (e_hi - e_lo + 31) >> 5;
  const long long w0 = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nw = (gridDim.x * (long long)blockDim.x) >> 5;
  for (long long s = w0; s < nslab; s += nw) {
    const long long e = e_lo + (s << 5) + lane;
    bool have = e < e_hi;
    int b0 = 0, b1 = 0, p0 = 0, p1 = 0;
    long long at = 0;
    if (have) {
      const long long r = (long long)a_row[e] - ri.row_begin;
      p0 = c_rp[r];
      p1 = c_rp[r + 1];
      have = !grad_row_staged(p1 - p0, ri.cmin[r], ri.cmax[r], cap, wlog);
      if (have) {
        const int k = A.ci[e];
        b0 = B.rp[k];
        b1 = B.rp[k + 1];
        at = p_off[e] - c0;
      }
    }
    if (!__any_sync(FULL, have)) continue;
    const bool wide = have && b1 - b0 > GRAD_LANE_MAX;
    T acc = T(0);
    if (have && !wide) {
      int lo = p0;
      for (int q = b0; q < b1; ++q) {
        const int j = B.ci[q];
        const int pos = find_col(c_ci, lo, p1, j);
        T d = T(0);
        if (pos < p1 && c_ci[pos] == j) {
          d = dc[pos];
          lo = pos + 1;
        } else {
          atomicOr(err, EB_INTERNAL);
        }
        acc = fma(d, bv[q], acc);
        if (buf) buf[at + (q - b0)] = d;
      }
    }
    unsigned wm = __ballot_sync(FULL, wide);
    while (wm) {
      const int L = __ffs(wm) - 1;
      wm &= wm - 1;
      const int lb0 = __shfl_sync(FULL, b0, L), lb1 = __shfl_sync(FULL, b1, L);
      const int lp0 = __shfl_sync(FULL, p0, L), lp1 = __shfl_sync(FULL, p1, L);
      const long long lat = __shfl_sync(FULL, at, L);
      T part = T(0);
      for (int q = lb0 + lane; q < lb1; q += 32) {
        const int j = B.ci[q];
        const int pos = find_col(c_ci, lp0, lp1, j);
        T d = T(0);
        if (pos < lp1 && c_ci[pos] == j) d = dc[pos];
        else atomicOr(err, EB_INTERNAL);
        part = fma(d, bv[q], part);
        if (buf) buf[lat + (q - lb0)] = d;
      }
      const T tot = warp_sum_fixed(part);
      if (lane == L) acc = tot;
    }
    if (have && da) da[e] = acc;
  }
}

// dB from one chunk of the buffer, in the order that k_grad_b sums in: slabs of
// 32 outputs of B per warp, an output of at most GRAD_LANE_MAX terms (of the
// whole column of A, not of the chunk) its lane's chain over the chunk's
// nonzeros of A^T(k,:), which the next chunk takes up from dB (lanes of one row
// of B read consecutive buffer entries).  Longer sums are 32 chains and a fixed
// tree; their chains cannot be taken up from one number, so they are summed here
// only when one chunk holds every product (LONG; a kernel of its own, because
// its registers leave fewer warps), by the whole block: warp w runs the chains
// w, w + 8, w + 16 and w + 24 of the slab's 32 outputs, each lane an output.
// (FP32, positive terms, root mean square error over the sum: 512 terms 3.0e-7
// in one chain, 4.5e-8 in 32.)
template <typename T>
__device__ __forceinline__ T grad_col_sum(const T* __restrict__ av, const int32_t* __restrict__ t_src,
                                          const long long* __restrict__ t_off, const T* __restrict__ buf,
                                          long long c0, int l, int t0, int t1, T acc) {
  int t = t0;
  for (; t + 4 <= t1; t += 4) {
    T a[4], d[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      a[u] = av[t_src[t + u]];
      d[u] = buf[t_off[t + u] - c0 + l];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) acc = fma(a[u], d[u], acc);
  }
  for (; t < t1; ++t) acc = fma(av[t_src[t]], buf[t_off[t] - c0 + l], acc);
  return acc;
}

// Chains w, w + 8, w + 16, w + 24 of the 32 over the terms [t0, t1), added as
// warp_sum_fixed adds their lanes (16 apart, then 8 apart).  Rows outside the
// plan's range (offsets -1 and LLONG_MAX) keep their place and add nothing.
template <typename T>
__device__ __forceinline__ T grad_wide_part(const T* __restrict__ av, const int32_t* __restrict__ t_src,
                                            const long long* __restrict__ t_off, const T* __restrict__ buf, int l,
                                            int t0, int t1, int w) {
  T p[4] = {T(0), T(0), T(0), T(0)};
  for (int t = t0 + w; t < t1; t += 32) {
    T a[4], d[4];
    bool in[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int x = t + 8 * u;
      const long long o = x < t1 ? t_off[x] : -1ll;
      in[u] = o >= 0 && o < LLONG_MAX;
      a[u] = in[u] ? av[t_src[x]] : T(0);
      d[u] = in[u] ? buf[o + l] : T(0);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (in[u]) p[u] = fma(a[u], d[u], p[u]);
  }
  return (p[0] + p[2]) + (p[1] + p[3]);
}

template <typename T, bool LONG>
__global__ void __launch_bounds__(256)
k_grad_cols(Csr B, const T* __restrict__ av, const int32_t* __restrict__ b_row, const int32_t* __restrict__ t_rp,
            const int32_t* __restrict__ t_src, const long long* __restrict__ t_off, const T* __restrict__ buf,
            T* __restrict__ db, long long c0, long long c1, int first, int whole) {
  const int warp = threadIdx.x >> 5, lane = lane_id();
  const long long nslab = (B.nnz + 31) >> 5;
  for (long long s0 = blockIdx.x * 8ll; s0 < nslab; s0 += gridDim.x * 8ll) {
    const long long q = ((s0 + warp) << 5) + lane;
    const bool have = q < B.nnz;
    int l = 0, t0 = 0, t1 = 0;
    if (have) {
      const int k = b_row[q];
      l = (int)(q - B.rp[k]);
      t0 = t_rp[k];
      t1 = t_rp[k + 1];
    }
    const bool wide = LONG && t1 - t0 > GRAD_LANE_MAX;
    if (have && !wide) {
      int u0 = t0, u1 = t1;
      if (!whole) {  // one chunk of every row of A needs no search
        u0 = first_at_least(t_off, t0, t1, c0);
        u1 = first_at_least(t_off, u0, t1, c1);
      }
      if (first || u1 > u0) db[q] = grad_col_sum(av, t_src, t_off, buf, c0, l, u0, u1, first ? T(0) : db[q]);
    }
    if constexpr (LONG) {
      __shared__ int s_any[8];
      __shared__ int s_l[32], s_t0[32], s_t1[32];
      __shared__ T s_part[8][32];
      const bool any = __any_sync(FULL, wide);
      if (lane == 0) s_any[warp] = any;
      if (!__syncthreads_or(any)) continue;
      for (int w = 0; w < 8; ++w) {
        if (!s_any[w]) continue;  // block-uniform
        if (warp == w) {
          s_l[lane] = l;
          s_t0[lane] = wide ? t0 : 0;
          s_t1[lane] = wide ? t1 : 0;
        }
        __syncthreads();
        s_part[warp][lane] = grad_wide_part(av, t_src, t_off, buf, s_l[lane], s_t0[lane], s_t1[lane], warp);
        __syncthreads();
        if (warp == w && wide)  // 4, 2 and 1 apart
          db[q] = ((s_part[0][lane] + s_part[4][lane]) + (s_part[2][lane] + s_part[6][lane])) +
                  ((s_part[1][lane] + s_part[5][lane]) + (s_part[3][lane] + s_part[7][lane]));
        __syncthreads();
      }
      __syncthreads();
    }
  }
}

static int grid_for(long long slabs, int nsm) {
  long long g = (slabs + 7) / 8;  // 8 warps (slabs in flight) per block
  const long long cap = (long long)nsm * 8;
  if (g > cap) g = cap;
  return (int)(g < 1 ? 1 : g);
}

cudaError_t launch_row_index(const LaunchCtx& c, const int32_t* rp, long long nrows, int32_t* out) {
  if (nrows <= 0) return cudaSuccess;
  k_row_index<<<grid_for(nrows / 8 + 1, c.nsm), 256, 0, c.stream>>>(rp, nrows, out);
  count_launch(c);
  return cudaGetLastError();
}

long long grad_buffer_entries(long long nnz_a, long long nnz_b, long long ncols_b, int vbytes) {
  const long long chunk = GRAD_BUFFER_BYTES / vbytes;
  const long long longest = ncols_b < nnz_b ? ncols_b : nnz_b;  // no row of B is longer
  if (longest > chunk || nnz_a <= 0 || longest <= 0) return 0;
  // a chunk's last nonzero may start just inside it
  const long long all = nnz_a < chunk / longest ? nnz_a * longest : chunk;
  return (all < chunk ? all : chunk) + longest;
}

cudaError_t launch_grad_offsets(const LaunchCtx& c, const Csr& A, const Csr& B, long long row_begin, long long mloc,
                                const long long* prod, const int32_t* t_rp, const int32_t* t_ci, const int32_t* t_src,
                                long long* row_off, long long* part, long long* p_off, long long* t_off) {
  if (mloc <= 0) return cudaSuccess;
  const long long tiles = (mloc + OFF_TILE - 1) / OFF_TILE;
  k_off_tiles<<<(unsigned)tiles, OFF_THREADS, 0, c.stream>>>(prod, mloc, part);
  k_off_partials<<<1, OFF_THREADS, 0, c.stream>>>(part, tiles);
  k_off_down<<<(unsigned)tiles, OFF_THREADS, 0, c.stream>>>(prod, mloc, part, row_off);
  k_product_offsets<<<grid_for(mloc, c.nsm), 256, 0, c.stream>>>(A, B, row_begin, mloc, row_off, p_off, c.st);
  k_transposed_offsets<<<grid_for((A.nnz + 31) / 32, c.nsm), 256, 0, c.stream>>>(
      A.nnz, t_ci, t_src, row_begin, row_begin + mloc, p_off, t_off, t_rp, B.rp, B.nrows, c.st);
  for (int i = 0; i < 5; ++i) count_launch(c);
  return cudaGetLastError();
}

template <int NT, int G, typename T>
static cudaError_t grad_rows(const LaunchCtx& c, const GradArgs& g, const T* bv, const T* dc, T* da, T* buf,
                             long long c0, long long c1, int cap, int wlog, long long rows) {
  auto k = k_grad_rows<NT, G, T>;
  const size_t smem = (size_t)cap * sizeof(T) + ((size_t)1 << wlog) / 32 * 6;
  const int occ = kernel_blocks_per_sm(k, NT, smem);
  if (occ <= 0) return cudaErrorInvalidConfiguration;
  k<<<persistent_grid(rows, 1, c.nsm, occ), NT, smem, c.stream>>>(g.A, g.B, bv, g.ri, g.row_off, g.p_off, g.c_rp,
                                                                 g.c_ci, dc, da, buf, c0, c1, cap, wlog, c.err);
  count_launch(c);
  return cudaGetLastError();
}

// dB with a search in C's rows per term.
template <typename T>
static cudaError_t search_db(const LaunchCtx& c, const GradArgs& g, const T* av, const T* dc, T* db) {
  k_grad_b<T><<<grid_for((g.B.nnz + 31) / 32, c.nsm), 256, 0, c.stream>>>(
      g.B, av, g.b_row, g.t_rp, g.t_ci, g.t_src, g.ri.row_begin, g.ri.row_begin + g.ri.mloc, g.c_rp, g.c_ci, dc, db,
      c.err);
  count_launch(c);
  return cudaGetLastError();
}

// dA with a search in C's rows per term.
template <typename T>
static cudaError_t search_da(const LaunchCtx& c, const GradArgs& g, const T* bv, const T* dc, T* da) {
  k_grad_a<T><<<grid_for(g.A.nnz / 32 + 1, c.nsm), 256, 0, c.stream>>>(  // (the kernel reads the range's own extent)
      g.A, g.B, bv, g.ri.row_begin, g.ri.mloc, g.a_row, g.c_rp, g.c_ci, dc, da, c.err);
  count_launch(c);
  return cudaGetLastError();
}

// How a plan's gradients are formed.
struct GradRoute {
  bool staged;    // rows of C of more than 128 entries in shared memory (k_grad_rows)
  bool buffered;  // dB through the product buffer
  int cap, wlog;  // entries and column bits that k_grad_rows stages
  int lanes;      // per nonzero of A
  long long rows, chunk;
};

// Staged rows pay where rows of C fit (more than half of the rows can have
// more than 128 entries, and a bitmap holds every column), where a row has
// enough products to carry its barriers (10,007 columns, k a row, dA alone, FP64:
// k = 20, 400 products, 75 us staged and 66 with searches; k = 24, 84 and 89;
// FP32: k = 18 58 and 50, k = 20 59 and 61) and where rows of B are alike: a
// group of lanes walks the longest of eight rows of B, so that on power-law
// graphs, whose products come from rows of B many times the average (weighted
// by their use 22 times on an R-MAT of 32,768 columns), most lanes wait: dA there
// 4.49 ms staged, 1.57 with searches.  At most 4 times the average, 8 with 32
// lanes (R-MAT of 2,000 vertices, edge factor 32: 0.25 and 0.40; of 9,000: 1.89
// and 1.16).  A row of B of more than 128 entries is summed by 32 lanes, or not
// here.  The choice depends on the plan alone: dA has the same bits with dB and
// without.  Where most rows stay inside half of B's columns, searches meet each
// other's cache lines and cost a fifth (6 ps a term instead of 30), and neither
// staging nor more than one chunk pays: 27-point stencil on 40^3 points, FP64,
// both gradients 0.96 ms and 0.52 with searches, blocks of 64 (20,032 rows) 2.20
// and 1.06, a band of 41 entries (20,000 rows) 0.63 and 0.35.
//
// Through the buffer dB shares dA's searches, or staged rows' look-ups.  Alone
// and without either a search per term is no more work (40^3 stencil, FP64: 37 us
// against 51; with dA 61 against 56), unless columns of A are long, whose terms
// one warp would search (R-MAT, 3,000 columns: 1.18 ms against 0.33).  More than
// one chunk: every chunk passes over all of dB, so what counts is the terms of an
// output in a chunk and the steps that the search of each would take.  With dA,
// buffered against searched, terms x steps: 5 (96^3 stencil FP64) 1.06 ms and
// 0.44, 11 (FP32) 0.48 and 0.41, 13 (200,000 columns, 16 to 48 a row, FP64) 13.0
// and 11.1, 16 (300,000 columns, 2 to 10, FP64) 0.28 and 0.35, 25 (200,000 columns
// in FP32) 6.7 and 9.9, 40 (65,536 columns, 32, FP64) 1.2 and 3.0.  Long sums do
// not go on from chunk to chunk (k_grad_cols).  A captured call stays off the
// buffer: nothing orders its replays against the plan's other calls.  Whichever
// way, dB's sums have the same order and bits.
template <typename T>
static GradRoute grad_route(const GradArgs& g, bool da, bool db) {
  GradRoute r{};
  // none: rows of B longer than one, and then no product offsets either
  const bool has_buffer = g.buf_entries > 0 && g.B.nnz > 0;
  int hi = 0;
  long long all = 0;
  for (int b = 1; b < NBINS; ++b) {
    all += g.hist[b];
    if (b >= bin_of(GRAD_ROW_MIN + 1) && g.hist[b]) {
      hi = b;
      r.rows += g.hist[b];
    }
  }
  // a row has at most its products' entries, so the rows' bins bound them
  r.cap = 256;
  while (r.cap < GRAD_ROW_CAP && r.cap < (hi > 0 ? (hi < 14 ? 1 << (hi - 1) : GRAD_ROW_CAP) : 0)) r.cap *= 2;
  r.wlog = 10;
  const int widest = r.cap > 2048 ? 18 : 17;
  while (r.wlog < widest && (1ll << r.wlog) < g.B.ncols) ++r.wlog;
  const double avg = g.B.nrows > 0 ? (double)g.B.nnz / (double)g.B.nrows : 0.0;
  r.lanes = avg >= 20 ? 32 : (avg >= 10 ? 16 : 8);
  const bool local = 2 * g.rows_local > r.rows;
  const double share = g.A.nrows > 0 ? (double)g.ri.mloc / (double)g.A.nrows : 0.0;  // of A's nonzeros, about
  const double alike = (r.lanes == 32 ? 8.0 : 4.0) * avg * share * (double)g.A.nnz;
  r.staged = has_buffer && !local && 2 * r.rows > all && g.total >= (sizeof(T) == 8 ? 512 : 384) * all &&
             (1ll << r.wlog) >= g.B.ncols && (double)g.total <= alike &&
             (r.lanes == 32 || g.max_row_b <= GRAD_LANE_MAX);
  const long long longest = g.B.ncols < g.B.nnz ? g.B.ncols : g.B.nnz;
  r.chunk = g.buf_entries - longest;
  r.buffered = db && has_buffer && !g.captured && (da || r.staged || g.max_col > GRAD_LANE_MAX);
  if (r.buffered && g.total > r.chunk) {
    const double chunks = (double)((g.total + r.chunk - 1) / r.chunk);
    const double terms = (double)g.total / (chunks * (double)g.B.nnz);
    const double steps = log2(1.0 + (double)g.nnz_c / (double)(all > 0 ? all : 1));
    r.buffered = g.max_col <= GRAD_LANE_MAX && !local && terms * steps >= 15.0;
  }
  return r;
}

template <typename T>
static cudaError_t backward_t(const LaunchCtx& c, const GradArgs& g, const T* av, const T* bv, const T* dc, T* da,
                              T* db) {
  const GradRoute r = grad_route<T>(g, da != nullptr, db != nullptr);
  if (db && g.B.nnz > 0 && !r.buffered) {
    const cudaError_t e = search_db(c, g, av, dc, db);
    if (e != cudaSuccess) return e;
  }
  if (!r.buffered) db = nullptr;
  if (!da && !db) return cudaSuccess;
  if (!db && !r.staged) return search_da(c, g, bv, dc, da);
  const long long chunk = db ? r.chunk : LLONG_MAX;
  T* const buf = db ? (T*)g.buf : nullptr;
  const int cap = r.staged ? r.cap : 0;
  for (long long c0 = 0; c0 < g.total || c0 == 0; c0 += chunk) {
    const bool last = c0 + chunk >= g.total || chunk == LLONG_MAX;
    const long long c1 = last ? LLONG_MAX - 1 : c0 + chunk;
    cudaError_t e = cudaSuccess;
    if (r.staged) {
#define SG_GRAD_ROWS(GG)                                                                                    \
  e = cap > 2048 ? grad_rows<256, GG, T>(c, g, bv, dc, da, buf, c0, c1, cap, r.wlog, r.rows)                 \
                 : grad_rows<128, GG, T>(c, g, bv, dc, da, buf, c0, c1, cap, r.wlog, r.rows)
      if (r.lanes == 32) SG_GRAD_ROWS(32);
      else if (r.lanes == 16) SG_GRAD_ROWS(16);
      else SG_GRAD_ROWS(8);
#undef SG_GRAD_ROWS
      if (e != cudaSuccess) return e;
    }
    k_grad_slabs<T><<<grid_for(g.A.nnz / 32 + 1, c.nsm), 256, 0, c.stream>>>(
        g.A, g.B, bv, g.ri, g.a_row, g.p_off, g.c_rp, g.c_ci, dc, da, buf, c0, c1, cap, r.wlog, c.err);
    count_launch(c);
    if (db) {
      auto k = g.max_col > GRAD_LANE_MAX ? k_grad_cols<T, true> : k_grad_cols<T, false>;
      k<<<grid_for((g.B.nnz + 31) / 32, c.nsm), 256, 0, c.stream>>>(
          g.B, av, g.b_row, g.t_rp, g.t_src, g.t_off, buf, db, c0, c1, c0 == 0 ? 1 : 0,
          c0 == 0 && last && g.ri.row_begin == 0 && g.ri.mloc == g.A.nrows ? 1 : 0);
      count_launch(c);
    }
    if ((e = cudaGetLastError()) != cudaSuccess || last) return e;
  }
  return cudaSuccess;
}

bool grad_uses_buffer(int dtype, const GradArgs& g, bool da, bool db) {
  return (dtype == SPGEMM_F32 ? grad_route<float>(g, da, db) : grad_route<double>(g, da, db)).buffered;
}

cudaError_t launch_backward(const LaunchCtx& c, int dtype, const GradArgs& g, const void* av, const void* bv,
                            const void* dc, void* da, void* db) {
  if (dtype == SPGEMM_F32)
    return backward_t<float>(c, g, (const float*)av, (const float*)bv, (const float*)dc, (float*)da, (float*)db);
  return backward_t<double>(c, g, (const double*)av, (const double*)bv, (const double*)dc, (double*)da, (double*)db);
}

}  // namespace sg
