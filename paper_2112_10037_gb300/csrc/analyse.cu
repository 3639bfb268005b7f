// Structure analysis: input validation, per-row product counts and column
// spans, and the counting sort of rows into bins by product count.
//
// The product count of row i is P_i = sum over the nonzeros A(i,k) of
// nnz(B(k,:)) -- the number of scalar-times-row products the row-wise
// Gustavson method (Sec. 2.2) forms for that row (the per-nonzero
// B_NUM_VEC of Table 1, summed).  Rows are later dispatched by P_i.
#include "internal.cuh"

namespace sg {

// One warp per row: column indices inside [0, ncols), strictly ascending;
// row_ptr non-decreasing and ending at nnz.
__global__ void k_validate(Csr M, uint32_t* err) {
  const int lane = lane_id();
  const long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nw = (gridDim.x * (long long)blockDim.x) >> 5;
  bool bad = false;
  if (w == 0 && lane == 0) {
    if (M.rp[0] != 0 || (long long)M.rp[M.nrows] != M.nnz) bad = true;
  }
  for (long long i = w; i < M.nrows; i += nw) {
    const int a0 = M.rp[i], a1 = M.rp[i + 1];
    if (a1 < a0 || a0 < 0 || (long long)a1 > M.nnz) { bad = true; continue; }
    for (int e = a0 + lane; e < a1; e += 32) {
      const int c = M.ci[e];
      if (c < 0 || (long long)c >= M.ncols) bad = true;
      if (e > a0 && M.ci[e - 1] >= c) bad = true;
    }
  }
  if (__any_sync(FULL, bad) && lane == 0) atomicOr(err, EB_UNSORTED);
}

// Sum, minimum and maximum over aligned groups of G lanes (every lane of the
// warp calls them; G = 32 uses the single-instruction warp reductions).
template <int G, typename V>
__device__ __forceinline__ V group_sum(V v) {
  if constexpr (G == 32) {
    return warp_sum(v);
  } else {
#pragma unroll
    for (int d = G / 2; d >= 1; d >>= 1) v += __shfl_xor_sync(FULL, v, d);
    return v;
  }
}
template <int G>
__device__ __forceinline__ int group_min(int v) {
  if constexpr (G == 32) {
    return warp_min(v);
  } else {
#pragma unroll
    for (int d = G / 2; d >= 1; d >>= 1) v = min(v, __shfl_xor_sync(FULL, v, d));
    return v;
  }
}
template <int G>
__device__ __forceinline__ int group_max(int v) {
  if constexpr (G == 32) {
    return warp_max(v);
  } else {
#pragma unroll
    for (int d = G / 2; d >= 1; d >>= 1) v = max(v, __shfl_xor_sync(FULL, v, d));
    return v;
  }
}

// This lane's share of the row of A at [a0, a1), a warp walking it: products,
// smallest and largest column reached.  Four entries per lane per step, their
// dependent loads in flight together (long rows of power-law matrices
// otherwise form the tail).
__device__ __forceinline__ void analyse_walk(const Csr& A, const Csr& B, int a0, int a1, long long* p, int* mn,
                                             int* mx, bool* bad) {
  for (int e0 = a0 + lane_id(); e0 < a1; e0 += 128) {
    int kk[4], ss[4], tt[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) kk[u] = e0 + 32 * u < a1 ? A.ci[e0 + 32 * u] : -1;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      ss[u] = tt[u] = 0;
      if (e0 + 32 * u < a1) {
        if (kk[u] < 0 || (long long)kk[u] >= B.nrows) {
          *bad = true;
        } else {
          ss[u] = B.rp[kk[u]];
          tt[u] = B.rp[kk[u] + 1];
        }
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (tt[u] > ss[u]) {
        *p += tt[u] - ss[u];
        *mn = min(*mn, B.ci[ss[u]]);
        *mx = max(*mx, B.ci[tt[u] - 1]);
      }
    }
  }
}

// Whether a row forms so many products on few columns that a warp with dense
// 1024-column windows sums it sooner than the paths that rank the columns (when
// such rows are many, see window_rows in api.cu): windows need neither marks
// nor ranks nor, for one row of B at a time, atomics, but a row walks every
// window of its span.  Up to 4096 products (block registers instead) four
// products per column of the span, or one window while the registers are half
// empty; above (bands instead) 256 per window.
__device__ __forceinline__ bool row_is_dense(long long p, int mn, int mx, bool count) {
  if (!count || p <= 128) return false;
  const int windows = (mx >> 10) - (mn >> 10) + 1;
  if (p > 4096) return p >= 256ll * windows;
  return p >= 4ll * (mx - mn + 1) || (p <= 256 && windows == 1);
}

// Rows that stay inside half of B's columns (bands, stencils, finite elements):
// neighbouring rows of C then share cache lines and searches in them are cheap
// (see grad_route in backward.cu).
__device__ __forceinline__ bool row_is_local(long long p, int mn, int mx, long long ncols) {
  return p > 128 && 2 * ((long long)mx - mn + 1) <= ncols;
}

// One warp per row of A: P_i, the smallest and largest column any product of
// the row reaches (first and last column of each touched B row, since B's rows
// are sorted), histogram of bins, total and maximum P.
__global__ void __launch_bounds__(256) k_analyse(Csr A, Csr B, long long row_begin, long long mloc,
                                                 long long* __restrict__ prod, int* __restrict__ cmin,
                                                 int* __restrict__ cmax, DevStats* st, bool count_dense) {
  __shared__ int s_hist[NBINS];
  __shared__ unsigned long long s_total, s_max;
  __shared__ unsigned s_wide, s_wide8, s_dense, s_local;
  if (threadIdx.x < NBINS) s_hist[threadIdx.x] = 0;
  if (threadIdx.x == 0) { s_total = 0; s_max = 0; s_wide = 0; s_wide8 = 0; s_dense = 0; s_local = 0; }
  if (block_skip(st)) return;  // validated input was rejected
  const int lane = lane_id(), gl = lane;
  const long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nw = (gridDim.x * (long long)blockDim.x) >> 5;
  unsigned long long my_total = 0, my_max = 0;
  unsigned my_wide = 0, my_wide8 = 0, my_dense = 0, my_local = 0;
  bool bad = false;
  for (long long r = w; r < mloc; r += nw) {
    const int a0 = A.rp[row_begin + r], a1 = A.rp[row_begin + r + 1];
    long long p = 0;
    int mn = INT_MAX, mx = -1;
    analyse_walk(A, B, a0, a1, &p, &mn, &mx, &bad);
    p = warp_sum(p);
    mn = warp_min(mn);
    mx = warp_max(mx);
    if (lane == 0) {
      my_wide += a1 - a0 > 32 ? 1u : 0u;
      my_wide8 += a1 - a0 > 8 ? 1u : 0u;
      my_dense += row_is_dense(p, mn, mx, count_dense) ? 1u : 0u;
      my_local += row_is_local(p, mn, mx, B.ncols) ? 1u : 0u;
      prod[r] = p;
      cmin[r] = mn;
      cmax[r] = mx;
      atomicAdd(&s_hist[bin_of(p)], 1);
      my_total += (unsigned long long)p;
      my_max = my_max > (unsigned long long)p ? my_max : (unsigned long long)p;
    }
  }
  if (gl == 0 && my_total) {
    atomicAdd(&s_total, my_total);
    atomicMax(&s_max, my_max);
  }
  if (gl == 0 && my_wide) atomicAdd(&s_wide, my_wide);
  if (gl == 0 && my_wide8) atomicAdd(&s_wide8, my_wide8);
  if (gl == 0 && my_dense) atomicAdd(&s_dense, my_dense);
  if (gl == 0 && my_local) atomicAdd(&s_local, my_local);
  if (__any_sync(FULL, bad) && lane == 0) atomicOr(&st->err, EB_UNSORTED);
  __syncthreads();
  if (threadIdx.x < NBINS && s_hist[threadIdx.x]) atomicAdd(&st->hist[threadIdx.x], s_hist[threadIdx.x]);
  if (threadIdx.x == 0 && s_total) {
    atomicAdd(&st->total_products, s_total);
    atomicMax(&st->max_products, s_max);
  }
  if (threadIdx.x == 0 && s_wide) atomicAdd(&st->rows_wide, s_wide);
  if (threadIdx.x == 0 && s_wide8) atomicAdd(&st->rows_wide8, s_wide8);
  if (threadIdx.x == 0 && s_dense) atomicAdd(&st->rows_dense, s_dense);
  if (threadIdx.x == 0 && s_local) atomicAdd(&st->rows_local, s_local);
}

// The same for matrices of short rows (stencils, aggregation operators): 8
// lanes per row, four rows per group in flight, so that the chain of dependent
// loads (row pointer, column, row pointer of B) is paid once per 16 rows of a
// warp; rows of more than 32 nonzeros are walked by the warp.  Column spans are read in a second walk and only for rows of more than
// span_min products (the paths of smaller rows never use them).  96^3 stencil
// squared: 76 us with one row per group and every row's span, 40 us here.
__global__ void __launch_bounds__(256) k_analyse_short(Csr A, Csr B, long long row_begin, long long mloc,
                                                       long long* __restrict__ prod, int* __restrict__ cmin,
                                                       int* __restrict__ cmax, DevStats* st, long long span_min,
                                                       bool count_dense) {
  constexpr int G = 8, RPW = 32 / G, U = 4;
  __shared__ int s_hist[NBINS];
  __shared__ unsigned long long s_total, s_max;
  __shared__ unsigned s_wide, s_wide8, s_dense, s_local;
  if (threadIdx.x < NBINS) s_hist[threadIdx.x] = 0;
  if (threadIdx.x == 0) { s_total = 0; s_max = 0; s_wide = 0; s_wide8 = 0; s_dense = 0; s_local = 0; }
  if (block_skip(st)) return;  // validated input was rejected
  const int lane = lane_id();
  const int gl = lane & (G - 1), g = lane / G;
  const long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nw = (gridDim.x * (long long)blockDim.x) >> 5;
  unsigned long long my_total = 0, my_max = 0;
  unsigned my_wide = 0, my_wide8 = 0, my_dense = 0, my_local = 0;
  bool bad = false;
  for (long long r0 = w * RPW * U; r0 < mloc; r0 += nw * RPW * U) {
    int a0[U], a1[U], k[U];
    long long p[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long r = r0 + u * RPW + g;
      a0[u] = a1[u] = 0;
      if (r < mloc) {
        a0[u] = A.rp[row_begin + r];
        a1[u] = A.rp[row_begin + r + 1];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) k[u] = (a0[u] + gl < a1[u] && a1[u] - a0[u] <= 32) ? A.ci[a0[u] + gl] : -1;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      p[u] = 0;
      if (a0[u] + gl < a1[u] && a1[u] - a0[u] <= 32) {
        if (k[u] < 0 || (long long)k[u] >= B.nrows) bad = true;
        else p[u] = B.rp[k[u] + 1] - B.rp[k[u]];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool wide = a1[u] - a0[u] > 32;
      if (!wide)
        for (int e = a0[u] + G + gl; e < a1[u]; e += G) {  // rows of more than 8 nonzeros
          const int kk = A.ci[e];
          if (kk < 0 || (long long)kk >= B.nrows) bad = true;
          else p[u] += B.rp[kk + 1] - B.rp[kk];
        }
      p[u] = group_sum<G>(p[u]);
      const long long r = r0 + u * RPW + g;
      unsigned wm = __ballot_sync(FULL, wide && gl == 0);
      while (wm) {
        const int L = __ffs(wm) - 1;
        wm &= wm - 1;
        long long wp = 0;
        int mn = INT_MAX, mx = -1;
        analyse_walk(A, B, __shfl_sync(FULL, a0[u], L), __shfl_sync(FULL, a1[u], L), &wp, &mn, &mx, &bad);
        wp = warp_sum(wp);
        mn = warp_min(mn);
        mx = warp_max(mx);
        if (g == L / G) p[u] = wp;
        if (lane == L) {
          my_dense += row_is_dense(wp, mn, mx, count_dense) ? 1u : 0u;
          my_local += row_is_local(wp, mn, mx, B.ncols) ? 1u : 0u;
          cmin[r] = mn;
          cmax[r] = mx;
        }
      }
      if (__any_sync(FULL, p[u] > span_min && !wide)) {
        int mn = INT_MAX, mx = -1;
        if (p[u] > span_min && !wide)
          for (int e = a0[u] + gl; e < a1[u]; e += G) {
            const int kk = A.ci[e];
            if (kk >= 0 && (long long)kk < B.nrows) {
              const int s = B.rp[kk], t = B.rp[kk + 1];
              if (t > s) {
                mn = min(mn, B.ci[s]);
                mx = max(mx, B.ci[t - 1]);
              }
            }
          }
        mn = group_min<G>(mn);
        mx = group_max<G>(mx);
        if (gl == 0 && r < mloc && p[u] > span_min && !wide) {
          my_dense += row_is_dense(p[u], mn, mx, count_dense) ? 1u : 0u;
          my_local += row_is_local(p[u], mn, mx, B.ncols) ? 1u : 0u;
          cmin[r] = mn;
          cmax[r] = mx;
        }
      }
      if (gl == 0 && r < mloc) {
        my_wide += a1[u] - a0[u] > 32 ? 1u : 0u;
        my_wide8 += a1[u] - a0[u] > 8 ? 1u : 0u;
        prod[r] = p[u];
        atomicAdd(&s_hist[bin_of(p[u])], 1);
        my_total += (unsigned long long)p[u];
        my_max = my_max > (unsigned long long)p[u] ? my_max : (unsigned long long)p[u];
      }
    }
  }
  if (gl == 0 && my_total) {
    atomicAdd(&s_total, my_total);
    atomicMax(&s_max, my_max);
  }
  if (gl == 0 && my_wide) atomicAdd(&s_wide, my_wide);
  if (gl == 0 && my_wide8) atomicAdd(&s_wide8, my_wide8);
  if (gl == 0 && my_dense) atomicAdd(&s_dense, my_dense);
  if (gl == 0 && my_local) atomicAdd(&s_local, my_local);
  if (__any_sync(FULL, bad) && lane == 0) atomicOr(&st->err, EB_UNSORTED);
  __syncthreads();
  if (threadIdx.x < NBINS && s_hist[threadIdx.x]) atomicAdd(&st->hist[threadIdx.x], s_hist[threadIdx.x]);
  if (threadIdx.x == 0 && s_total) {
    atomicAdd(&st->total_products, s_total);
    atomicMax(&st->max_products, s_max);
  }
  if (threadIdx.x == 0 && s_wide) atomicAdd(&st->rows_wide, s_wide);
  if (threadIdx.x == 0 && s_wide8) atomicAdd(&st->rows_wide8, s_wide8);
  if (threadIdx.x == 0 && s_dense) atomicAdd(&st->rows_dense, s_dense);
  if (threadIdx.x == 0 && s_local) atomicAdd(&st->rows_local, s_local);
}

// Counting sort of the non-empty rows by bin, largest bin first.  Each block
// takes a contiguous chunk of rows: counts per bin in shared memory, reserves
// one range per bin with a single global atomic, then places its rows.
// (1024 rows: a matrix of a few thousand rows otherwise fits one block.)  Lanes
// of one bin -- in a stencil's product all of them -- count with one atomic.
constexpr int SCATTER_ROWS = 1024;

// Adds one per lane to cnt[b] (active lanes: b > 0); returns the lane's place.
__device__ __forceinline__ int bin_add(int* cnt, int b) {
  const int lane = lane_id();
  const unsigned act = __ballot_sync(FULL, b > 0);
  if (!act) return 0;
  const int b0 = __shfl_sync(FULL, b, __ffs(act) - 1);
  if (__all_sync(FULL, b == 0 || b == b0)) {
    int at = 0;
    if (lane == __ffs(act) - 1) at = atomicAdd(&cnt[b0], __popc(act));
    return __shfl_sync(FULL, at, __ffs(act) - 1) + __popc(act & lanemask_lt());
  }
  return b > 0 ? atomicAdd(&cnt[b], 1) : 0;
}

__global__ void __launch_bounds__(256) k_bin_scatter(const long long* __restrict__ prod, long long mloc,
                                                     DevStats* st, int* __restrict__ rows) {
  __shared__ int s_start[NBINS];
  __shared__ int s_cnt[NBINS];
  __shared__ int s_base[NBINS];
  if (block_skip(st)) return;
  if (threadIdx.x < NBINS) {
    int b = threadIdx.x, acc = 0;
    for (int k = NBINS - 1; k > b; --k) acc += st->hist[k];
    s_start[b] = acc;
    s_cnt[b] = 0;
  }
  __syncthreads();
  const long long r0 = (long long)blockIdx.x * SCATTER_ROWS;
  const long long r1 = min(mloc, r0 + SCATTER_ROWS);
  int bins[SCATTER_ROWS / 256];
#pragma unroll
  for (int u = 0; u < SCATTER_ROWS / 256; ++u) {
    const long long r = r0 + u * 256 + threadIdx.x;
    bins[u] = r < r1 ? bin_of(prod[r]) : 0;
  }
#pragma unroll
  for (int u = 0; u < SCATTER_ROWS / 256; ++u) bin_add(s_cnt, bins[u]);
  __syncthreads();
  if (threadIdx.x < NBINS) {
    const int b = threadIdx.x;
    s_base[b] = s_cnt[b] ? s_start[b] + atomicAdd(&st->fill[b], s_cnt[b]) : 0;
    s_cnt[b] = 0;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < SCATTER_ROWS / 256; ++u) {
    const int at = bin_add(s_cnt, bins[u]);
    if (bins[u]) rows[s_base[bins[u]] + at] = (int)(r0 + u * 256 + threadIdx.x);
  }
}

static int grid_for_warps(long long nwarps, int warps_per_block, int nsm);

// Window-run lists of B (see SplitInfo), at two window widths (shifts s1
// and s2) from one read of B: pass 1 counts the runs of each row (plus its
// sentinel), an exclusive scan turns counts into run pointers, pass 2 writes
// (window id, first position) of every run.  One warp per row; a run starts
// where the window id differs from the previous entry's.  A null second list
// is skipped.  With no row in a window bin (win_lo, see no_window_rows) the
// lists stay unbuilt.
__global__ void __launch_bounds__(256) k_runs_count(Csr B, int s1, int32_t* __restrict__ rr1, int s2,
                                                    int32_t* __restrict__ rr2, const DevStats* st, int win_lo) {
  if (block_skip(st)) return;
  if (no_window_rows(st, win_lo)) return;
  const int lane = lane_id();
  const long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nw = (gridDim.x * (long long)blockDim.x) >> 5;
  for (long long k = w; k < B.nrows; k += nw) {
    const int rs = B.rp[k], re = B.rp[k + 1];
    int n1 = 0, n2 = 0;
    for (int base = rs; base < re; base += 128) {  // 4 chunks of loads in flight per step
      int c[4], pc[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int idx = base + 32 * u + lane;
        c[u] = idx < re ? B.ci[idx] : 0;
        pc[u] = (idx < re && idx > rs) ? B.ci[idx - 1] : -1;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int idx = base + 32 * u + lane;
        const bool in = idx < re;
        const bool b1 = in && (idx == rs || (pc[u] >> s1) != (c[u] >> s1));
        const bool b2 = in && (idx == rs || (pc[u] >> s2) != (c[u] >> s2));
        n1 += __popc(__ballot_sync(FULL, b1));
        n2 += __popc(__ballot_sync(FULL, b2));
      }
    }
    if (lane == 0) {
      rr1[k] = n1 + 1;
      if (rr2) rr2[k] = n2 + 1;
    }
  }
}

__device__ __forceinline__ void runs_fill_row(const Csr& B, int k, int shift, const int32_t* __restrict__ rr,
                                              int2* __restrict__ runs) {
  const int lane = lane_id();
  const int rs = B.rp[k], re = B.rp[k + 1];
  int pos = rr[k];
  for (int base = rs; base < re; base += 128) {  // 4 chunks of loads in flight per step
    int c[4], pc[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int idx = base + 32 * u + lane;
      c[u] = idx < re ? B.ci[idx] : 0;
      pc[u] = (idx < re && idx > rs) ? B.ci[idx - 1] : -1;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int idx = base + 32 * u + lane;
      const int wid = c[u] >> shift;
      const bool start = idx < re && (idx == rs || (pc[u] >> shift) != wid);
      const unsigned m = __ballot_sync(FULL, start);
      if (start) runs[pos + __popc(m & lanemask_lt())] = make_int2(wid, idx);
      pos += __popc(m);
    }
  }
  if (lane == 0) runs[rr[k + 1] - 1] = make_int2(INT_MAX, re);
}

__global__ void __launch_bounds__(256) k_runs_fill(Csr B, int s1, const int32_t* __restrict__ rr1,
                                                   int2* __restrict__ runs1, int s2, const int32_t* __restrict__ rr2,
                                                   int2* __restrict__ runs2, const DevStats* st, int win_lo) {
  if (block_skip(st)) return;
  if (no_window_rows(st, win_lo)) return;
  const long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nw = (gridDim.x * (long long)blockDim.x) >> 5;
  for (long long k = w; k < B.nrows; k += nw) {
    runs_fill_row(B, (int)k, s1, rr1, runs1);
    if (runs2) runs_fill_row(B, (int)k, s2, rr2, runs2);
  }
}

cudaError_t launch_runs(const LaunchCtx& c, const Csr& B, const SplitInfo& sp, long long* partials, int win_lo) {
  if (!sp.rr || !sp.runs) return cudaSuccess;
  const bool two = sp.rrb && sp.runsb;
  if (B.nrows <= 0) {
    cudaError_t e = cudaMemsetAsync(sp.rr, 0, sizeof(int32_t), c.stream);
    if (e == cudaSuccess && two) e = cudaMemsetAsync(sp.rrb, 0, sizeof(int32_t), c.stream);
    return e;
  }
  const int grid = grid_for_warps(B.nrows, 8, c.nsm);
  k_runs_count<<<grid, 256, 0, c.stream>>>(B, sp.wf_shift, sp.rr, sp.wb_shift, two ? sp.rrb : nullptr, c.st,
                                           win_lo);
  count_launch(c);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = launch_scan_runs(c, sp.rr, two ? sp.rrb : nullptr, B.nrows, partials, win_lo);
  if (e != cudaSuccess) return e;
  k_runs_fill<<<grid, 256, 0, c.stream>>>(B, sp.wf_shift, sp.rr, sp.runs, sp.wb_shift, two ? sp.rrb : nullptr,
                                          two ? sp.runsb : nullptr, c.st, win_lo);
  count_launch(c);
  return cudaGetLastError();
}

static int grid_for_warps(long long nwarps, int warps_per_block, int nsm) {
  long long blocks = (nwarps + warps_per_block - 1) / warps_per_block;
  long long cap = (long long)nsm * 8;
  if (blocks > cap) blocks = cap;
  return (int)(blocks < 1 ? 1 : blocks);
}

cudaError_t launch_validate(const LaunchCtx& c, const Csr& M) {
  k_validate<<<grid_for_warps(M.nrows > 0 ? M.nrows : 1, 8, c.nsm), 256, 0, c.stream>>>(M, c.err);
  count_launch(c);
  return cudaGetLastError();
}

cudaError_t launch_analyse(const LaunchCtx& c, const Csr& A, const Csr& B, long long row_begin,
                           long long mloc, long long* prod, int* cmin, int* cmax, int* rows,
                           long long span_min, bool count_dense) {
  if (mloc <= 0) return cudaSuccess;
  timer_mark(c, T_ANALYSE, 0);
  // short rows on average (stencils, aggregation operators): 8 lanes per row
  if (A.nrows > 0 && A.nnz <= 12 * A.nrows)
    k_analyse_short<<<grid_for_warps((mloc + 15) / 16, 8, c.nsm), 256, 0, c.stream>>>(A, B, row_begin, mloc, prod,
                                                                                     cmin, cmax, c.st, span_min, count_dense);
  else
    k_analyse<<<grid_for_warps(mloc, 8, c.nsm), 256, 0, c.stream>>>(A, B, row_begin, mloc, prod, cmin, cmax, c.st,
                                                                    count_dense);
  count_launch(c);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const long long blocks = (mloc + SCATTER_ROWS - 1) / SCATTER_ROWS;
  k_bin_scatter<<<(unsigned)blocks, 256, 0, c.stream>>>(prod, mloc, c.st, rows);
  count_launch(c);
  timer_mark(c, T_ANALYSE, 1);
  return cudaGetLastError();
}

}  // namespace sg
