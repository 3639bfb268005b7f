// Exclusive prefix sum of the per-row sizes of C into C's row pointer.
//
// No inter-block waiting.  Up to SCAN_SMALL rows one block does it all; up to
// SCAN_TWO tiles two launches: each block reduces one tile, then each block
// adds up the sums of the tiles before its own (a few loads per thread) and
// scans its tile; beyond, a launch of one block between them scans the tile
// sums.  Sums are carried in int64; a total of 2^31 or more sets the overflow
// bit (row pointers are int32).  In place: c_rp[0..m-1] holds the row sizes on
// entry and the row starts on exit, c_rp[m] = nnz(C).
//
// A tile passes through shared memory, so that global loads and stores are
// coalesced while a thread scans 16 consecutive rows: 884,736 rows took 8.2 us
// in the last launch with 16 strided loads and stores per thread, 5.5 us now.
#include "internal.cuh"

namespace sg {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_PER_THREAD = 16;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_PER_THREAD;  // 4096 rows per tile
constexpr int SCAN_TWO = 2048;                             // tiles whose sums every block adds up itself
constexpr int SCAN_SMALL_THREADS = 1024;
constexpr long long SCAN_SMALL = 4 * SCAN_SMALL_THREADS * 4;  // rows of the one-block scan: four steps

size_t scan_partials_count(long long mloc) {
  return (size_t)((mloc + SCAN_TILE - 1) / SCAN_TILE) + 1;
}

// Block-wide exclusive scan of one int64 per thread; returns the block total.
template <int NT>
__device__ __forceinline__ long long block_excl_scan(long long v, long long* total) {
  __shared__ long long s_warp[NT / 32];
  __shared__ long long s_total;
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  long long incl = warp_incl_scan(v);
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    long long w = lane < NT / 32 ? s_warp[lane] : 0;
    long long wi = warp_incl_scan(w);
    if (lane < NT / 32) s_warp[lane] = wi - w;
    if (lane == 31) s_total = wi;
  }
  __syncthreads();
  long long r = incl - v + s_warp[warp];
  *total = s_total;
  __syncthreads();
  return r;
}

// One sum of a launch: two of them may share their launches (blockIdx.y).
struct ScanArgs {
  int32_t* rp;
  long long* part;
  long long* total;
  int win_lo;  // > 0: nothing to do when no row is in bins win_lo and above
};

__device__ __forceinline__ int scan_size(const int32_t* __restrict__ rp, const long long* __restrict__ prod,
                                         long long r, long long m) {
  return r < m && (!prod || prod[r] > 0) ? rp[r] : 0;
}

// Every thread of the last block must call it.
__device__ __forceinline__ void scan_finish(const ScanArgs& a, long long m, long long total, DevStats* st,
                                            unsigned* reset, DevStats* mirror) {
  if (threadIdx.x == 0) {
    *a.total = total;
    if (total >= (1ll << 31)) atomicOr(&st->err, EB_OVERFLOW);
    a.rp[m] = (int32_t)(total < (1ll << 31) ? total : 0);
    if (reset) reset[0] = reset[1] = 0u;
  }
  if (!mirror) return;
  __threadfence();
  __syncthreads();
  static_assert(sizeof(DevStats) % 4 == 0, "copied by words");
  for (unsigned w = threadIdx.x; w < sizeof(DevStats) / 4; w += blockDim.x)
    reinterpret_cast<volatile unsigned*>(mirror)[w] = reinterpret_cast<const volatile unsigned*>(st)[w];
}

__global__ void __launch_bounds__(SCAN_SMALL_THREADS) k_scan_small(ScanArgs a0, ScanArgs a1, long long m,
                                                                  const long long* __restrict__ prod, DevStats* st,
                                                                  unsigned* reset, DevStats* mirror) {
  const ScanArgs a = blockIdx.y ? a1 : a0;
  if (no_window_rows(st, a.win_lo)) return;
  long long carry = 0, total;
  for (long long b = 0; b < m; b += 4 * SCAN_SMALL_THREADS) {
    const long long r = b + 4 * (long long)threadIdx.x;
    int v[4];
    long long sum = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[j] = scan_size(a.rp, prod, r + j, m);
      sum += v[j];
    }
    long long ex = carry + block_excl_scan<SCAN_SMALL_THREADS>(sum, &total);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (r + j < m) a.rp[r + j] = (int32_t)ex;  // wraps only when the overflow bit is set
      ex += v[j];
    }
    carry += total;
  }
  scan_finish(a, m, carry, st, blockIdx.y ? nullptr : reset, blockIdx.y ? nullptr : mirror);
}

__global__ void __launch_bounds__(SCAN_THREADS) k_scan_reduce(ScanArgs a0, ScanArgs a1, long long m,
                                                             const long long* __restrict__ prod,
                                                             const DevStats* st) {
  const ScanArgs a = blockIdx.y ? a1 : a0;
  if (no_window_rows(st, a.win_lo)) return;
  const long long base = (long long)blockIdx.x * SCAN_TILE;
  long long v = 0, total;
#pragma unroll
  for (int j = 0; j < SCAN_PER_THREAD; ++j)
    v += scan_size(a.rp, prod, base + (long long)j * SCAN_THREADS + threadIdx.x, m);
  block_excl_scan<SCAN_THREADS>(v, &total);
  if (threadIdx.x == 0) a.part[blockIdx.x] = total;
}

// One block: exclusive scan of the tile sums in place, their total behind them.
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_partials(ScanArgs a0, ScanArgs a1, long long ntiles,
                                                               const DevStats* st) {
  const ScanArgs a = blockIdx.y ? a1 : a0;
  if (no_window_rows(st, a.win_lo)) return;
  long long carry = 0, total;
  for (long long b = 0; b < ntiles; b += SCAN_THREADS) {
    const long long i = b + threadIdx.x;
    const long long ex = block_excl_scan<SCAN_THREADS>(i < ntiles ? a.part[i] : 0, &total);
    if (i < ntiles) a.part[i] = carry + ex;
    carry += total;
  }
  if (threadIdx.x == 0) a.part[ntiles] = carry;
}

// SCANNED: part holds the tiles' offsets (and their total behind them), not
// their sums.
template <bool SCANNED>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_down(ScanArgs a0, ScanArgs a1, long long m,
                                                           const long long* __restrict__ prod, DevStats* st,
                                                           unsigned* reset, DevStats* mirror) {
  __shared__ int s_tile[SCAN_TILE + SCAN_TILE / 16];  // one word of padding per thread's 16
  const ScanArgs a = blockIdx.y ? a1 : a0;
  if (no_window_rows(st, a.win_lo)) return;
  const long long base = (long long)blockIdx.x * SCAN_TILE;
  const int tid = threadIdx.x;
#pragma unroll
  for (int j = 0; j < SCAN_PER_THREAD; ++j) {
    const int q = j * SCAN_THREADS + tid;
    s_tile[q + (q >> 4)] = scan_size(a.rp, prod, base + q, m);
  }
  long long before = 0, total;
  if (SCANNED) {
    before = a.part[blockIdx.x];
    __syncthreads();
  } else {
    long long v = 0;
    for (int t = tid; t < (int)blockIdx.x; t += SCAN_THREADS) v += a.part[t];
    block_excl_scan<SCAN_THREADS>(v, &before);  // its barriers publish the tile as well
  }
  int v[SCAN_PER_THREAD];
  long long sum = 0;
#pragma unroll
  for (int j = 0; j < SCAN_PER_THREAD; ++j) {
    v[j] = s_tile[tid * 17 + j];
    sum += v[j];
  }
  long long ex = before + block_excl_scan<SCAN_THREADS>(sum, &total);
#pragma unroll
  for (int j = 0; j < SCAN_PER_THREAD; ++j) {
    s_tile[tid * 17 + j] = (int32_t)ex;  // wraps only when the overflow bit is set
    ex += v[j];
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < SCAN_PER_THREAD; ++j) {
    const int q = j * SCAN_THREADS + tid;
    if (base + q < m) a.rp[base + q] = s_tile[q + (q >> 4)];
  }
  if (blockIdx.x == gridDim.x - 1)
    scan_finish(a, m, before + total, st, blockIdx.y ? nullptr : reset, blockIdx.y ? nullptr : mirror);
}

static cudaError_t scan_launch(const LaunchCtx& c, int sums, const ScanArgs& a0, const ScanArgs& a1, long long m,
                               const long long* prod, unsigned* reset, DevStats* mirror) {
  const long long ntiles = (m + SCAN_TILE - 1) / SCAN_TILE;
  timer_mark(c, T_SCAN, 0);
  if (m <= SCAN_SMALL) {
    k_scan_small<<<dim3(1, sums), SCAN_SMALL_THREADS, 0, c.stream>>>(a0, a1, m, prod, c.st, reset, mirror);
    count_launch(c);
  } else {
    k_scan_reduce<<<dim3((unsigned)ntiles, sums), SCAN_THREADS, 0, c.stream>>>(a0, a1, m, prod, c.st);
    count_launch(c);
    if (ntiles <= SCAN_TWO) {
      k_scan_down<false><<<dim3((unsigned)ntiles, sums), SCAN_THREADS, 0, c.stream>>>(a0, a1, m, prod, c.st, reset, mirror);
    } else {
      k_scan_partials<<<dim3(1, sums), SCAN_THREADS, 0, c.stream>>>(a0, a1, ntiles, c.st);
      count_launch(c);
      k_scan_down<true><<<dim3((unsigned)ntiles, sums), SCAN_THREADS, 0, c.stream>>>(a0, a1, m, prod, c.st, reset, mirror);
    }
    count_launch(c);
  }
  timer_mark(c, T_SCAN, 1);
  return cudaGetLastError();
}

cudaError_t launch_scan(const LaunchCtx& c, int32_t* c_rp, long long m, long long* part, long long* total_out,
                        const long long* prod, unsigned* reset, DevStats* mirror) {
  const ScanArgs a{c_rp, part, total_out ? total_out : &c.st->nnz_c, 0};
  return scan_launch(c, 1, a, a, m, prod, reset, mirror);
}

cudaError_t launch_scan_runs(const LaunchCtx& c, int32_t* rr, int32_t* rrb, long long m, long long* partials,
                             int win_lo) {
  const ScanArgs a{rr, partials, &c.st->nruns, win_lo};
  const ScanArgs b{rrb, partials + scan_partials_count(m), &c.st->nruns_b, win_lo};
  return scan_launch(c, rrb ? 2 : 1, a, b, m, nullptr, nullptr, nullptr);
}

}  // namespace sg
