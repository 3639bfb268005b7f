// Numeric pass for rows whose products all fit in a block's registers.
//
// Row i of C is the sum over A(i,k) of A(i,k) * B(k,:) (Sec. 2.2).  One block
// of NT threads owns one row of at most 8 * NT products at a time and reads
// every product once: thread t keeps 8 of them (column and value) in
// registers.  The sorted position of a column in the output row is its rank
// among the row's distinct columns, taken from a presence bitmap in shared
// memory:
//
//  1. the nonzeros of A become a list of segments of B with their offsets in
//     the row's product stream; a bit per product marks where a segment
//     starts, so the segment of a product is a popcount (32 products share one
//     word of the marks, read as a broadcast),
//  2. every product sets its column's bit; the one that sets it first is the
//     column's owner (the others found the bit set),
//  3. a prefix sum of the words' popcounts turns (word, bit) into the rank,
//  4. owners store their product and column at their rank, the others add
//     theirs there (HeldProduct in semiring.cuh) after a barrier,
//  5. the row leaves in one coalesced copy.
//
// A bitmap spans up to 262,144 columns; a wider row takes the next
// window from its smallest column not yet emitted, its products still in
// registers.
//
// Why this split: the window kernels (numwarp.cuh) keep one accumulator per
// COLUMN, so a row of 1,000 products over 65,536 columns walks 64 windows of
// 16 products each and pays a segment search, an emission and a clear for
// every one.  Here a row costs one pass whatever its width.  What bounds it is
// instruction issue (2.5 of 4 per clock, 155 warp instructions per 32 products
// at 16,384 rows of 32 x 32, FP64, 0.11 ms) and the shared-memory traffic of
// random bits and ranks (L1 72 % busy).  65,536 rows of 32 x 32 products over 65,536 columns
// in FP32: 1.58 ms with the warp window, 0.40 ms here; 64 products of 1,024 to
// 50,000 rows (rows of up to 4,096 products, FP64): 10.9 ms and 4.1 ms; R-MAT
// scale 18, rows of 129 to 8,192 products: 6.0 ms and 2.6 ms.
//
// The threads follow the row's products, 8 per thread: rows of up to 8192 fit
// the 64 registers of a block's 1024 threads.  Rows that form many products on
// few columns stay with the warps' windows, which add them without marks and
// ranks (row_is_dense in analyse.cu).
#pragma once

#include "internal.cuh"
#include "semiring.cuh"

namespace sg {

constexpr int ONCE_E = 8;       // products per thread

// Shared memory of a block of NT threads with bitmaps of 2^wlog columns.
template <int NT, typename T>
__host__ __device__ constexpr size_t once_smem_bytes(int wlog) {
  return (size_t)NT * ONCE_E * (sizeof(T) + sizeof(int))  // values and columns by rank (the segment list before)
         + ((size_t)1 << wlog) / 32 * 6                   // presence words and their prefixes (16 bits)
         + (size_t)NT / 4 * 4                             // segment-start marks: a bit per product
         + (size_t)(NT / 32) * 8;                         // per-warp sums and next columns
}

template <int NT>
__host__ __device__ constexpr int once_blocks_per_sm() {
  return NT >= 1024 ? 1 : (NT >= 128 ? 1024 / NT : 12);  // 64 registers per thread (80 for 64 threads)
}

// Widest bitmap (log2 columns) of a block of NT threads: as wide as leaves
// the blocks per SM that the registers allow (R-MAT scale 18, 2^18 columns,
// rows of 4,097 to 8,192 products: 2.97 ms with 2^16 columns, 1.61 ms with
// 2^18; rows of 2,049 to 4,096: 1.32 and 0.73 ms).
template <int NT>
__host__ __device__ constexpr int once_wlog_max() {
  return NT >= 512 ? 18 : (NT >= 128 ? 17 : 16);
}

// Exclusive sum of the NW warps' entries of v before this warp, and the total
// of all (lane w reads entry w: a loop over the entries in every thread of a
// 1024-thread block was a quarter of the kernel's instructions).
template <int NW>
__device__ __forceinline__ int once_before(const int* v, int warp, int* total) {
  const int lane = lane_id();
  const int x = lane < NW ? v[lane] : 0;
  *total = __reduce_add_sync(FULL, x);
  return __reduce_add_sync(FULL, lane < warp ? x : 0);
}

template <int NT, typename T, int SR = SPGEMM_PLUS_TIMES>
__global__ void __launch_bounds__(NT, once_blocks_per_sm<NT>())
k_num_once(Csr A, Csr B, const T* __restrict__ av, const T* __restrict__ bv, RowInfo ri, const DevStats* st,
           int bin_lo, int bin_hi, int wlog, const int32_t* __restrict__ c_rp, int32_t* __restrict__ c_ci,
           T* __restrict__ c_v, uint32_t* err) {
  constexpr int E = ONCE_E, CAP = NT * E, NW = NT / 32, HW = CAP / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_lb, s_le;
  const int W = 1 << wlog;
  T* const acc = reinterpret_cast<T*>(smem_raw);              // by rank; the segments' multipliers before
  int* const ccol = reinterpret_cast<int*>(acc + CAP);        // by rank; the segments' positions before
  uint32_t* const bits = reinterpret_cast<uint32_t*>(ccol + CAP);
  uint32_t* const marks = bits + W / 32;
  int* const wsum = reinterpret_cast<int*>(marks + HW);
  int* const wnext = wsum + NW;
  uint16_t* const pre = reinterpret_cast<uint16_t*>(wnext + NW);
  const int tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
  for (int t = tid; t < W / 32; t += NT) bits[t] = 0u;
  for (int t = tid; t < HW; t += NT) marks[t] = 0u;
  block_bin_range(st, bin_lo, bin_hi, &s_lb, &s_le);
  if (block_skip(st)) return;
  const int lb = s_lb, le = s_le;
  const unsigned le_mask = lane == 31 ? FULL : (2u << lane) - 1u;

  // rows are read ahead: the list entry three rows, the bounds in A two and
  // this thread's first nonzero with its row of B one row before their turn,
  // so a row starts with its first segments in registers
  long long idx = (long long)lb + blockIdx.x;
  int r = 0, a0 = 0, a1 = 0, rn = 0, a0n = 0, a1n = 0, s0 = 0, len0 = 0;
  T m0 = T(0);
  if (idx < le) {
    r = ri.rows[idx];
    a0 = A.rp[ri.row_begin + r];
    a1 = A.rp[ri.row_begin + r + 1];
    if (a0 + tid < a1) {
      const int k = A.ci[a0 + tid];
      s0 = B.rp[k];
      len0 = B.rp[k + 1] - s0;
      m0 = av[a0 + tid];
    }
    if (idx + gridDim.x < le) {
      rn = ri.rows[idx + gridDim.x];
      a0n = A.rp[ri.row_begin + rn];
      a1n = A.rp[ri.row_begin + rn + 1];
    }
  }
  for (; idx < le; idx += gridDim.x) {
    const int rnn = idx + 2 * (long long)gridDim.x < le ? ri.rows[idx + 2 * (long long)gridDim.x] : -1;
    const int kn = a0n + tid < a1n ? A.ci[a0n + tid] : -1;  // (no next row: a0n == a1n == 0)
    int out = c_rp[r];
    const int out_end = c_rp[r + 1];
    const int cmx = ri.cmax[r];
    int base = ri.cmin[r] & ~31;

    // ---- segments of B with their stream offsets: (count << 16) + products
    unsigned carry = 0;
    for (int e0 = a0; e0 < a1; e0 += NT) {
      const int e = e0 + tid;
      int s = s0, len = len0;
      T a = m0;
      if (e0 != a0) {
        len = 0;
        if (e < a1) {
          const int k = A.ci[e];
          s = B.rp[k];
          len = B.rp[k + 1] - s;
          a = av[e];
        }
      }
      if (len > CAP) len = CAP + 1;  // the row's bin rules this out; caught below
      const unsigned v = len > 0 ? (1u << 16) + (unsigned)len : 0u;
      const unsigned incl = warp_incl_scan(v);
      if (lane == 31) wsum[warp] = (int)incl;
      __syncthreads();
      int total;
      const unsigned before = carry + (unsigned)once_before<NW>(wsum, warp, &total) + incl - v;
      const int off = (int)(before & 0xffffu), k = (int)(before >> 16);
      if (len > 0) {
        if (off + len <= CAP && k < CAP) {
          ccol[k] = s - off;  // product p of the segment is entry ccol[k] + p of B
          acc[k] = a;
          atomicOr(&marks[off >> 5], 1u << (off & 31));
        } else {
          atomicOr(err, EB_INTERNAL);
        }
      }
      carry += (unsigned)total;
      __syncthreads();
    }
    const int P = min((int)(carry & 0xffffu), CAP);

    // ---- products: batches of 32, 8 consecutive batches per warp
    int col[E];
    HeldProduct<T, SR> pv[E];
    {
      int k0 = 0;  // segments that start before this warp's products
      for (int t = lane; t < warp * E; t += 32) k0 += __popc(marks[t]);
      k0 = warp_sum(k0) - 1;
      T bb[E];
      int ks[E];
#pragma unroll
      for (int u = 0; u < E; ++u) {
        const unsigned m = marks[warp * E + u];
        const int p = (warp * E + u) * 32 + lane;
        ks[u] = k0 + __popc(m & le_mask);
        k0 += __popc(m);
        col[u] = -1;
        bb[u] = T(0);
        if (p < P && ks[u] >= 0) {
          const int q = ccol[ks[u]] + p;
          col[u] = B.ci[q];
          bb[u] = bv[q];
        }
      }
#pragma unroll
      for (int u = 0; u < E; ++u)
        if (col[u] >= 0) pv[u].set(acc[ks[u]], bb[u]);
    }
    // the next row's first nonzeros and the row after that, in flight from here on
    m0 = T(0);
    s0 = len0 = 0;
    if (kn >= 0) {
      m0 = av[a0n + tid];
      s0 = B.rp[kn];
      len0 = B.rp[kn + 1] - s0;
    }
    int a0nn = 0, a1nn = 0;
    if (rnn >= 0) {
      a0nn = A.rp[ri.row_begin + rnn];
      a1nn = A.rp[ri.row_begin + rnn + 1];
    }
    __syncthreads();  // the list is read: its memory becomes the accumulators
    for (int t = tid; t < HW; t += NT) marks[t] = 0u;

    while (true) {  // windows of W columns from base on
      // ---- presence bits; owners are the products that set them.  Columns
      // outside [base, cmx], only in unsorted rows of B, would use words of the
      // bitmap that have no rank and are not cleared: reported and left out
      const int nwords = (min(W, cmx - base + 1) + 31) >> 5;
      unsigned own = 0, here = 0;
      int next = INT_MAX;
#pragma unroll
      for (int u = 0; u < E; ++u) {
        if (col[u] < 0) continue;  // no product, or emitted with an earlier window
        const int j = col[u] - base;
        if ((j >> 5) >= 0 && (j >> 5) < nwords) {
          const unsigned m = 1u << (j & 31);
          here |= 1u << u;
          if (!(atomicOr(&bits[j >> 5], m) & m)) own |= 1u << u;
        } else if (j >= W && col[u] <= cmx) {
          next = min(next, col[u]);
        } else {
          atomicOr(err, EB_UNSORTED);
          col[u] = -1;
        }
      }
      next = warp_min(next);
      if (lane == 0) wnext[warp] = next;
      __syncthreads();

      // ---- prefix of the words' popcounts; a lane takes 8 consecutive words
      const int tiles = (nwords + 255) >> 8, per = (tiles + NW - 1) / NW;
      const int t0 = min(tiles, warp * per), t1 = min(tiles, t0 + per);
      int sum = 0;
      for (int t = t0; t < t1; ++t) {
        const int w0 = (t << 8) + lane * 8;
        if (w0 < nwords) {
          const uint4 x = *reinterpret_cast<const uint4*>(bits + w0);
          const uint4 y = *reinterpret_cast<const uint4*>(bits + w0 + 4);
          sum += __popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w) + __popc(y.x) + __popc(y.y) + __popc(y.z) +
                 __popc(y.w);
        }
      }
      sum = warp_sum(sum);
      if (lane == 0) wsum[warp] = sum;
      __syncthreads();
      int total;
      int run = once_before<NW>(wsum, warp, &total);
      next = warp_min(lane < NW ? wnext[lane] : INT_MAX);
      for (int t = t0; t < t1; ++t) {
        const int w0 = (t << 8) + lane * 8;
        uint4 x = make_uint4(0, 0, 0, 0), y = x;
        if (w0 < nwords) {
          x = *reinterpret_cast<const uint4*>(bits + w0);
          y = *reinterpret_cast<const uint4*>(bits + w0 + 4);
        }
        const int c0 = __popc(x.x), c1 = c0 + __popc(x.y), c2 = c1 + __popc(x.z), c3 = c2 + __popc(x.w);
        const int c4 = c3 + __popc(y.x), c5 = c4 + __popc(y.y), c6 = c5 + __popc(y.z), c7 = c6 + __popc(y.w);
        const int incl = warp_incl_scan(c7);
        const unsigned b = (unsigned)(run + incl - c7);
        if (w0 < nwords) {  // ranks stay below CAP <= 8192: two per word
          const unsigned bb = b | (b << 16);
          uint4 o;
          o.x = bb + ((unsigned)c0 << 16);
          o.y = bb + ((unsigned)c2 << 16 | (unsigned)c1);
          o.z = bb + ((unsigned)c4 << 16 | (unsigned)c3);
          o.w = bb + ((unsigned)c6 << 16 | (unsigned)c5);
          *reinterpret_cast<uint4*>(pre + w0) = o;
        }
        run += __shfl_sync(FULL, incl, 31);
      }
      __syncthreads();

      // ---- ranks: owners store, the others (col -2 - rank from here) add
      // after the barrier
#pragma unroll
      for (int u = 0; u < E; ++u) {
        if (here >> u & 1u) {
          const int j = col[u] - base;
          const int rk = pre[j >> 5] + __popc(bits[j >> 5] & ((1u << (j & 31)) - 1u));
          if (own >> u & 1u) {
            acc[rk] = pv[u].first();
            ccol[rk] = col[u];
            col[u] = -1;
          } else {
            col[u] = -2 - rk;
          }
        }
      }
      __syncthreads();
      int at[E];
#pragma unroll
      for (int u = 0; u < E; ++u) {
        at[u] = -1;
        if (col[u] < -1) {
          at[u] = -2 - col[u];
          col[u] = -1;
        }
      }
      add_held<1>(pv, acc, at, err);
      // the bitmap is clear again for the next window or row
      for (int t = tid * 4; t < nwords; t += NT * 4) *reinterpret_cast<uint4*>(bits + t) = make_uint4(0, 0, 0, 0);
      __syncthreads();
      if (out + total > out_end) {  // the symbolic count rules this out
        if (tid == 0) atomicOr(err, EB_INTERNAL);
        total = max(out_end - out, 0);
      }
      for (int t = tid; t < total; t += NT) {
        __stcs(c_ci + out + t, ccol[t]);
        __stcs(c_v + out + t, acc[t]);
      }
      out += total;
      if (next == INT_MAX) break;
      base = next & ~31;
      __syncthreads();  // the accumulators are read before the next window refills them
    }
    if (tid == 0 && out != out_end) atomicOr(err, EB_INTERNAL);
    __syncthreads();  // ... or the next row's segment list
    r = rn;
    a0 = a0n;
    a1 = a1n;
    rn = rnn;
    a0n = a0nn;
    a1n = a1nn;
  }
}

}  // namespace sg
