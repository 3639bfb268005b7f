// Numeric pass for long rows: rank-compacted accumulators, a band of ranks at a
// time.
//
// Row i of C is the sum over A(i,k) of A(i,k) * B(k,:) (Sec. 2.2).  One block
// owns one row.  A first walk over the columns of the row's products sets a
// presence bitmap over (up to) 262,144 columns in shared memory, and a prefix
// sum of its words' popcounts gives every column its rank in the row.  The
// ranks are then taken in bands of at most CAP: a band is an interval of
// columns (cut at a word of the bitmap), so every nonzero's part of B(k,:) in
// it is one segment, found by a binary search from the previous band's end.
// Products add to the accumulator at their rank and leave the low 16 bits of
// their column there; the band leaves as one coalesced copy (the columns' high
// bits follow from the rank, since 65,536 columns are 8 tiles of the prefix
// sum).
//
// Compared with a dense window of 8192 columns (numblock.cuh), a band holds as
// many OUTPUTS as that window holds columns: a row of 35,000 outputs over
// 262,144 columns takes 6 bands instead of 32 windows, and its segments are
// five times as long, so that a warp's 32 products mostly come from one row of
// B -- distinct columns, no retries of the shared-memory compare-and-swap --
// without mapping products to segments one by one.  The price is the first
// walk over the columns and a bitmap look-up per product; rows on few columns,
// which need one or two windows, stay with the warps' windows (numwarp.cuh).
//
// What bounds it is the shared-memory pipe (the swap of 64-bit words at 17
// cycles a warp, look-ups and stores of a batch of 32 products about 30 more)
// and, below 65,536 products, the latency of a row's phases with two rows on
// an SM.  R-MAT scale 18, FP64: rows of 8,193 to 65,536 products 10.3 ms with
// a warp's 1024-column windows and 7.4 in bands; with the longer rows, which a
// block's 8192-column windows took 14.6 ms for, 22.9 ms together.  262,144
// columns, edge factor 8, FP32: 8.5 and 4.4 ms; 150,000 columns, edge factor 4,
// FP64: 1.4 and 1.2 ms.
#pragma once

#include "segstream.cuh"
#include "semiring.cuh"
#include "symblock.cuh"

namespace sg {

constexpr int BAND_THREADS = 512;
constexpr int BAND_WLOG = 18;  // widest bitmap

template <typename T>
__host__ __device__ constexpr int band_cap() {
  return sizeof(T) == 8 ? 5120 : 8192;  // ranks per band: two blocks share an SM
}

template <typename T>
__host__ __device__ constexpr size_t band_smem_bytes(int wlog) {
  return (size_t)band_cap<T>() * (sizeof(T) + 2)               // accumulators and columns by rank
         + (size_t)BAND_THREADS * (sizeof(T) + 2 * sizeof(int))  // segments: multiplier, stream offset, start in B
         + ((size_t)1 << wlog) / 32 * 6;                       // presence words and their prefixes (16 bits)
}

// One product: acc[rank of col] += a * b.  col: relative to the window; first:
// rank (modulo 65,536) of the band's first column.
template <typename T, int SR>
__device__ __forceinline__ void band_add(int col, T a, T b, unsigned first, int W, const uint32_t* bits,
                                         const uint16_t* pre, T* acc, uint16_t* ccol, int cap,
                                         uint32_t* err) {
  const unsigned j = min((unsigned)col, (unsigned)W - 1u);  // (outside only in unsorted rows of B, reported already)
  const uint32_t word = bits[j >> 5];
  const unsigned rank = ((unsigned)pre[j >> 5] + (unsigned)__popc(word & ((1u << (j & 31)) - 1u)) - first) & 0xffffu;
  if (rank < (unsigned)cap) {
    ccol[rank] = (uint16_t)j;
    SrOps<T, SR>::madd_shared(&acc[rank], a, b, err);
  } else {
    atomicOr(err, EB_INTERNAL);
  }
}

// The products [lo, hi) of the band's stream (tot products, nseg segments).
// While at least 32 products of the current segment are left, lanes walk it
// directly, four loads in flight per lane; batches that straddle segments find
// each lane's segment from the segment ends.  Every lane must call it.
template <typename T, int SR>
__device__ __forceinline__ void band_range(const Csr& B, const T* __restrict__ bv, const int* off, const int* sstart,
                                           const T* sa, int nseg, int tot, int lo, int hi, int base, unsigned first, int W,
                                           const uint32_t* bits, const uint16_t* pre, T* acc, uint16_t* ccol, int cap,
                                           uint32_t* err) {
  const int lane = lane_id();
  int f = seg_find(off, nseg, lo);
  int p = lo;
  while (p < hi) {
    const int sb = off[f];
    const int se = f + 1 < nseg ? off[f + 1] : tot;
    const int run = min(se, hi) - p;
    if (run >= 32) {  // whole batches inside segment f
      const int n = run & ~31;
      const int q = sstart[f] + (p - sb);
      const int* __restrict__ ci = B.ci + q;
      const T* __restrict__ v = bv + q;
      const T a = sa[f];
      int t = lane;
      for (; t + 96 < n; t += 128) {
        const int c0 = ci[t], c1 = ci[t + 32], c2 = ci[t + 64], c3 = ci[t + 96];
        const T b0 = v[t], b1 = v[t + 32], b2 = v[t + 64], b3 = v[t + 96];
        band_add<T, SR>(c0 - base, a, b0, first, W, bits, pre, acc, ccol, cap, err);
        band_add<T, SR>(c1 - base, a, b1, first, W, bits, pre, acc, ccol, cap, err);
        band_add<T, SR>(c2 - base, a, b2, first, W, bits, pre, acc, ccol, cap, err);
        band_add<T, SR>(c3 - base, a, b3, first, W, bits, pre, acc, ccol, cap, err);
      }
      for (; t < n; t += 32) band_add<T, SR>(ci[t] - base, a, v[t], first, W, bits, pre, acc, ccol, cap, err);
      p += n;
      if (p == se) ++f;
      continue;
    }
    // one batch across segments: lane j holds the end of segment f + j
    const int nx = f + lane + 1;
    const int end = nx < nseg ? off[nx] : (nx == nseg ? tot : INT_MAX);
    const int d = end == INT_MAX ? INT_MAX : end - p;
    const unsigned m = __reduce_or_sync(FULL, d <= 31 ? (1u << d) : 0u);
    const int k = f + __popc(m & (lane == 31 ? FULL : ((2u << lane) - 1u)));
    const int q = p + lane;
    if (q < hi) {
      const int x = sstart[k] + (q - off[k]);
      band_add<T, SR>(B.ci[x] - base, sa[k], bv[x], first, W, bits, pre, acc, ccol, cap, err);
    }
    const int pn = p + 32;
    if (pn < hi) {  // segment of the next product
      const int c = __popc(__ballot_sync(FULL, end <= pn));
      f = c < 32 ? f + c : seg_find(off, nseg, pn);
    }
    p = pn;
  }
}

// First entry of B in [lo, hi) whose column is at least c (hi if none).
__device__ __forceinline__ int band_bound(const int32_t* __restrict__ ci, int lo, int hi, int c) {
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (ci[mid] < c) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// gcur, gend: per nonzero of A, the first entry of its row of B not yet added
// and the end of its part in the current window (rows of more than
// BAND_THREADS nonzeros; shorter ones keep both in registers).
template <typename T, int SR = SPGEMM_PLUS_TIMES>
__global__ void __launch_bounds__(BAND_THREADS, 2)
k_num_band(Csr A, Csr B, const T* __restrict__ av, const T* __restrict__ bv, RowInfo ri, const DevStats* st,
           int bin_lo, int bin_hi, int wlog, int32_t* __restrict__ gcur, int32_t* __restrict__ gend,
           const int32_t* __restrict__ c_rp, int32_t* __restrict__ c_ci, T* __restrict__ c_v, unsigned* counter,
           uint32_t* err) {
  constexpr int NT = BAND_THREADS, NW = NT / 32, CAP = band_cap<T>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_lb, s_le, s_item;
  __shared__ unsigned long long s_pack[2];  // (segments << 32) | products, alternate rounds
  __shared__ int s_tile[33];                // ranks before each tile of 256 words (past the last: all)
  __shared__ int s_next[NW];
  const int W = 1 << wlog;
  T* const acc = reinterpret_cast<T*>(smem_raw);
  T* const seg_a = acc + CAP;
  uint32_t* const bits = reinterpret_cast<uint32_t*>(seg_a + NT);
  int* const seg_off = reinterpret_cast<int*>(bits + W / 32);
  int* const seg_s = seg_off + NT;
  uint16_t* const pre = reinterpret_cast<uint16_t*>(seg_s + NT);
  uint16_t* const ccol = pre + W / 32;
  const int tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
  for (int t = tid; t < CAP; t += NT) acc[t] = SrOps<T, SR>::zero();
  for (int t = tid; t < W / 32; t += NT) bits[t] = 0u;
  block_bin_range(st, bin_lo, bin_hi, &s_lb, &s_le);
  if (tid == 0) s_pack[0] = s_pack[1] = 0ull;
  if (block_skip(st)) return;
  const int lb = s_lb, le = s_le;
  int parity = 0;

  while (true) {
    if (tid == 0) s_item = (int)atomicAdd(counter, 1u);
    __syncthreads();
    const long long idx = (long long)lb + s_item;
    if (idx >= le) break;
    const int r = ri.rows[idx];
    const int a0 = A.rp[ri.row_begin + r], a1 = A.rp[ri.row_begin + r + 1];
    const int cmx = ri.cmax[r];
    int base = ri.cmin[r] & ~31;
    int out = c_rp[r];
    const int out_end = c_rp[r + 1];
    const bool regc = a1 - a0 <= NT;  // block-uniform
    int cur = 0, re = 0, wend = 0;    // this thread's nonzero: cursor, row end, window end
    T ra = T(0);
    if (regc) {
      if (a0 + tid < a1) {
        const int k = A.ci[a0 + tid];
        cur = B.rp[k];
        re = B.rp[k + 1];
        ra = av[a0 + tid];
      }
    } else {
      for (int e = a0 + tid; e < a1; e += NT) gcur[e] = B.rp[A.ci[e]];
    }
    while (true) {  // windows of W columns from base on
      const bool last_window = (long long)base + W > cmx;
      // ---- presence bits of the window's products
      int next = INT_MAX;
      for (int r0 = a0; r0 < a1; r0 += NT) {
        const int e = r0 + tid;
        if (!regc) {
          cur = re = 0;
          if (e < a1) {
            cur = gcur[e];
            re = B.rp[A.ci[e] + 1];
          }
        }
        wend = last_window ? re : band_bound(B.ci, cur, re, base + W);
        if (wend < re) next = min(next, B.ci[wend]);
        if (!regc && e < a1) gend[e] = wend;
        seg_append(&s_pack[parity], cur, wend - cur, seg_off, seg_s);
        __syncthreads();  // the list is complete
        const unsigned long long pv = s_pack[parity];
        const int nseg = (int)(pv >> 32), tot = (int)(unsigned)(pv & 0xffffffffull);
        if (tid == 0) s_pack[parity ^ 1] = 0ull;
        const int share = ((tot + NT - 1) / NT) * 32;
        const int lo = warp * share, hi = min(tot, lo + share);
        if (lo < hi) sb_range(B, seg_off, seg_s, nseg, tot, lo, hi, base, W, bits, err);
        __syncthreads();  // bits set; the list may be refilled
        parity ^= 1;
      }
      next = warp_min(next);
      if (lane == 0) s_next[warp] = next;
      // ---- ranks: words in tiles of 256, a warp per tile (at most 32 tiles)
      const int nwords = (min(W, cmx - base + 1) + 31) >> 5;
      const int ntiles = (nwords + 255) >> 8;
      for (int t = warp; t < ntiles; t += NW) {
        const int w0 = (t << 8) + lane * 8;
        uint4 x = make_uint4(0, 0, 0, 0), y = x;
        if (w0 < nwords) {
          x = *reinterpret_cast<const uint4*>(bits + w0);
          y = *reinterpret_cast<const uint4*>(bits + w0 + 4);
        }
        const int c0 = __popc(x.x), c1 = c0 + __popc(x.y), c2 = c1 + __popc(x.z), c3 = c2 + __popc(x.w);
        const int c4 = c3 + __popc(y.x), c5 = c4 + __popc(y.y), c6 = c5 + __popc(y.z), c7 = c6 + __popc(y.w);
        const int incl = warp_incl_scan(c7);
        if (w0 < nwords) {  // ranks inside the tile: at most 8192
          const unsigned b = (unsigned)(incl - c7), bb = b | (b << 16);
          uint4 o;
          o.x = bb + ((unsigned)c0 << 16);
          o.y = bb + ((unsigned)c2 << 16 | (unsigned)c1);
          o.z = bb + ((unsigned)c4 << 16 | (unsigned)c3);
          o.w = bb + ((unsigned)c6 << 16 | (unsigned)c5);
          *reinterpret_cast<uint4*>(pre + w0) = o;
        }
        if (lane == 31) s_tile[t + 1] = incl;
      }
      __syncthreads();
      next = warp_min(lane < NW ? s_next[lane] : INT_MAX);
      int total;
      {
        const int v = lane < ntiles ? s_tile[lane + 1] : 0;
        const int incl = warp_incl_scan(v);
        total = __shfl_sync(FULL, incl, 31);
        __syncthreads();  // every warp has read the tile counts
        if (warp == 0) {
          if (lane == 0) s_tile[0] = 0;
          s_tile[lane + 1] = incl;  // tiles past the last: the total
        }
        for (int t = warp; t < ntiles; t += NW) {  // add the tiles' offsets (modulo 65,536) to the words'
          const unsigned tb = (unsigned)__shfl_sync(FULL, incl - v, t) & 0xffffu;
          const int w0 = (t << 8) + lane * 8;
          if (w0 < nwords) {
            uint4 o = *reinterpret_cast<const uint4*>(pre + w0);
            auto add2 = [&](unsigned p) { return ((p + tb) & 0xffffu) | ((p & 0xffff0000u) + (tb << 16)); };
            o.x = add2(o.x); o.y = add2(o.y); o.z = add2(o.z); o.w = add2(o.w);
            *reinterpret_cast<uint4*>(pre + w0) = o;
          }
        }
      }
      __syncthreads();
      if (out + total > out_end) {  // the symbolic count rules this out
        if (tid == 0) atomicOr(err, EB_INTERNAL);
        total = max(out_end - out, 0);
      }
      // ---- bands of at most CAP ranks [rank0, rank1), cut at word w1
      int rank0 = 0;
      while (rank0 < total) {
        int w1 = nwords, rank1 = total;
        if (total - rank0 > CAP) {
          // the last tile, then the last word, with at most CAP ranks before it
          const unsigned tb = __ballot_sync(FULL, lane < ntiles && s_tile[lane] - rank0 <= CAP);
          const int t = 31 - __clz(tb);
          const int tile0 = s_tile[t];
          int ok = 0;
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int w = (t << 8) + u * 32 + lane;
            if (w < nwords && tile0 + (int)(((unsigned)pre[w] - (unsigned)tile0) & 0xffffu) - rank0 <= CAP) ++ok;
          }
          w1 = (t << 8) + __reduce_add_sync(FULL, ok) - 1;
          rank1 = tile0 + (int)(((unsigned)pre[w1] - (unsigned)tile0) & 0xffffu);
        }
        const int c1 = base + 32 * w1;  // first column of the next band
        const bool last_band = w1 == nwords;
        for (int r0 = a0; r0 < a1; r0 += NT) {
          const int e = r0 + tid;
          T a = ra;
          if (!regc) {
            cur = wend = 0;
            a = T(0);
            if (e < a1) {
              cur = gcur[e];
              wend = gend[e];
              a = av[e];
            }
          }
          const int end = last_band ? wend : band_bound(B.ci, cur, wend, c1);
          seg_append<T>(&s_pack[parity], cur, end - cur, a, seg_off, seg_s, seg_a);
          cur = end;
          if (!regc && e < a1) gcur[e] = end;
          __syncthreads();  // the list is complete
          const unsigned long long pv = s_pack[parity];
          const int nseg = (int)(pv >> 32), tot = (int)(unsigned)(pv & 0xffffffffull);
          if (tid == 0) s_pack[parity ^ 1] = 0ull;
          const int share = ((tot + NT - 1) / NT) * 32;
          const int lo = warp * share, hi = min(tot, lo + share);
          if (lo < hi)
            band_range<T, SR>(B, bv, seg_off, seg_s, seg_a, nseg, tot, lo, hi, base, (unsigned)rank0, W, bits, pre,
                              acc, ccol, CAP, err);
          __syncthreads();  // all products in; the list may be refilled
          parity ^= 1;
        }
        // ---- the band leaves; rank of the columns at 65,536, 131,072, 196,608
        const int n = rank1 - rank0;
        const int h1 = s_tile[8] - rank0, h2 = s_tile[16] - rank0, h3 = s_tile[24] - rank0;
#pragma unroll 4
        for (int t = tid; t < n; t += NT) {
          const T v = acc[t];
          const int j = (int)ccol[t] + 65536 * ((t >= h1) + (t >= h2) + (t >= h3));
          acc[t] = SrOps<T, SR>::zero();
          __stcs(c_ci + out + t, base + j);
          __stcs(c_v + out + t, v);
        }
        out += n;
        rank0 = rank1;
        // the next round's list barrier orders these stores before its products
      }
      for (int t = tid * 4; t < nwords; t += NT * 4) *reinterpret_cast<uint4*>(bits + t) = make_uint4(0, 0, 0, 0);
      __syncthreads();
      if (next == INT_MAX) break;
      base = next & ~31;
    }
    if (tid == 0 && out != out_end) atomicOr(err, EB_INTERNAL);
  }
}

}  // namespace sg
