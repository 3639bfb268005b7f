// Masked product C<M> = (A*B) .* M on the pattern of M: the sampled product
// behind triangle counting and Markov clustering, two of the SpGEMM
// applications Sec. 1 lists.  For entry p = (i,j) of M,
//   C[p] = M(i,j) * sum_k A(i,k) * B(k,j)     (factor 1 without M's values),
// 0 when no product reaches (i,j).  Every row runs the row-wise Gustavson
// order of Sec. 2.2 (A's entries of the row, each with its row of B) and
// keeps only the products whose column lies in M's row.
//
// Rows of A with at least 64 nonzeros, and a mask row of at most 4 columns for
// each, go to blocks (k_masked_rows, below), the other rows to warps
// (k_masked): their work is cut into units of 32 consecutive nonzeros of A.  A
// warp finds the row of its unit's first nonzero by a 32-way search over A's
// row pointer, the others follow from it.
// A product whose column lies in its row of M adds its rounded value
// A(i,k)*B(k,j) to that entry.
//
// Few products do (6 % in triangle counting on R-MAT graphs), so turning the
// others away decides the speed.  The part of a row of A inside the unit that
// forms at least MASK_MIN_PRODUCTS products, and MASK_RATIO for each mask
// column, is handled by itself, with the row's mask columns and one
// accumulator each in shared memory (up to MASK_CAP columns; longer mask rows
// stay in global memory):
//  * a row of B much longer than the mask row is not read at all: each mask
//    column is searched in it, four rows of B at a time,
//  * otherwise the mask columns set bits of a hashed bitmap in shared memory
//    (the column's low 12 bits) and a product costs one load of its column
//    and one test; rows of B of at least 32 entries are walked directly by
//    the warp, shorter ones are flattened so that every lane has a product,
//  * products that pass wait in a queue and are looked up 32 at a time, all
//    lanes busy, by a binary search over the mask row; hits add with a
//    shared-memory reduction, and the row ends by adding its nonzero
//    accumulators to the output with global reductions (other units of the
//    row add to the same entries).
// The remaining products are flattened over all their rows and search the
// mask row in global memory one by one: parts of few products, where staging
// does not pay, and masks that most products hit (the full pattern of A*B has
// no more columns than products).
//
// A block is two warps and takes two units, so that the hardware's block
// scheduler balances units of very different work.  (One warp a block spends
// more on starting blocks: 96^3 stencil with its square's pattern 0.58 ms, 0.54
// with two and with four; R-MAT of 65,536 columns with its square's 4.84, 4.44
// and 4.78.  Long rows on warps left 40 % of the SM cycles idle: the warps of the
// longest row of a power-law graph alone took two thirds of the kernel's time.)
//
// Strictly lower triangles of R-MAT graphs, with a search of the mask row per
// product, with warps alone, and now: scale 16 (147 M products) 1.61, 1.15 and
// 0.47 ms (blocks 0.31, warps 0.15), scale 18 (1.1 G products) 10.1, 5.6 and
// 2.2 ms.  Masks that nearly every product hits, with a search per product and
// now: the pattern of a square, 96^3 stencil 0.55 and 0.54 ms (min-plus 0.96 and
// 0.93), R-MAT of 65,536 columns 6.3 and 4.4 ms.  The stencil with its own
// pattern as the mask pays for the pass that looks for long rows: 0.43 and
// 0.49 ms.
//
// The output is zeroed before and, with M's values, scaled by them after
// (the sum is finished before the factor, as in the definition).
#include <type_traits>

#include "launch_util.cuh"
#include "segstream.cuh"

namespace sg {

constexpr int MASK_WARPS = 2;             // warps per block, each with a unit of its own
constexpr int MASK_CAP = 384;             // mask columns staged per warp (32 warps share an SM)
constexpr int MASK_BITS = 4096;           // bits of the hashed bitmap
constexpr int MASK_FILTER_MAX = 2048;     // longest mask row worth the bitmap (two bits per column)
constexpr int MASK_MIN_PRODUCTS = 128;    // fewest products worth staging a row,
constexpr int MASK_RATIO = 4;             // and per mask column,
constexpr int MASK_UNIT_PRODUCTS = 512;   // in a unit of this many in all (a stencil's units have 224)
constexpr int MASK_ROW_MIN = 64;          // nonzeros of a row that blocks take,
constexpr int MASK_ROW_RATIO = 4;         // with at most this many mask columns each
constexpr int MASK_BLOCK = 256;           // threads of such a block, most nonzeros of its unit
constexpr int MASK_UNITS_PER_SM = 10;     // units below which they are made smaller
constexpr int MASK_BLOCK_CAP = 1536;      // mask columns staged with accumulators per block
constexpr int MASK_BLOCK_BITS = 65536;    // bits of its hashed bitmap
constexpr int MASK_BLOCK_QUEUE = 160;     // products of a warp that passed it (fewer than 32 wait)
constexpr int MASK_ROUND = 1 << 22;       // entries of one row of B in a block's list at a time
constexpr int MASK_QUEUE = 64;            // products that passed the bitmap (fewer than 32 wait)

// Largest r with rp[r] <= e (the row holding position e) over rows [0, m),
// the same e on every lane: 32 probes a step.
__device__ __forceinline__ int warp_row_of(const int32_t* __restrict__ rp, int m, int e) {
  int lo = 0, hi = m;  // rp[lo] <= e, rp[hi] > e or hi == m
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) >> 5;
    const long long q = (long long)lo + (long long)lane_id() * step;
    const unsigned b = __ballot_sync(FULL, q < hi && rp[q < hi ? q : lo] <= e);
    const int last = b ? 31 - __clz(b) : 0;
    lo += last * step;
    hi = min(hi, lo + step);
  }
  return lo;
}

// Row holding position e, searched upward from `row` (rp[row] <= e).
__device__ __forceinline__ int row_from(const int32_t* __restrict__ rp, int m, int row, int e) {
  if (row + 1 >= m || rp[row + 1] > e) return row;
  int lo = row + 1, step = 1;  // rp[lo] <= e
  while (lo + step < m && rp[lo + step] <= e) {
    lo += step;
    step <<= 1;
  }
  int hi = min(lo + step, m);
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (rp[mid] <= e) lo = mid; else hi = mid;
  }
  return lo;
}

// Position of column j in the ascending ci[lo, end), or -1.
__device__ __forceinline__ int find_in(const int32_t* __restrict__ ci, int lo, int end, int j) {
  int hi = end;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (ci[mid] < j) lo = mid + 1; else hi = mid;
  }
  return (lo < end && ci[lo] == j) ? lo : -1;
}

// Semirings (sum, product, zero): 0 plus-times (+, *, 0); 1 min-plus (min,
// +, +inf); 2 max-plus (max, +, -inf); 3 or-and (or, both nonzero, 0 with
// true written as 1).
template <int SR, typename T>
__device__ __forceinline__ T sr_zero() {
  if (SR == 1) return T(INFINITY);
  if (SR == 2) return T(-INFINITY);
  return T(0);
}

template <int SR, typename T>
__device__ __forceinline__ T sr_product(T a, T b) {
  if (SR == 0) return a * b;
  if (SR == 3) return (a != T(0) && b != T(0)) ? T(1) : T(0);
  return a + b;
}

__device__ __forceinline__ unsigned long long to_bits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ unsigned to_bits(float v) { return __float_as_uint(v); }
__device__ __forceinline__ double from_bits(unsigned long long u) { return __longlong_as_double((long long)u); }
__device__ __forceinline__ float from_bits(unsigned u) { return __uint_as_float(u); }

// *p = min(*p, v) (MIN) or max(*p, v), shared or global memory, by
// compare-and-swap on the bit pattern (no FP64 min/max atomics exist).  A
// failed swap means another update improved the value first, so the loop
// ends after at most as many rounds as there are updates of *p; the bound
// is a guard that no input reaches.
template <bool MIN, typename T>
__device__ __forceinline__ void atomic_minmax(T* p, T v) {
  using U = decltype(to_bits(v));
  U* up = reinterpret_cast<U*>(p);
  U old = *reinterpret_cast<volatile U*>(up);
  for (int it = 0; it < CAS_RETRY_LIMIT; ++it) {
    const T cur = from_bits(old);
    if (MIN ? !(v < cur) : !(v > cur)) return;
    const U prev = atomicCAS(up, old, to_bits(v));
    if (prev == old) return;
    old = prev;
  }
}

// acc (+)= v in shared memory for semiring SR.
template <int SR, typename T>
__device__ __forceinline__ void sr_reduce_shared(T* p, T v) {
  if (SR == 0) red_add_shared(p, v);
  else if (SR == 1) atomic_minmax<true>(p, v);
  else if (SR == 2) atomic_minmax<false>(p, v);
  else if (v != T(0)) *p = T(1);  // every writer writes the same value
}

// out (+)= v in global memory for semiring SR; v equal to the zero is skipped.
template <int SR, typename T>
__device__ __forceinline__ void sr_reduce_global(T* p, T v) {
  if (v == sr_zero<SR, T>()) return;
  if (SR == 0) atomicAdd(p, v);
  else if (SR == 1) atomic_minmax<true>(p, v);
  else if (SR == 2) atomic_minmax<false>(p, v);
  else *p = T(1);
}

// Rows that k_masked_rows takes whole; k_masked leaves them out.
__device__ __forceinline__ bool mask_row_blocked(int la, int n) {
  return la >= MASK_ROW_MIN && n > 0 && (n + MASK_ROW_RATIO - 1) / MASK_ROW_RATIO <= la;
}

// Shared memory of one warp.
template <typename T>
struct MaskWarp {
  T acc[MASK_CAP];
  int2 queue[MASK_QUEUE];  // (entry of B, lane whose nonzero of A owns it)
  int col[MASK_CAP];
  uint32_t bits[MASK_BITS / 32];
};

// acc (+)= v for an accumulator that only this lane updates meanwhile.
template <int SR, typename T>
__device__ __forceinline__ void sr_add_own(T* p, T v) {
  if (SR == 0) *p += v;
  else if (SR == 1) { if (v < *p) *p = v; }
  else if (SR == 2) { if (v > *p) *p = v; }
  else if (v != T(0)) *p = T(1);
}

// Searching the mask's n columns in a row of B of len entries costs about
// 10 * log2(len) instructions per 32 columns, reading the row 50 per 32
// entries.
__device__ __forceinline__ bool mask_search_pays(int n, int len) {
  return len >= 32 && ((n + 31) >> 5) * (32 - __clz(len)) * 6 < len;
}

template <typename T, int SR>
__global__ void __launch_bounds__(MASK_WARPS * 32, 32 / MASK_WARPS)
k_masked(Csr A, Csr B, Csr M, const T* __restrict__ av, const T* __restrict__ bv, T* __restrict__ out, bool blocks) {
  __shared__ MaskWarp<T> s_warp[MASK_WARPS];
  MaskWarp<T>& sm = s_warp[threadIdx.x >> 5];
  const int lane = lane_id();
  const unsigned lt = lanemask_lt();
  {
    const long long u = (long long)blockIdx.x * MASK_WARPS + (threadIdx.x >> 5);
    if (32 * u >= A.nnz) return;
    const int e = (int)(32 * u) + lane;
    const bool ve = e < A.nnz;
    int i = warp_row_of(A.rp, (int)A.nrows, (int)(32 * u)), sb = 0, len = 0;
    T a = T(0);
    if (ve) {
      i = row_from(A.rp, (int)A.nrows, i, e);
      const int k = blocks && mask_row_blocked(A.rp[i + 1] - A.rp[i], M.rp[i + 1] - M.rp[i]) ? -1 : A.ci[e];
      if (k >= 0 && (long long)k < B.nrows) {  // a column of A out of range names no row of B
        sb = B.rp[k];
        len = B.rp[k + 1] - sb;
        a = av[e];
      }
    }
    const int mr0 = M.rp[i], mr1 = M.rp[i + 1];  // the row's mask range (lanes past the end: unused)
    unsigned todo = __ballot_sync(FULL, ve && len > 0 && mr1 > mr0);
    if (!(todo >> lane & 1u)) len = 0;
    // ---- rows of many products, one at a time
    unsigned left = warp_sum(min(len, 1 << 20)) >= MASK_UNIT_PRODUCTS ? todo : 0u;
    while (left) {
      const int L = __ffs(left) - 1;
      const int i0 = __shfl_sync(FULL, i, L);
      const int m0 = __shfl_sync(FULL, mr0, L), n = __shfl_sync(FULL, mr1, L) - m0;
      const unsigned mine = __ballot_sync(FULL, i == i0) & left;
      left &= ~mine;
      const bool in = mine >> lane & 1u;
      // (lengths capped: the sum only decides whether staging pays)
      const int products = warp_sum(in ? min(len, 1 << 20) : 0);
      if (products < MASK_MIN_PRODUCTS || products < MASK_RATIO * n || n > MASK_FILTER_MAX) continue;
      const bool staged = n <= MASK_CAP;
      const bool search = in && mask_search_pays(n, len);
      const bool filter = __any_sync(FULL, in && !search);  // some row of B is read
      if (filter)
        for (int t = lane; t < MASK_BITS / 32; t += 32) sm.bits[t] = 0u;
      __syncwarp();
      for (int t = lane; t < n; t += 32) {
        const int c = M.ci[m0 + t];
        if (filter) atomicOr(&sm.bits[(c >> 5) & (MASK_BITS / 32 - 1)], 1u << (c & 31));
        if (staged) {
          sm.col[t] = c;
          sm.acc[t] = sr_zero<SR, T>();
        }
      }
      __syncwarp();
      // ---- mask columns searched in long rows of B, four rows at a time
      unsigned sm4 = __ballot_sync(FULL, search);
      while (sm4) {
        int s4[4], n4[4];
        T a4[4];
        int most = 0;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int o = sm4 ? __ffs(sm4) - 1 : -1;
          sm4 &= sm4 - 1;  // 0 stays 0
          s4[v] = __shfl_sync(FULL, sb, o & 31);
          n4[v] = __shfl_sync(FULL, len, o & 31);
          a4[v] = __shfl_sync(FULL, a, o & 31);
          if (o < 0) n4[v] = 0;
          most = max(most, n4[v]);
        }
        const int top = 1 << (31 - __clz(most));
        for (int t = lane; t < n; t += 32) {
          const int c = staged ? sm.col[t] : M.ci[m0 + t];
          int at[4] = {0, 0, 0, 0};  // entries of the row below c
          for (int step = top; step > 0; step >>= 1) {
#pragma unroll
            for (int v = 0; v < 4; ++v)
              if (at[v] + step <= n4[v] && B.ci[s4[v] + at[v] + step - 1] < c) at[v] += step;
          }
#pragma unroll
          for (int v = 0; v < 4; ++v)
            if (at[v] < n4[v] && B.ci[s4[v] + at[v]] == c) {
              const T x = sr_product<SR>(a4[v], bv[s4[v] + at[v]]);
              if (staged) sr_add_own<SR>(&sm.acc[t], x);
              else sr_reduce_global<SR>(&out[m0 + t], x);
            }
        }
      }
      __syncwarp();
      const bool rd = in && !search;
      int qn = 0;  // waiting products
      auto look_up = [&](int cnt) {  // the last cnt (at most 32) of the queue
        int2 x = make_int2(0, 0);
        if (lane < cnt) x = sm.queue[qn - cnt + lane];
        const T oa = __shfl_sync(FULL, a, x.y);
        if (lane < cnt) {
          const int j = B.ci[x.x];
          if (staged) {
            const int p = find_in(sm.col, 0, n, j);
            if (p >= 0) sr_reduce_shared<SR>(&sm.acc[p], sr_product<SR>(oa, bv[x.x]));
          } else {
            const int p = find_in(M.ci, m0, m0 + n, j);
            if (p >= 0) sr_reduce_global<SR>(&out[p], sr_product<SR>(oa, bv[x.x]));
          }
        }
        qn -= cnt;
        __syncwarp();  // the entries are read before later ones overwrite them
      };
      auto offer = [&](int j, int bi, int owner, bool act) {
        const bool pass = act && (sm.bits[(j >> 5) & (MASK_BITS / 32 - 1)] >> (j & 31) & 1u);
        const unsigned b = __ballot_sync(FULL, pass);
        if (!b) return;
        if (pass) sm.queue[qn + __popc(b & lt)] = make_int2(bi, owner);
        qn += __popc(b);
        __syncwarp();
        if (qn >= 32) look_up(32);
      };
      // rows of B of at least 32 entries, four loads in flight
      unsigned lm = __ballot_sync(FULL, rd && len >= 32);
      const int sl = rd && len < 32 ? len : 0;
      while (lm) {
        const int o = __ffs(lm) - 1;
        lm &= lm - 1;
        const int s = __shfl_sync(FULL, sb, o), ln = __shfl_sync(FULL, len, o);
        for (int t = lane; t - lane < ln; t += 128) {
          int j[4];
#pragma unroll
          for (int v = 0; v < 4; ++v) j[v] = t + 32 * v < ln ? B.ci[s + t + 32 * v] : 0;
#pragma unroll
          for (int v = 0; v < 4; ++v)
            if (t - lane + 32 * v < ln) offer(j[v], s + t + 32 * v, o, t + 32 * v < ln);  // warp-uniform
        }
      }
      // shorter ones, flattened
      const int incl = warp_incl_scan(sl);
      const int tot = __shfl_sync(FULL, incl, 31);
      const int delta = sb - (incl - sl);  // entry of B minus stream position
      for (int q0 = 0; q0 < tot; q0 += 32) {
        const int q = q0 + lane;
        const int o = warp_owner(incl, q);
        const int bi = __shfl_sync(FULL, delta, o & 31) + q;
        offer(q < tot ? B.ci[bi] : 0, bi, o & 31, q < tot);
      }
      if (qn > 0) look_up(qn);
      if (staged) {
        __syncwarp();
        for (int t = lane; t < n; t += 32) sr_reduce_global<SR>(&out[m0 + t], sm.acc[t]);
      }
      __syncwarp();  // the row's columns and bits are read before the next row's
      if (in) len = 0;
    }
    // ---- the others: every lane a product, searched in global memory
    const int incl = warp_incl_scan(len);
    const int tot = __shfl_sync(FULL, incl, 31);
    const int excl = incl - len;
    for (int q0 = 0; q0 < tot; q0 += 32) {
      const int q = q0 + lane;
      const int o = warp_owner(incl, q);
      const int os = __shfl_sync(FULL, sb, o);
      const int oex = __shfl_sync(FULL, excl, o);
      const T oa = __shfl_sync(FULL, a, o);
      const int olo = __shfl_sync(FULL, mr0, o), ohi = __shfl_sync(FULL, mr1, o);
      if (q < tot) {
        const int bi = os + q - oex;
        const int j = B.ci[bi];
        const int p = find_in(M.ci, olo, ohi, j);
        if (p >= 0) sr_reduce_global<SR>(&out[p], sr_product<SR>(oa, bv[bi]));
      }
    }
  }
}

// Shared memory of a block of k_masked_rows.
template <typename T>
struct MaskBlock {
  // up to MASK_BLOCK_CAP accumulators and columns, or COLS columns alone
  static constexpr int COLS = MASK_BLOCK_CAP * (int)(sizeof(T) + sizeof(int)) / (int)sizeof(int);
  union {
    struct {
      T acc[MASK_BLOCK_CAP];
      int col[MASK_BLOCK_CAP];
    };
    int only_col[COLS];
  };
  T seg_a[MASK_BLOCK];                                // the list: multiplier,
  unsigned long long pack;                            // (segments << 32) | products,
  int seg_off[MASK_BLOCK], seg_s[MASK_BLOCK];         // stream offset, start in B
  int2 queue[MASK_BLOCK / 32][MASK_BLOCK_QUEUE];            // per warp: (entry of B, segment)
  int row[MASK_BLOCK];                                // row of each nonzero
  int part[MASK_BLOCK / MASK_ROW_MIN + 4], parts;     // first nonzeros of the rows to take
  uint32_t bits[MASK_BLOCK_BITS / 32];
};

// Long rows: a block takes a unit of up to 256 consecutive nonzeros of A and
// one after the other the rows in it that mask_row_blocked names (the other
// parts of such a row are other blocks'; their sums meet in the output).  The
// mask row's columns set bits of a hashed bitmap (the low 16 bits) and are
// listed in shared memory with an accumulator each (up to 1536 columns; up to
// 4608, 3072 in FP32, without accumulators; in global memory beyond).  The
// products of the part are one stream, cut into equal shares for the warps
// (segstream.cuh): rows of B of hundreds of entries and of one weigh the same.
// A product costs its column, one test of the bitmap and a ballot; those that
// pass wait in the warp's queue and are looked up 32 at a time, because an FP64
// product and its addition cost a warp the same with one lane as with all.
//
// What bounds it: the latency of a batch's loads in a warp (four batches in
// flight) in units of hundreds of thousands of products, and about 30
// instructions a batch elsewhere.  R-MAT scale 16: 0.31 ms; 0.35 with a queue
// check after each batch or with 2048 columns (four blocks on an SM instead of
// five), 0.39 without the list for rows beyond the accumulators, 0.35 and 0.41
// with 512 and 128 threads, and no less with the next four loads issued before
// the tests.  Rows from 32 and from 128 nonzeros on: 2 % slower and 5 %.
template <typename T, int SR>
__global__ void __launch_bounds__(MASK_BLOCK, 5)
k_masked_rows(Csr A, Csr B, Csr M, const T* __restrict__ av, const T* __restrict__ bv, T* __restrict__ out,
              int unit) {
  constexpr int NT = MASK_BLOCK;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  MaskBlock<T>& sm = *reinterpret_cast<MaskBlock<T>*>(smem_raw);
  const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
  const unsigned lt = lanemask_lt();
  const int u0 = (int)(unit * (long long)blockIdx.x), u1 = (int)min(A.nnz - u0, (long long)unit);  // u0 + [0, u1)
  // ---- rows of the unit's nonzeros, and the parts to take
  int row = -1, sb = 0, len = 0;
  bool take = false;
  if (warp * 32 < u1) {
    row = warp_row_of(A.rp, (int)A.nrows, u0 + warp * 32);
    if (tid < u1) {
      row = row_from(A.rp, (int)A.nrows, row, u0 + tid);
      take = mask_row_blocked(A.rp[row + 1] - A.rp[row], M.rp[row + 1] - M.rp[row]);
    }
  }
  sm.row[tid] = row;
  if (tid == 0) {
    sm.parts = 0;
    sm.pack = 0ull;
  }
  if (!__syncthreads_or(take)) return;
  if (take && (tid == 0 || sm.row[tid - 1] != row)) {  // (rows of at least MASK_ROW_MIN nonzeros: a few parts)
    const int x = atomicAdd(&sm.parts, 1);
    if (x < MASK_BLOCK / MASK_ROW_MIN + 4) sm.part[x] = tid;
  }
  T a = T(0);
  if (take) {
    const int k = A.ci[u0 + tid];
    if (k >= 0 && (long long)k < B.nrows) {  // a column of A out of range names no row of B
      sb = B.rp[k];
      len = max(B.rp[k + 1] - sb, 0);
      a = av[u0 + tid];
    }
  }
  for (int t = tid; t < MASK_BLOCK_BITS / 32; t += NT) sm.bits[t] = 0u;
  __syncthreads();
  const int parts = min(sm.parts, MASK_BLOCK / MASK_ROW_MIN + 4);
  int2* const queue = sm.queue[warp];
  for (int x = 0; x < parts; ++x) {
    const int i = sm.row[sm.part[x]];
    const int m0 = M.rp[i], n = M.rp[i + 1] - m0;
    const bool staged = n <= MASK_BLOCK_CAP;  // accumulators; products go to the output otherwise
    const bool listed = n <= MaskBlock<T>::COLS;
    int* const cols = staged ? sm.col : sm.only_col;
    for (int t = tid; t < n; t += NT) {
      const int c = M.ci[m0 + t];
      atomicOr(&sm.bits[(c >> 5) & (MASK_BLOCK_BITS / 32 - 1)], 1u << (c & 31));
      if (listed) cols[t] = c;
      if (staged) sm.acc[t] = sr_zero<SR, T>();
    }
    int rest = take && row == i ? len : 0;
    do {  // one round, but for rows of B of millions of entries
      const int now = min(rest, MASK_ROUND);
      seg_append<T>(&sm.pack, sb, now, a, sm.seg_off, sm.seg_s, sm.seg_a);
      rest -= now;
      sb += now;
      __syncthreads();  // the list and the mask are complete
      const int nseg = (int)(sm.pack >> 32), tot = (int)(unsigned)(sm.pack & 0xffffffffull);
      const int share = ((tot + NT - 1) / NT) * 32;
      const int lo = warp * share, hi = min(tot, lo + share);
      int qn = 0;  // waiting products
      auto look_up = [&](int cnt) {  // the last cnt (at most 32) of the queue
        if (lane < cnt) {
          const int2 w = queue[qn - cnt + lane];
          const int j = B.ci[w.x];
          const T b = bv[w.x];
          const int p = listed ? find_in(cols, 0, n, j) : find_in(M.ci + m0, 0, n, j);
          if (p >= 0) {
            const T x = sr_product<SR>(sm.seg_a[w.y], b);
            if (staged) sr_reduce_shared<SR>(&sm.acc[p], x);
            else sr_reduce_global<SR>(&out[m0 + p], x);
          }
        }
        qn -= cnt;
        __syncwarp();  // the entries are read before later ones overwrite them
      };
      auto offer = [&](int j, int bi, int k, bool act) {
        const bool pass = act && (sm.bits[(j >> 5) & (MASK_BLOCK_BITS / 32 - 1)] >> (j & 31) & 1u);
        const unsigned b = __ballot_sync(FULL, pass);
        if (!b) return;
        if (pass) queue[qn + __popc(b & lt)] = make_int2(bi, k);
        qn += __popc(b);
        __syncwarp();
        if (qn >= 32) look_up(32);
      };
      if (lo < hi) {
        int f = seg_find(sm.seg_off, nseg, lo);
        int p = lo;
        while (p < hi) {
          const int so = sm.seg_off[f];
          const int se = f + 1 < nseg ? sm.seg_off[f + 1] : tot;
          const int run = min(se, hi) - p;
          if (run >= 32) {  // whole batches inside segment f, four loads in flight
            const int nw = run & ~31;
            const int q = sm.seg_s[f] + (p - so) + lane;
            const int* __restrict__ ci = B.ci + q;
            int t = 0;
            for (; t + 96 < nw; t += 128) {
              const int j[4] = {ci[t], ci[t + 32], ci[t + 64], ci[t + 96]};
              bool pass[4];
              unsigned b[4];
#pragma unroll
              for (int v = 0; v < 4; ++v) {
                pass[v] = sm.bits[(j[v] >> 5) & (MASK_BLOCK_BITS / 32 - 1)] >> (j[v] & 31) & 1u;
                b[v] = __ballot_sync(FULL, pass[v]);
              }
              if (!(b[0] | b[1] | b[2] | b[3])) continue;
#pragma unroll
              for (int v = 0; v < 4; ++v) {
                if (pass[v]) queue[qn + __popc(b[v] & lt)] = make_int2(q + t + 32 * v, f);
                qn += __popc(b[v]);
              }
              __syncwarp();
              while (qn >= 32) look_up(32);
            }
            for (; t < nw; t += 32) offer(ci[t], q + t, f, true);
            p += nw;
            if (p == se) ++f;
            continue;
          }
          // one batch across segments: lane j holds the end of segment f + j
          const int nx = f + lane + 1;
          const int end = nx < nseg ? sm.seg_off[nx] : (nx == nseg ? tot : INT_MAX);
          const int d = end == INT_MAX ? INT_MAX : end - p;
          const unsigned m = __reduce_or_sync(FULL, d <= 31 ? (1u << d) : 0u);
          const int k = f + __popc(m & (lane == 31 ? FULL : ((2u << lane) - 1u)));
          const int q = p + lane;
          const bool act = q < hi;
          const int bi = act ? sm.seg_s[k] + (q - sm.seg_off[k]) : 0;
          offer(act ? B.ci[bi] : 0, bi, k, act);
          const int pn = p + 32;
          if (pn < hi) {  // segment of the next product
            const int c = __popc(__ballot_sync(FULL, end <= pn));
            f = c < 32 ? f + c : seg_find(sm.seg_off, nseg, pn);
          }
          p = pn;
        }
        if (qn > 0) look_up(qn);
      }
      __syncthreads();  // all products in; the list may be refilled
      if (tid == 0) sm.pack = 0ull;
    } while (__syncthreads_or(rest > 0));
    // (the barrier above: every accumulator is final)
    for (int t = tid; t < n; t += NT) {
      const int c = listed ? cols[t] : M.ci[m0 + t];
      sm.bits[(c >> 5) & (MASK_BLOCK_BITS / 32 - 1)] = 0u;
      if (staged) sr_reduce_global<SR>(&out[m0 + t], sm.acc[t]);
    }
    __syncthreads();  // the next row's columns and bits come after
  }
}

// out[p] *= mv[p] for the nnz(M) entries.
template <typename T>
__global__ void __launch_bounds__(256) k_scale(T* __restrict__ out, const T* __restrict__ mv, long long n) {
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x)
    out[p] = out[p] * mv[p];
}

// out[p] = the semiring's zero (+inf or -inf) for the nnz(M) entries.
template <typename T, int SR>
__global__ void __launch_bounds__(256) k_fill_zero(T* __restrict__ out, long long n) {
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x)
    out[p] = sr_zero<SR, T>();
}

template <typename T, int SR>
static cudaError_t masked_t(const LaunchCtx& c, const Csr& A, const Csr& B, const Csr& M, const T* av, const T* bv,
                            const T* mv, T* out) {
  const long long blocks = (M.nnz + 255) / 256;
  const int eg = (int)(blocks < 4096 ? blocks : 4096);
  cudaError_t e;
  if (SR == 1 || SR == 2) {
    k_fill_zero<T, SR><<<eg, 256, 0, c.stream>>>(out, M.nnz);
    count_launch(c);
    e = cudaGetLastError();
  } else {
    e = cudaMemsetAsync(out, 0, sizeof(T) * (size_t)M.nnz, c.stream);
  }
  if (e != cudaSuccess || A.nnz <= 0) return e;
  auto k = k_masked<T, SR>;
  // A mask with more than twice A's entries has few rows that blocks take: its
  // long rows stay with the warps, and looking for such rows is saved (the 96^3
  // stencil with its square's pattern, min-plus: 1.04 -> 0.94 ms).
  const bool long_rows = M.nnz <= 2 * A.nnz;
  if (long_rows) {
    auto kr = k_masked_rows<T, SR>;
    if (kernel_blocks_per_sm(kr, MASK_BLOCK, sizeof(MaskBlock<T>)) <= 0) return cudaErrorInvalidConfiguration;
    // smaller units where few would be left for the SMs: 3000 rows 68 -> 49 us
    int unit = MASK_BLOCK;
    while (unit > 32 && A.nnz < (long long)MASK_UNITS_PER_SM * c.nsm * unit) unit >>= 1;
    kr<<<(unsigned)((A.nnz + unit - 1) / unit), MASK_BLOCK, sizeof(MaskBlock<T>), c.stream>>>(A, B, M, av, bv, out,
                                                                                          unit);
    count_launch(c);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  const long long per_block = 32 * MASK_WARPS;
  k<<<(unsigned)((A.nnz + per_block - 1) / per_block), MASK_WARPS * 32, 0, c.stream>>>(A, B, M, av, bv, out, long_rows);
  count_launch(c);
  if ((e = cudaGetLastError()) != cudaSuccess || SR != 0 || !mv) return e;
  k_scale<T><<<eg, 256, 0, c.stream>>>(out, mv, M.nnz);
  count_launch(c);
  return cudaGetLastError();
}

cudaError_t launch_masked(const LaunchCtx& c, int dtype, int semiring, const Csr& A, const Csr& B, const Csr& M,
                          const void* av, const void* bv, const void* mv, void* out) {
  if (M.nrows <= 0 || M.nnz <= 0) return cudaSuccess;
  auto run = [&](auto* tag) -> cudaError_t {
    using T = std::remove_pointer_t<decltype(tag)>;
    const T* a = (const T*)av;
    const T* b = (const T*)bv;
    T* o = (T*)out;
    switch (semiring) {
      case 1: return masked_t<T, 1>(c, A, B, M, a, b, nullptr, o);
      case 2: return masked_t<T, 2>(c, A, B, M, a, b, nullptr, o);
      case 3: return masked_t<T, 3>(c, A, B, M, a, b, nullptr, o);
      default: return masked_t<T, 0>(c, A, B, M, a, b, (const T*)mv, o);
    }
  };
  return dtype == SPGEMM_F32 ? run((float*)nullptr) : run((double*)nullptr);
}

}  // namespace sg
