// Batched products C_i = A_i * B_i.
//
// The instances are stacked into one block-diagonal product
//   diag(A_1, ..., A_n) * diag(B_1, ..., B_n) = diag(A_1 B_1, ..., A_n B_n),
// so a single analysis bins the rows of all instances together and each pass
// (symbolic, numeric) is one persistent launch per path over that global
// (instance, row) work list, largest rows first.  Instance i's rows of A sit
// at row offset roff_i and its columns (rows of B) at koff_i.  Columns of B
// and C keep each instance's own numbering: a row of C only meets rows of B
// of its own instance, so the instances' column ranges may overlap and C
// comes out with the instances' columns as they are.  These kernels build the
// stacked index arrays once and gather the instances' values before each
// numeric pass.
//
// All of them are copies bound by memory, over instances whose sizes differ
// by orders of magnitude, so the work is cut into equal chunks of the stacked
// arrays and each thread finds its instance from the stacked offsets.  (A
// fixed number of blocks per instance left the largest instances with a few
// blocks: 64 instances of 1,024 to 50,000 rows, 553 M products, took 0.55 ms
// for the structure, 0.60 ms for the values and 0.38 ms for the products, and
// 8.9 ms for a pass that shifted C's columns back from a stacked numbering;
// the whole call went from 24.8 to 14.1 ms.)
#include "launch_util.cuh"

namespace sg {

constexpr int STACK_THREADS = 256;
constexpr int STACK_ITEMS = 8;                              // entries per thread and chunk
constexpr long long STACK_CHUNK = STACK_THREADS * STACK_ITEMS;

static long long stack_chunks(long long n) { return (n + STACK_CHUNK - 1) / STACK_CHUNK; }

// Last instance whose offset (its member `off` of the descriptor) is <= p.
__device__ __forceinline__ int instance_at(const BatchDesc* __restrict__ d, int n, long long BatchDesc::*off,
                                           long long p) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (d[mid].*off <= p) lo = mid; else hi = mid;
  }
  return lo;
}

// out[off_i + q] = add_i + in_i[q] over one chunk of the stacked array
// (total entries); `in` is the instance's array, `add` gives add_i.  The loads
// of a thread's entries are issued together.
template <typename T, typename In, typename Add>
__device__ __forceinline__ void stack_chunk(const BatchDesc* __restrict__ d, int n, long long BatchDesc::*off,
                                            long long chunk, long long total, T* __restrict__ out, In in, Add add) {
  const long long p0 = chunk * STACK_CHUNK + threadIdx.x;
  if (p0 >= total) return;
  int i = instance_at(d, n, off, p0);
  T v[STACK_ITEMS];
#pragma unroll
  for (int u = 0; u < STACK_ITEMS; ++u) {
    const long long p = p0 + u * STACK_THREADS;
    if (p < total) {
      while (i + 1 < n && d[i + 1].*off <= p) ++i;
      v[u] = in(d[i])[p - d[i].*off] + add(d[i]);
    }
  }
#pragma unroll
  for (int u = 0; u < STACK_ITEMS; ++u) {
    const long long p = p0 + u * STACK_THREADS;
    if (p < total) out[p] = v[u];
  }
}

// Chunks of the four stacked index arrays one after another: A's row
// pointers, A's columns, B's row pointers, B's columns.
__global__ void __launch_bounds__(STACK_THREADS)
k_stack_structure(const BatchDesc* __restrict__ d, int n, int32_t* __restrict__ a_rp, int32_t* __restrict__ a_ci,
                  int32_t* __restrict__ b_rp, int32_t* __restrict__ b_ci, long long total_rows, long long total_a_nnz,
                  long long total_k, long long total_b_nnz, long long c0, long long c1, long long c2) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // closing row pointers
    a_rp[total_rows] = (int32_t)total_a_nnz;
    b_rp[total_k] = (int32_t)total_b_nnz;
  }
  const long long c = blockIdx.x;
  if (c < c0)
    stack_chunk(d, n, &BatchDesc::roff, c, total_rows, a_rp, [](const BatchDesc& D) { return D.a_rp; },
                [](const BatchDesc& D) { return (int32_t)D.aoff; });
  else if (c < c1)
    stack_chunk(d, n, &BatchDesc::aoff, c - c0, total_a_nnz, a_ci, [](const BatchDesc& D) { return D.a_ci; },
                [](const BatchDesc& D) { return (int32_t)D.koff; });
  else if (c < c2)
    stack_chunk(d, n, &BatchDesc::koff, c - c1, total_k, b_rp, [](const BatchDesc& D) { return D.b_rp; },
                [](const BatchDesc& D) { return (int32_t)D.boff; });
  else
    stack_chunk(d, n, &BatchDesc::boff, c - c2, total_b_nnz, b_ci, [](const BatchDesc& D) { return D.b_ci; },
                [](const BatchDesc&) { return 0; });
}

// Columns of every instance inside its own matrices: the stacked arrays alone
// allow B_i the columns of the widest instance, and A_i the rows of the next
// instance's B.  Chunks of A's entries, then of B's (only with opts.validate).
__global__ void __launch_bounds__(STACK_THREADS)
k_batch_validate(const BatchDesc* __restrict__ d, int n, long long total_a_nnz, long long total_b_nnz, long long c0,
                 uint32_t* err) {
  const bool b = blockIdx.x >= c0;
  const long long p0 = (b ? blockIdx.x - c0 : (long long)blockIdx.x) * STACK_CHUNK + threadIdx.x;
  const long long total = b ? total_b_nnz : total_a_nnz;
  long long BatchDesc::*const off = b ? &BatchDesc::boff : &BatchDesc::aoff;
  if (p0 >= total) return;
  int i = instance_at(d, n, off, p0);
  bool bad = false;
  for (int u = 0; u < STACK_ITEMS; ++u) {
    const long long p = p0 + u * STACK_THREADS;
    if (p >= total) break;
    while (i + 1 < n && d[i + 1].*off <= p) ++i;
    const int c = (b ? d[i].b_ci : d[i].a_ci)[p - d[i].*off];
    bad |= c < 0 || (long long)c >= (b ? d[i].n : d[i].k);
  }
  if (bad) atomicOr(err, EB_UNSORTED);
}

cudaError_t launch_batch_validate(const LaunchCtx& c, int n, const BatchDesc* d, long long total_a_nnz,
                                  long long total_b_nnz) {
  const long long c0 = stack_chunks(total_a_nnz), blocks = c0 + stack_chunks(total_b_nnz);
  if (n <= 0 || blocks <= 0) return cudaSuccess;
  k_batch_validate<<<(unsigned)blocks, STACK_THREADS, 0, c.stream>>>(d, n, total_a_nnz, total_b_nnz, c0, c.err);
  count_launch(c);
  return cudaGetLastError();
}

// V: an unsigned type of the values' width (the values are only moved).
template <typename V>
__global__ void __launch_bounds__(STACK_THREADS)
k_stack_values(const BatchDesc* __restrict__ d, int n, V* __restrict__ a_v, V* __restrict__ b_v, long long total_a_nnz,
               long long total_b_nnz, long long c0) {
  const long long c = blockIdx.x;
  if (c < c0)
    stack_chunk(d, n, &BatchDesc::aoff, c, total_a_nnz, a_v, [](const BatchDesc& D) { return (const V*)D.a_v; },
                [](const BatchDesc&) { return V(0); });
  else
    stack_chunk(d, n, &BatchDesc::boff, c - c0, total_b_nnz, b_v, [](const BatchDesc& D) { return (const V*)D.b_v; },
                [](const BatchDesc&) { return V(0); });
}

cudaError_t launch_stack_structure(const LaunchCtx& c, int n, const BatchDesc* d, long long total_rows,
                                   long long total_k, int32_t* a_rp, int32_t* a_ci, int32_t* b_rp, int32_t* b_ci,
                                   long long total_a_nnz, long long total_b_nnz) {
  if (n <= 0) return cudaSuccess;
  const long long c0 = stack_chunks(total_rows), c1 = c0 + stack_chunks(total_a_nnz), c2 = c1 + stack_chunks(total_k);
  long long blocks = c2 + stack_chunks(total_b_nnz);
  if (blocks < 1) blocks = 1;  // the closing row pointers
  k_stack_structure<<<(unsigned)blocks, STACK_THREADS, 0, c.stream>>>(d, n, a_rp, a_ci, b_rp, b_ci, total_rows,
                                                                     total_a_nnz, total_k, total_b_nnz, c0, c1, c2);
  count_launch(c);
  return cudaGetLastError();
}

cudaError_t launch_stack_values(const LaunchCtx& c, int n, int dtype, const BatchDesc* d, void* a_v, void* b_v,
                                long long total_a_nnz, long long total_b_nnz) {
  const long long c0 = stack_chunks(total_a_nnz), blocks = c0 + stack_chunks(total_b_nnz);
  if (n <= 0 || blocks <= 0) return cudaSuccess;
  if (dtype == SPGEMM_F32)
    k_stack_values<unsigned><<<(unsigned)blocks, STACK_THREADS, 0, c.stream>>>(d, n, (unsigned*)a_v, (unsigned*)b_v,
                                                                              total_a_nnz, total_b_nnz, c0);
  else
    k_stack_values<unsigned long long><<<(unsigned)blocks, STACK_THREADS, 0, c.stream>>>(
        d, n, (unsigned long long*)a_v, (unsigned long long*)b_v, total_a_nnz, total_b_nnz, c0);
  count_launch(c);
  return cudaGetLastError();
}

// c_rp at each instance's first row (and the end): per-instance nnz on the host.
__global__ void k_batch_bounds(const BatchDesc* __restrict__ d, int n, const int32_t* __restrict__ c_rp,
                               long long total_rows, int32_t* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += gridDim.x * blockDim.x)
    out[i] = c_rp[i < n ? d[i].roff : total_rows];
}

cudaError_t launch_batch_bounds(const LaunchCtx& c, int n, const BatchDesc* d, const int32_t* c_rp, long long total_rows,
                                int32_t* out) {
  k_batch_bounds<<<(n + 256) / 256, 256, 0, c.stream>>>(d, n, c_rp, total_rows, out);
  count_launch(c);
  return cudaGetLastError();
}

// Per-instance product counts: products[i] += sum over A_i's nonzeros (r,k)
// of nnz(B_i(k,:)), over chunks of the instances' nonzeros laid end to end
// (offsets aoff).  Threads of a chunk inside one instance reduce in the block
// and add once; a chunk over a boundary adds per thread and instance.
__global__ void __launch_bounds__(STACK_THREADS) k_batch_products(const BatchDesc* __restrict__ d, int n,
                                                                 long long total,
                                                                 unsigned long long* __restrict__ products) {
  __shared__ unsigned long long s_part[STACK_THREADS / 32];
  const long long first = blockIdx.x * STACK_CHUNK;
  const long long last = (first + STACK_CHUNK < total ? first + STACK_CHUNK : total) - 1;
  const int i0 = instance_at(d, n, &BatchDesc::aoff, first);
  const bool one = last < d[i0].aoff + d[i0].a_nnz;  // block-uniform
  int i = i0;
  unsigned long long sum = 0;
  for (int u = 0; u < STACK_ITEMS; ++u) {
    const long long p = first + threadIdx.x + u * STACK_THREADS;
    if (p > last) break;
    if (!one && d[i].aoff + d[i].a_nnz <= p) {
      if (sum) atomicAdd(&products[i], sum);
      sum = 0;
      while (d[i].aoff + d[i].a_nnz <= p) ++i;
    }
    const int k = d[i].a_ci[p - d[i].aoff];
    sum += (unsigned long long)(d[i].b_rp[k + 1] - d[i].b_rp[k]);
  }
  if (!one) {
    if (sum) atomicAdd(&products[i], sum);
    return;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(FULL, sum, o);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long tot = 0;
    for (int w = 0; w < STACK_THREADS / 32; ++w) tot += s_part[w];
    if (tot) atomicAdd(&products[i0], tot);
  }
}

cudaError_t launch_batch_products(const LaunchCtx& c, int n, const BatchDesc* d, long long total_a_nnz,
                                  long long* products) {
  if (n <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(products, 0, sizeof(long long) * (size_t)n, c.stream);
  if (e != cudaSuccess || total_a_nnz <= 0) return e;
  k_batch_products<<<(unsigned)stack_chunks(total_a_nnz), STACK_THREADS, 0, c.stream>>>(
      d, n, total_a_nnz, (unsigned long long*)products);
  count_launch(c);
  return cudaGetLastError();
}

}  // namespace sg
