// Sum and product of the numeric pass.  Row i of C is the sum over the
// nonzeros A(i,k) of A(i,k) * B(k,:) (Sec. 2.2); the same row-wise step
// computes a product over another semiring when + and * are replaced:
// min-plus (shortest paths), max-plus (longest paths) and or-and
// (reachability).  Min and max do not depend on the order of their
// operands, so those products are exact.
//
// Each policy gives the sum's identity (the cleared state of an
// accumulator word), the product, the sum, their fusion acc (+) a (*) b, what
// an accumulator holds after its first product (first: the product itself, but
// in min-plus and max-plus the identity where the product is not a number, so
// that a NaN counts for nothing whichever product comes first), and
// shared-memory updates that other lanes may race with: red_value (*p (+)=
// x), red_shared (*p (+)= a (*) b) and madd_shared (the same, returning
// whether the word still held the identity when read, i.e. whether this may
// be the column's first product).
#pragma once

#include "internal.cuh"

namespace sg {

__device__ __forceinline__ unsigned long long sr_bits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ unsigned sr_bits(float v) { return __float_as_uint(v); }

template <typename T> __device__ __forceinline__ T sr_inf();
template <> __device__ __forceinline__ double sr_inf<double>() { return __longlong_as_double(0x7ff0000000000000ll); }
template <> __device__ __forceinline__ float sr_inf<float>() { return __int_as_float(0x7f800000); }

__device__ __forceinline__ unsigned long long sr_cas(double* p, unsigned long long old, unsigned long long nv) {
  return atomicCAS(reinterpret_cast<unsigned long long*>(p), old, nv);
}
__device__ __forceinline__ unsigned sr_cas(float* p, unsigned old, unsigned nv) {
  return atomicCAS(reinterpret_cast<unsigned*>(p), old, nv);
}

// *p = min(*p, x) (MIN) or max(*p, x) by compare-and-swap, written only
// when x improves the word; returns whether the word held `zero` when read.
template <bool MIN, typename T>
__device__ __forceinline__ bool minmax_shared(T* p, T x, T zero, uint32_t* err) {
  T old = *reinterpret_cast<volatile T*>(p);
  const bool first = sr_bits(old) == sr_bits(zero);
  for (int it = 0; it < CAS_RETRY_LIMIT; ++it) {
    if (MIN ? !(x < old) : !(x > old)) return first;
    const auto prev = sr_cas(p, sr_bits(old), sr_bits(x));
    if (prev == sr_bits(old)) return first;
    if (sizeof(T) == 8) old = __longlong_as_double((long long)prev);
    else old = __uint_as_float((unsigned)prev);
  }
  atomicOr(err, EB_INTERNAL);  // never expected: each failed swap is another update's improvement
  return first;
}

template <typename T, int SR> struct SrOps;

// A product that its lane holds in registers until its place in a row is
// known: the value, or in FP32 plus-times both factors, so that a product that
// meets another is fused into the sum.  (Rounded first it made small FP32
// products 9 to 15 % less exact than the lane tables and windows that such rows
// took before, grid operators and 700 rows of 30 to 60 products alike.  In FP64
// the factors cost k_num_once 8 % -- 64 products of 1,024 to 50,000 rows 6.7 and
// 7.3 ms -- for 7 to 14 % of an error below one unit of the last place.)
template <typename T, int SR> struct HeldProduct {
  T x;
  __device__ HeldProduct() : x(T(0)) {}
  __device__ void set(T a, T b) { x = SrOps<T, SR>::mul(a, b); }
  __device__ T first() const { return SrOps<T, SR>::first(x); }
};
template <> struct HeldProduct<float, SPGEMM_PLUS_TIMES> {
  float a, b;
  __device__ HeldProduct() : a(0.f), b(0.f) {}
  __device__ void set(float x, float y) { a = x; b = y; }
  __device__ float first() const { return a * b; }
};

// acc[at[u]] (+)= p[u] for the at[u] >= 0, G products in flight at a time where
// they are fused (all of a row's in a warp's table, where many meet: 18.2 and 17.6
// us for two products of a small Galerkin chain; one in block registers, where
// four take 9 % longer on a 27-point stencil).
template <int G, typename T, int SR, int N>
__device__ __forceinline__ void add_held(const HeldProduct<T, SR> (&p)[N], T* acc, const int (&at)[N], uint32_t* err) {
#pragma unroll
  for (int u = 0; u < N; ++u)
    if (at[u] >= 0) SrOps<T, SR>::red_value(&acc[at[u]], p[u].x, err);
}
template <int G, int N>
__device__ __forceinline__ void add_held(const HeldProduct<float, SPGEMM_PLUS_TIMES> (&p)[N], float* acc,
                                         const int (&at)[N], uint32_t* err) {
  static_assert(N % G == 0, "whole groups");
#pragma unroll
  for (int g = 0; g < N; g += G) {
    float a[G], b[G];
    int x[G];
#pragma unroll
    for (int u = 0; u < G; ++u) {
      a[u] = p[g + u].a;
      b[u] = p[g + u].b;
      x[u] = at[g + u];
    }
    fma_shared_cas(acc, a, b, x, err);
  }
}

template <typename T> struct SrOps<T, SPGEMM_PLUS_TIMES> {
  __device__ static T zero() { return T(0); }
  __device__ static bool cleared(T v) { return is_cleared(v); }
  __device__ static T mul(T a, T b) { return a * b; }
  __device__ static T first(T x) { return x; }
  __device__ static T add(T x, T y) { return x + y; }
  __device__ static T madd(T a, T b, T acc) { return fma(a, b, acc); }
  __device__ static void red_value(T* p, T x, uint32_t*) { red_add_shared(p, x); }
  __device__ static void red_shared(T* p, T a, T b, uint32_t*) { red_add_shared(p, a * b); }
  __device__ static bool madd_shared(T* p, T a, T b, uint32_t* err) { return fma_shared(p, a, b, err); }
};

template <typename T> struct SrOps<T, SPGEMM_MIN_PLUS> {
  __device__ static T zero() { return sr_inf<T>(); }
  __device__ static bool cleared(T v) { return sr_bits(v) == sr_bits(zero()); }
  __device__ static T mul(T a, T b) { return a + b; }
  __device__ static T add(T x, T y) { return y < x ? y : x; }
  __device__ static T first(T x) { return add(zero(), x); }
  __device__ static T madd(T a, T b, T acc) { return add(acc, a + b); }
  __device__ static void red_value(T* p, T x, uint32_t* err) { minmax_shared<true>(p, x, zero(), err); }
  __device__ static void red_shared(T* p, T a, T b, uint32_t* err) { minmax_shared<true>(p, a + b, zero(), err); }
  __device__ static bool madd_shared(T* p, T a, T b, uint32_t* err) {
    return minmax_shared<true>(p, a + b, zero(), err);
  }
};

template <typename T> struct SrOps<T, SPGEMM_MAX_PLUS> {
  __device__ static T zero() { return -sr_inf<T>(); }
  __device__ static bool cleared(T v) { return sr_bits(v) == sr_bits(zero()); }
  __device__ static T mul(T a, T b) { return a + b; }
  __device__ static T add(T x, T y) { return y > x ? y : x; }
  __device__ static T first(T x) { return add(zero(), x); }
  __device__ static T madd(T a, T b, T acc) { return add(acc, a + b); }
  __device__ static void red_value(T* p, T x, uint32_t* err) { minmax_shared<false>(p, x, zero(), err); }
  __device__ static void red_shared(T* p, T a, T b, uint32_t* err) { minmax_shared<false>(p, a + b, zero(), err); }
  __device__ static bool madd_shared(T* p, T a, T b, uint32_t* err) {
    return minmax_shared<false>(p, a + b, zero(), err);
  }
};

template <typename T> struct SrOps<T, SPGEMM_OR_AND> {
  __device__ static T zero() { return T(0); }
  __device__ static bool cleared(T v) { return is_cleared(v); }
  __device__ static T mul(T a, T b) { return (a != T(0) && b != T(0)) ? T(1) : T(0); }
  __device__ static T first(T x) { return x; }
  __device__ static T add(T x, T y) { return (x != T(0) || y != T(0)) ? T(1) : T(0); }
  __device__ static T madd(T a, T b, T acc) { return add(acc, mul(a, b)); }
  // every writer stores the same 1, so racing stores need no atomics
  __device__ static void red_value(T* p, T x, uint32_t*) {
    if (x != T(0)) *reinterpret_cast<volatile T*>(p) = T(1);
  }
  __device__ static void red_shared(T* p, T a, T b, uint32_t*) {
    if (a != T(0) && b != T(0)) *reinterpret_cast<volatile T*>(p) = T(1);
  }
  __device__ static bool madd_shared(T* p, T a, T b, uint32_t*) {
    const T old = *reinterpret_cast<volatile T*>(p);
    if (a != T(0) && b != T(0) && old == T(0)) *reinterpret_cast<volatile T*>(p) = T(1);
    return is_cleared(old);
  }
};

}  // namespace sg
