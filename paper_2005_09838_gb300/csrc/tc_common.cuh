// Shared device types and helpers of the TCTF2R CUDA library.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <type_traits>

namespace tc {

// Static shared memory the library's kernels declare (block reductions) is at
// most this; sizes of dynamic shared memory are checked against the opt-in
// limit less it.
constexpr int kStaticSmemReserve = 2048;

// The dynamic shared-memory limit is an attribute of the kernel itself, shared
// by every live context that launches it: raise it to `bytes` if it is lower,
// never lower it (a smaller context created later must not break the launches
// of a larger one).
inline cudaError_t allow_dynamic_smem(const void* f, size_t bytes) {
  static std::mutex m;
  std::lock_guard<std::mutex> g(m);
  cudaFuncAttributes a{};
  cudaError_t e = cudaFuncGetAttributes(&a, f);
  if (e != cudaSuccess) return e;
  if ((size_t)a.maxDynamicSharedSizeBytes >= bytes) return cudaSuccess;
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Complex value in (re, im) order; layout-compatible with float2 / double2.
template <typename T>
struct alignas(2 * sizeof(T)) cx {
  T re, im;
};

template <typename T>
__host__ __device__ __forceinline__ cx<T> mk(T a, T b) { return cx<T>{a, b}; }
template <typename T>
__host__ __device__ __forceinline__ cx<T> operator+(cx<T> a, cx<T> b) { return {a.re + b.re, a.im + b.im}; }
template <typename T>
__host__ __device__ __forceinline__ cx<T> operator-(cx<T> a, cx<T> b) { return {a.re - b.re, a.im - b.im}; }
template <typename T>
__host__ __device__ __forceinline__ cx<T> operator*(cx<T> a, T s) { return {a.re * s, a.im * s}; }
template <typename T>
__host__ __device__ __forceinline__ cx<T> cmul(cx<T> a, cx<T> b) {
  return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
// a * conj(b)
template <typename T>
__host__ __device__ __forceinline__ cx<T> cmulc(cx<T> a, cx<T> b) {
  return {a.re * b.re + a.im * b.im, a.im * b.re - a.re * b.im};
}
// conj(a) * b
template <typename T>
__host__ __device__ __forceinline__ cx<T> cconjmul(cx<T> a, cx<T> b) {
  return {a.re * b.re + a.im * b.im, a.re * b.im - a.im * b.re};
}
template <typename T>
__host__ __device__ __forceinline__ cx<T> conj(cx<T> a) { return {a.re, -a.im}; }
// acc += a * b
template <typename T>
__host__ __device__ __forceinline__ void cfma(cx<T>& acc, cx<T> a, cx<T> b) {
  acc.re = fma(a.re, b.re, acc.re);
  acc.re = fma(-a.im, b.im, acc.re);
  acc.im = fma(a.re, b.im, acc.im);
  acc.im = fma(a.im, b.re, acc.im);
}
// acc += a * conj(b)
template <typename T>
__host__ __device__ __forceinline__ void cfmac(cx<T>& acc, cx<T> a, cx<T> b) {
  acc.re = fma(a.re, b.re, acc.re);
  acc.re = fma(a.im, b.im, acc.re);
  acc.im = fma(a.im, b.re, acc.im);
  acc.im = fma(-a.re, b.im, acc.im);
}
// acc += conj(a) * b
template <typename T>
__host__ __device__ __forceinline__ void cfmaconj(cx<T>& acc, cx<T> a, cx<T> b) {
  acc.re = fma(a.re, b.re, acc.re);
  acc.re = fma(a.im, b.im, acc.re);
  acc.im = fma(a.re, b.im, acc.im);
  acc.im = fma(-a.im, b.re, acc.im);
}

// |a|
template <typename T>
__host__ __device__ __forceinline__ T cabs(cx<T> a) {
  return sqrt(a.re * a.re + a.im * a.im);
}

// Read-only cached load of a complex value.
__device__ __forceinline__ cx<float> ldg_cx(const cx<float>* p) {
  const float2 v = __ldg(reinterpret_cast<const float2*>(p));
  return {v.x, v.y};
}
__device__ __forceinline__ cx<double> ldg_cx(const cx<double>* p) {
  const double2 v = __ldg(reinterpret_cast<const double2*>(p));
  return {v.x, v.y};
}

// Device error word (first error wins).  Kernels record a code and return
// instead of trapping, so the context stays usable.
enum DevErr : int {
  DEV_OK = 0,
  DEV_BAD_LAUNCH = 1,   // launch shape does not match the sizes
  DEV_BAD_SIZE = 2,     // size outside what a kernel instance supports
  DEV_NONFINITE = 3,    // a non-finite value where a finite one is required
  DEV_TIMEOUT = 4,      // a bounded wait on the tensor core gave up
};

__device__ __forceinline__ void set_err(int* err, int code) {
  if (err) atomicCAS(err, 0, code);
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 1/a.  FP64: a correctly rounded FP32 seed and two Newton steps
// y <- y (2 - a y) (the error squares at each step); FP64 division is slow on
// this part.  FP32: the IEEE quotient.
__device__ __forceinline__ double rcp_refined(double a) {
  const float af = (float)a;
  if (!(fabsf(af) > 1e-30f && fabsf(af) < 1e30f)) return 1.0 / a;
  double y = (double)__frcp_rn(af);
  y = y * fma(-a, y, 2.0);
  y = y * fma(-a, y, 2.0);
  return y;
}
__device__ __forceinline__ float rcp_refined(float a) { return 1.0f / a; }

// s + c += a b with the rounding errors of the product (FMA) and of the sum
// (Knuth's two-sum) collected in c: about twice the working precision.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

template <typename T>
__device__ __forceinline__ void dot2(T& s, T& c, T a, T b) {
  const T p = mul_rn(a, b);  // not contracted: the FMA below recovers its rounding error
  const T pe = fma(a, b, -p);
  const T t = s + p;
  const T z = t - s;
  c += ((s - (t - z)) + (p - z)) + pe;
  s = t;
}

// (s, c) += (s2, c2) for sums kept as value and collected rounding errors.
template <typename T>
__device__ __forceinline__ void pair_add(T& s, T& c, T s2, T c2) {
  const T t = s + s2;
  const T z = t - s;
  c += ((s - (t - z)) + (s2 - z)) + c2;
  s = t;
}

// (s, e) <- s + a and the rounding error of it (Knuth's two-sum).
__device__ __forceinline__ float two_sum(float& s, float a) {
  const float t = s + a, z = t - s, e = (s - (t - z)) + (a - z);
  s = t;
  return e;
}

// Sum of squares of a thread's values, no less accurate than FP64 additions.  FP32: every
// square is taken with its rounding error and added without one to three FP32 words
// (error some 2^-70 of the sum), on the FP32 pipe; GB300 issues one FP64 warp
// instruction per scheduler in about 60 clocks, and an FP64 conversion and
// multiply-add per value took more than half of the read-back kernels.  Squares past
// FP32's range make the sum infinite or NaN, and squares or rounding errors below it
// are at most 2^-149 each, so the block's sum tells whether it stands (sq_again); where
// it does not, the kernel sums its block again with SqSum64.  (Objective of 144 x 288 x
// 168 147 us, gradient call of 300 x 150 x 92 130, of 529 x 288 x 168 427; with every value
// tested and the far ones added in FP64 on the spot 161, 137, 430; with one error word,
// which keeps 2^-43 of a long sum and fails outside 2^+-63, 135, 130, 414.)
template <typename T>
struct SqSum {
  T s = T(0);
  __device__ __forceinline__ void add(T v) { s = fma(v, v, s); }
  __device__ __forceinline__ void add_diff(T a, T b) { add(a - b); }
  __device__ __forceinline__ bool nonzero() const { return false; }
  __device__ __forceinline__ double total() const { return s; }
};
template <>
struct SqSum<float> {
  float s = 0.f, c = 0.f, e = 0.f;
  unsigned any = 0;  // bits of the values
  __device__ __forceinline__ void term(float a) { e += two_sum(c, a); }  // a: of the size of a rounding error
  __device__ __forceinline__ void add(float v) {
    any |= __float_as_uint(v);
    const float p = mul_rn(v, v), pe = fmaf(v, v, -p);
    term(two_sum(s, p));
    term(pe);
  }
  // (a - b)^2 of the difference as it is, not rounded: h + z
  __device__ __forceinline__ void add_diff(float a, float b) {
    const float h = a - b, w = h - a, z = (a - (h - w)) - (b + w);
    const float q = mul_rn(2.f * h, z), qe = fmaf(2.f * h, z, -q);
    add(h);
    term(q);
    e += fmaf(z, z, qe);
  }
  __device__ __forceinline__ bool nonzero() const { return (any << 1) != 0; }
  __device__ __forceinline__ double total() const { return (double)s + (double)c + (double)e; }
};
// Whether the block has to sum again: total (valid in thread 0) of the threads' SqSum
// is outside the range in which they are exact, though some value is not 0.  A slab has
// at most 2^24 values, whose underflows (a few of 2^-149 each) come to 2^-123 at most,
// 2^-59 of the smallest sum that stands.
template <typename T>
__device__ __forceinline__ bool sq_again(double total, bool nonzero) {
  if (sizeof(T) == 8) return false;
  const bool any = __syncthreads_or(nonzero);
  return __syncthreads_or(any && threadIdx.x == 0 && !(total >= 0x1p-64 && total <= 1e300));
}
struct SqSum64 {
  double s = 0.0;
  template <typename T>
  __device__ __forceinline__ void add(T v) {
    s = fma((double)v, (double)v, s);
  }
  template <typename T>
  __device__ __forceinline__ void add_diff(T a, T b) {
    add((double)a - (double)b);
  }
};
// Sum of values and rounding errors in the working precision.
template <typename T>
struct SqPair {
  T s = T(0), c = T(0);
  __device__ __forceinline__ void add(T v) { dot2(s, c, v, v); }
  __device__ __forceinline__ bool nonzero() const { return false; }
  __device__ __forceinline__ double total() const { return (double)s + (double)c; }
};

// A truth value as a type, for generic lambdas.
template <bool B>
struct BoolC {
  static constexpr bool value = B;
};

constexpr int kMaxRank = 32;

// Asynchronous 4-, 8- or 16-byte global -> shared copy (cp.async, L1-allocating);
// both addresses aligned to the element size.
template <typename T>
__device__ __forceinline__ void cp_async_elem(T* smem_dst, const T* gsrc) {
  static_assert(sizeof(T) == 4 || sizeof(T) == 8 || sizeof(T) == 16, "cp.async element size");
  const unsigned dst = (unsigned)__cvta_generic_to_shared(smem_dst);
  if constexpr (sizeof(T) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(gsrc) : "memory");
  else if constexpr (sizeof(T) == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(gsrc) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(gsrc) : "memory");
}

// Wait for every cp.async of this thread (the block still needs a barrier).
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

}  // namespace tc
