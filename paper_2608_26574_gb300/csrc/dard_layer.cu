// dard_layer.cu - the elementwise work between a layer's projections: residual add with
// RMSNorm, and the gate of a SwiGLU MLP.
//
// As separate tensor operations a norm is seven launches and a gate two, each a pass over the
// activations: a forward pass of small layers spent its time launching them (two layers of
// d_model 1024 over 2688 rows: about 70 launches, 1246 us). Here a row's residual sum, its mean
// square and the normalised row are one launch, and so is the gate (759 us for the whole
// pass). Arithmetic in fp32; the residual sum is rounded to the storage type before it is
// squared, as the stored sum is what later layers see. Bound: memory (each operand once; the
// activations of such layers stay in L2).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "dard_internal.h"

namespace dard {
namespace {

constexpr int kNormThreads = 256;  // at most, one row per CTA
constexpr int kHold = 4;           // vectors of its row a thread keeps in registers
constexpr int kGateThreads = 256;

__device__ __forceinline__ float to_f(float x) { return x; }
__device__ __forceinline__ float to_f(__nv_bfloat16 x) { return __bfloat162float(x); }
template <class T>
__device__ __forceinline__ T from_f(float x) {
  if constexpr (sizeof(T) == 2) return __float2bfloat16_rn(x);
  else return x;
}

// W elements of T: 16 bytes, or one element where rows or pointers are not 16-byte aligned.
template <class T, int W>
struct __align__(W == 1 ? sizeof(T) : 16) Vec {
  T e[W];
};

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// One row per CTA: s = x + add (or x), stored to `sum` if given; out = s / rms(s). A thread
// reads back only what it wrote or read itself, so that sum may be x or add, and out any of
// them.
template <class T, int W>
__global__ void __launch_bounds__(kNormThreads)
    add_rmsnorm(const T* x, const T* add, T* sum, T* out, int width, float eps) {
  using V = Vec<T, W>;
  __shared__ float s_part[kNormThreads / 32];
  const size_t base = static_cast<size_t>(blockIdx.x) * width;
  const V* xv = reinterpret_cast<const V*>(x + base);
  const V* av = reinterpret_cast<const V*>(add + base);
  V* sv = reinterpret_cast<V*>(sum + base);
  V* ov = reinterpret_cast<V*>(out + base);
  const int n = width / W, nt = blockDim.x;
  auto row_sum = [&](int i) {
    V v = xv[i];
    if (add != nullptr) {
      const V a = av[i];
#pragma unroll
      for (int e = 0; e < W; ++e) v.e[e] = from_f<T>(to_f(v.e[e]) + to_f(a.e[e]));
    }
    return v;
  };
  V keep[kHold];
  float sq = 0.f;
#pragma unroll
  for (int k = 0; k < kHold; ++k) {
    const int i = threadIdx.x + k * nt;
    if (i < n) keep[k] = row_sum(i);
  }
#pragma unroll
  for (int k = 0; k < kHold; ++k) {
    const int i = threadIdx.x + k * nt;
    if (i >= n) continue;
    if (sum != nullptr) sv[i] = keep[k];
#pragma unroll
    for (int e = 0; e < W; ++e) sq = fmaf(to_f(keep[k].e[e]), to_f(keep[k].e[e]), sq);
  }
  for (int i = threadIdx.x + kHold * nt; i < n; i += nt) {
    const V v = row_sum(i);
    if (sum != nullptr) sv[i] = v;
#pragma unroll
    for (int e = 0; e < W; ++e) sq = fmaf(to_f(v.e[e]), to_f(v.e[e]), sq);
  }
  sq = warp_sum(sq);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = sq;
  __syncthreads();
  float total = 0.f;
  for (int w = 0; w < nt / 32; ++w) total += s_part[w];
  const float r = rsqrtf(total / width + eps);
  auto put = [&](int i, V v) {
#pragma unroll
    for (int e = 0; e < W; ++e) v.e[e] = from_f<T>(to_f(v.e[e]) * r);
    ov[i] = v;
  };
#pragma unroll
  for (int k = 0; k < kHold; ++k) {
    const int i = threadIdx.x + k * nt;
    if (i < n) put(i, keep[k]);
  }
  for (int i = threadIdx.x + kHold * nt; i < n; i += nt) put(i, sum != nullptr ? sv[i] : row_sum(i));
}

// out = silu(a) * b, rounded once.
template <class T, int W>
__global__ void __launch_bounds__(kGateThreads) swiglu(const T* a, const T* b, T* out, long long n) {
  using V = Vec<T, W>;
  const long long i = static_cast<long long>(blockIdx.x) * kGateThreads + threadIdx.x;
  if (i >= n) return;
  V u = reinterpret_cast<const V*>(a)[i];
  const V v = reinterpret_cast<const V*>(b)[i];
#pragma unroll
  for (int e = 0; e < W; ++e) {
    const float g = to_f(u.e[e]);
    u.e[e] = from_f<T>(g / (1.f + expf(-g)) * to_f(v.e[e]));
  }
  reinterpret_cast<V*>(out)[i] = u;
}

bool aligned(const void* p, size_t to) { return reinterpret_cast<uintptr_t>(p) % to == 0; }

template <class T, int W>
cudaError_t launch_norm(const void* x, const void* add, void* sum, void* out, int rows, int width,
                        float eps, cudaStream_t stream) {
  const int threads = std::min(kNormThreads, (width / W + 31) / 32 * 32);
  add_rmsnorm<T, W><<<rows, threads, 0, stream>>>(
      static_cast<const T*>(x), static_cast<const T*>(add), static_cast<T*>(sum),
      static_cast<T*>(out), width, eps);
  return cudaGetLastError();
}

template <class T>
dard_status norm(const void* x, const void* add, void* sum, void* out, int rows, int width,
                 float eps, cudaStream_t stream) {
  for (const void* p : {x, add, static_cast<const void*>(sum), static_cast<const void*>(out)})
    if (!aligned(p, sizeof(T))) return report(DARD_ERR_ALIGN, "a pointer is not aligned to its elements");
  if (rows == 0) return DARD_OK;
  constexpr int W = 16 / sizeof(T);
  const bool wide = width % W == 0 && aligned(x, 16) && aligned(add, 16) && aligned(sum, 16) &&
                    aligned(out, 16);
  const cudaError_t e = wide ? launch_norm<T, W>(x, add, sum, out, rows, width, eps, stream)
                             : launch_norm<T, 1>(x, add, sum, out, rows, width, eps, stream);
  return e == cudaSuccess ? DARD_OK
                          : report(DARD_ERR_CUDA, "add_rmsnorm launch failed: %s", cudaGetErrorString(e));
}

template <class T, int W>
cudaError_t launch_gate(const void* a, const void* b, void* out, long long n, cudaStream_t stream) {
  const long long blocks = (n / W + kGateThreads - 1) / kGateThreads;
  if (blocks > 0x7fffffffll) return cudaErrorInvalidValue;
  swiglu<T, W><<<static_cast<unsigned>(blocks), kGateThreads, 0, stream>>>(
      static_cast<const T*>(a), static_cast<const T*>(b), static_cast<T*>(out), n / W);
  return cudaGetLastError();
}

template <class T>
dard_status gate(const void* a, const void* b, void* out, long long n, cudaStream_t stream) {
  for (const void* p : {a, b, static_cast<const void*>(out)})
    if (!aligned(p, sizeof(T))) return report(DARD_ERR_ALIGN, "a pointer is not aligned to its elements");
  if (n == 0) return DARD_OK;
  constexpr int W = 16 / sizeof(T);
  const bool wide = n % W == 0 && aligned(a, 16) && aligned(b, 16) && aligned(out, 16);
  const cudaError_t e = wide ? launch_gate<T, W>(a, b, out, n, stream)
                             : launch_gate<T, 1>(a, b, out, n, stream);
  return e == cudaSuccess ? DARD_OK
                          : report(DARD_ERR_CUDA, "swiglu launch failed: %s", cudaGetErrorString(e));
}

}  // namespace
}  // namespace dard

extern "C" {

dard_status dard_add_rmsnorm(const void* x, const void* add, void* sum, void* out, int32_t rows,
                             int32_t width, int32_t dtype, float eps, void* stream) {
  using namespace dard;
  if (rows < 0 || width < 1) return report(DARD_ERR_SHAPE, "rows %d, width %d", rows, width);
  if (rows > 0 && (!x || !out)) return report(DARD_ERR_NULL, "x or out is NULL");
  if (dtype != DARD_BF16 && dtype != DARD_F32)
    return report(DARD_ERR_VALUE, "dtype %d is neither DARD_F32 nor DARD_BF16", dtype);
  if (!(eps >= 0.f) || !std::isfinite(eps)) return report(DARD_ERR_VALUE, "eps must be finite and >= 0");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return dtype == DARD_BF16 ? norm<__nv_bfloat16>(x, add, sum, out, rows, width, eps, s)
                            : norm<float>(x, add, sum, out, rows, width, eps, s);
}

dard_status dard_swiglu(const void* a, const void* b, void* out, int64_t n, int32_t dtype,
                        void* stream) {
  using namespace dard;
  if (n < 0) return report(DARD_ERR_SHAPE, "n is negative");
  if (n > 0 && (!a || !b || !out)) return report(DARD_ERR_NULL, "a, b or out is NULL");
  if (dtype != DARD_BF16 && dtype != DARD_F32)
    return report(DARD_ERR_VALUE, "dtype %d is neither DARD_F32 nor DARD_BF16", dtype);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return dtype == DARD_BF16 ? gate<__nv_bfloat16>(a, b, out, n, s) : gate<float>(a, b, out, n, s);
}

}  // extern "C"
