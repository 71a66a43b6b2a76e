// FastVR's one-step restoration update (Eq. `eq:one_step`): after the DiT
// predicts the velocity v from the low-quality latent z_LQ at t = tau, the
// restored latent is z_hat = z_LQ - sigma_tau * v.  Elementwise and purely
// bandwidth-bound: 16-byte loads of z_LQ with the matching elements of v, one
// fp32 FMA per element, a single rounding to the output type.
#include <cuda_bf16.h>

#include "fastvr_internal.h"

namespace fastvr {
namespace {

// The elements of one thread's access: 16 bytes of z (8 bf16 or 4 fp32) and
// the matching bf16 of v, so that a warp's accesses to each of the three
// buffers are contiguous.  (8 fp32 in two 16-byte halves per thread, at a
// stride of 32 bytes, touched every sector twice and wrote it in halves: 200 M
// elements 324 us, now 299, 6.7 TB/s; 50 M 81.8 -> 75.6.)
template <typename T>
struct Vec;
template <>
struct Vec<__nv_bfloat16> {
  static constexpr int kN = 8;
  using V = uint4;
  uint4 u;
  __device__ float get(int i) const {
    const __nv_bfloat16* e = reinterpret_cast<const __nv_bfloat16*>(&u);
    return __bfloat162float(e[i]);
  }
  __device__ void set(int i, float x) {
    reinterpret_cast<__nv_bfloat16*>(&u)[i] = __float2bfloat16_rn(x);
  }
};
template <>
struct Vec<float> {
  static constexpr int kN = 4;
  using V = uint2;
  float4 a;
  __device__ float get(int i) const { return (&a.x)[i]; }
  __device__ void set(int i, float x) { (&a.x)[i] = x; }
};
template <typename V>
__device__ __forceinline__ float bf16_at(const V& v, int i) {
  return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(&v)[i]);
}

__device__ __forceinline__ float to_f(float x) { return x; }
__device__ __forceinline__ float to_f(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ void from_f(float& d, float x) { d = x; }
__device__ __forceinline__ void from_f(__nv_bfloat16& d, float x) {
  d = __float2bfloat16_rn(x);
}

// z and out may be the same buffer (in-place update): every element is read
// and then written by the same thread.  Each thread keeps a few groups of loads
// in flight before it computes and stores, so that a few CTAs per SM cover the
// HBM latency: four groups at bf16 (128 bytes), eight at fp32 (192 bytes), then,
// since an fp32 latent of a few million elements gives a thread only two or
// three groups, two at a time.
template <typename T>
__device__ __forceinline__ void update(const Vec<T>& zv,
                                       const typename Vec<T>::V& vv,
                                       float neg_sigma, Vec<T>* dst) {
  Vec<T> o;
#pragma unroll
  for (int e = 0; e < Vec<T>::kN; ++e)
    o.set(e, fmaf(neg_sigma, bf16_at(vv, e), zv.get(e)));
  *dst = o;
}

// kU groups at a time, as long as that many are left; i moves on.
template <int kU, typename T>
__device__ __forceinline__ void run_groups(const Vec<T>* zg,
                                           const typename Vec<T>::V* vg,
                                           Vec<T>* og, int64_t& i,
                                           int64_t groups, int64_t stride,
                                           float neg_sigma) {
  for (; i + (kU - 1) * stride < groups; i += kU * stride) {
    Vec<T> zv[kU];
    typename Vec<T>::V vv[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      zv[u] = zg[i + u * stride];
      vv[u] = __ldcs(vg + i + u * stride);
    }
#pragma unroll
    for (int u = 0; u < kU; ++u)
      update(zv[u], vv[u], neg_sigma, og + i + u * stride);
  }
}

template <typename T>
__global__ void __launch_bounds__(256)
one_step_kernel(const T* z, const __nv_bfloat16* __restrict__ v, T* out,
                int64_t n, float neg_sigma) {
  constexpr int kN = Vec<T>::kN;
  pdl_trigger();
  pdl_wait();  // z and v may come from the previous kernel on the stream
  const int64_t groups = n / kN;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const Vec<T>* zg = reinterpret_cast<const Vec<T>*>(z);
  const typename Vec<T>::V* vg = reinterpret_cast<const typename Vec<T>::V*>(v);
  Vec<T>* og = reinterpret_cast<Vec<T>*>(out);
  int64_t i = tid;
  run_groups<32 / kN>(zg, vg, og, i, groups, stride, neg_sigma);
  if (kN == 4) run_groups<2>(zg, vg, og, i, groups, stride, neg_sigma);
  run_groups<1>(zg, vg, og, i, groups, stride, neg_sigma);
  for (int64_t i = groups * kN + tid; i < n; i += stride)  // fewer than kN left
    from_f(out[i], fmaf(neg_sigma, __bfloat162float(v[i]), to_f(z[i])));
}

}  // namespace

cudaError_t launch_one_step(const void* z, const void* v, void* out, int64_t n,
                            float sigma, int dtype, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms <= 0) sms = 152;
  int64_t blocks = (int64_t)sms * 8;
  const int64_t need = (n / (dtype == 0 ? 8 : 4) + 255) / 256 + 1;
  if (blocks > need) blocks = need;
  const float neg_sigma = -sigma;
  if (dtype == 0)
    return launch_pdl(one_step_kernel<__nv_bfloat16>, dim3((unsigned)blocks),
                      dim3(256), 0, stream,
                      static_cast<const __nv_bfloat16*>(z),
                      static_cast<const __nv_bfloat16*>(v),
                      static_cast<__nv_bfloat16*>(out), n, neg_sigma);
  return launch_pdl(one_step_kernel<float>, dim3((unsigned)blocks), dim3(256),
                    0, stream, static_cast<const float*>(z),
                    static_cast<const __nv_bfloat16*>(v),
                    static_cast<float*>(out), n, neg_sigma);
}

}  // namespace fastvr
