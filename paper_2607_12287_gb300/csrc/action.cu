// The 2-step action combine of Sec. III-C (Eq. 9): the final action state from the two
// anchor velocities of the flow-matching solver,
//   x_T[s][i] = x_0[s][i] + alpha[s] v_0[s][i] + beta[s] v_7[s][i] + b[s][i].
// The velocity network and the adaptor that predicts (alpha, beta, b) are not part of
// this library; the caller passes their outputs.  Elementwise; bound by the launch up to a few
// thousand samples, then by HBM.  The arrays are contiguous, so 128-bit loads and stores need
// only aligned arrays, not rows of a multiple of four values: a vector that crosses into the
// next sample takes its coefficients value by value.  4096 samples of 350 values (in L2) took 6.5 us
// with one value per thread and a 64-bit division each, and take 3.6; 65536 took 120 and take 66.
#include "internal.h"
#include "ptx.cuh"
#include "ivit.h"

namespace ivit {
namespace {

// Index: 32-bit unsigned while the values number less than 2^31 (a 64-bit division is a
// subroutine), else 64-bit.
template <typename Index>
__global__ void action_combine_kernel(const float* __restrict__ x0, const float* __restrict__ v0,
                                      const float* __restrict__ v7, const float* __restrict__ alpha,
                                      const float* __restrict__ beta, const float* __restrict__ b,
                                      Index dim, Index n, int vec4, float* __restrict__ xT) {
  pdl_wait();
  pdl_launch_dependents();
  const Index stride = static_cast<Index>(gridDim.x) * blockDim.x;
  const Index first = blockIdx.x * static_cast<Index>(blockDim.x) + threadIdx.x;
  const Index n4 = vec4 ? n / 4 : 0;
  const float4* x4 = reinterpret_cast<const float4*>(x0);
  const float4* a4 = reinterpret_cast<const float4*>(v0);
  const float4* c4 = reinterpret_cast<const float4*>(v7);
  const float4* b4 = reinterpret_cast<const float4*>(b);
  float4* y4 = reinterpret_cast<float4*>(xT);
  for (Index k = first; k < n4; k += stride) {
    const float4 x = x4[k], p = a4[k], q = c4[k];
    const float4 o = b ? b4[k] : make_float4(0.f, 0.f, 0.f, 0.f);
    const Index s = 4 * k / dim;
    float al[4], be[4];
    al[0] = alpha[s];
    be[0] = beta[s];
    if (4 * k + 3 < (s + 1) * dim) {
#pragma unroll
      for (int j = 1; j < 4; ++j) {
        al[j] = al[0];
        be[j] = be[0];
      }
    } else {
#pragma unroll
      for (int j = 1; j < 4; ++j) {
        const Index sj = (4 * k + j) / dim;
        al[j] = alpha[sj];
        be[j] = beta[sj];
      }
    }
    y4[k] = make_float4(fmaf(be[0], q.x, fmaf(al[0], p.x, x.x)) + o.x, fmaf(be[1], q.y, fmaf(al[1], p.y, x.y)) + o.y,
                        fmaf(be[2], q.z, fmaf(al[2], p.z, x.z)) + o.z, fmaf(be[3], q.w, fmaf(al[3], p.w, x.w)) + o.w);
  }
  for (Index k = 4 * n4 + first; k < n; k += stride) {
    const Index s = k / dim;
    xT[k] = fmaf(beta[s], v7[k], fmaf(alpha[s], v0[k], x0[k])) + (b ? b[k] : 0.f);
  }
}

}  // namespace
}  // namespace ivit

extern "C" int ivit_action_combine(const float* x0_dev, const float* v0_dev, const float* v7_dev,
                                   const float* alpha_dev, const float* beta_dev, const float* b_dev,
                                   int32_t batch, int32_t dim, float* xT_dev, void* stream) {
  if (batch < 0 || dim < 0) return IVIT_ERR_ARG;
  const long long n = static_cast<long long>(batch) * dim;
  if (n == 0) return IVIT_OK;
  if (!x0_dev || !v0_dev || !v7_dev || !alpha_dev || !beta_dev || !xT_dev) return IVIT_ERR_ARG;
  // 128-bit accesses need 16-byte aligned arrays; others take the scalar loop (alignment 4
  // bytes, checked here).
  auto aligned = [](const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; };
  for (const void* p : {static_cast<const void*>(x0_dev), static_cast<const void*>(v0_dev),
                        static_cast<const void*>(v7_dev), static_cast<const void*>(alpha_dev),
                        static_cast<const void*>(beta_dev), static_cast<const void*>(b_dev),
                        static_cast<const void*>(xT_dev)})
    if (p && !aligned(p, 4)) return IVIT_ERR_ARG;
  const bool vec4 = n >= 4 && aligned(x0_dev, 16) && aligned(v0_dev, 16) && aligned(v7_dev, 16) &&
                    aligned(xT_dev, 16) && (!b_dev || aligned(b_dev, 16));
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))
    return IVIT_ERR_CUDA;
  const long long items = vec4 ? n / 4 : n;
  const long long blocks = (items + 255) / 256;
  const int grid = static_cast<int>(blocks < 4LL * sms ? blocks : 4LL * sms);
  auto launch = [&](auto kern, auto index) {
    using Index = decltype(index);
    return ivit::launch_ex(kern, dim3(grid), dim3(256), 0, static_cast<cudaStream_t>(stream), 1, x0_dev, v0_dev, v7_dev,
                           alpha_dev, beta_dev, b_dev, static_cast<Index>(dim), static_cast<Index>(n), vec4 ? 1 : 0,
                           xT_dev);
  };
  const cudaError_t e = n < (1LL << 31) ? launch(ivit::action_combine_kernel<uint32_t>, uint32_t{})
                                        : launch(ivit::action_combine_kernel<uint64_t>, uint64_t{});
  return e == cudaSuccess ? IVIT_OK : IVIT_ERR_CUDA;
}
