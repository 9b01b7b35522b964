// msp_loss.cuh -- the training loss of the proposal network (msp_learn.cu) and its gradient.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "msp_kernels.cuh"

namespace msp {
namespace learn {

// Mean squared error against target / s_D and its gradient with respect to the last layer's
// pre-activation (bf16 NHWC, padded channels 0); per-block loss partials (FP64).
// One thread per pixel: its 16 channels are four 16-byte loads and two 16-byte stores, the target's planes are read in
// rows.  A thread sums its squares in compensated FP32, rounding errors of the products included, and a pixel whose
// sum leaves the range where these are exact to FP64's rounding again in FP64: in FP64 alone, whose pipe takes about one
// conversion or addition per cycle and SM, the kernel took 19 us at 384 x 384 with either split; it takes 11.
__global__ void __launch_bounds__(256) loss_kernel(const float* __restrict__ pre, const float* __restrict__ target, int L,
                                                   size_t P, float inv_sd, __nv_bfloat16* __restrict__ g,
                                                   double* __restrict__ part) {
  __shared__ double red[8];
  const double inv_n = 1.0 / ((double)P * L);
  Compensated sum;
  double acc = 0.0;
  const float scale = (float)(2.0 * inv_n);
  for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < P; p += (size_t)gridDim.x * blockDim.x) {
    float x[16], y[16];
#pragma unroll
    for (int c = 0; c < 16; c += 4) {
      const float4 v = c < L ? reinterpret_cast<const float4*>(pre + p * 16)[c / 4] : make_float4(0.f, 0.f, 0.f, 0.f);
      x[c] = v.x; x[c + 1] = v.y; x[c + 2] = v.z; x[c + 3] = v.w;
    }
#pragma unroll
    for (int c = 0; c < 16; ++c) y[c] = c < L ? target[(size_t)c * P + p] : 0.f;
    alignas(16) __nv_bfloat16 o[16];
    Compensated pixel;
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const float d = c < L ? x[c] - inv_sd * y[c] : 0.f;
      const float d2 = __fmul_rn(d, d);   // rounded here: its error is added beside it
      pixel.add(d2);
      pixel.add_error(fmaf(d, d, -d2));
      x[c] = d;
      o[c] = __float2bfloat16_rn(c < L ? scale * d : 0.f);
    }
    if (pixel.s > 1e-25f && pixel.s < 1e36f) {
      sum.add(pixel);
      if (sum.s > 1e36f) {   // a thread takes up to 512 pixels: their sum stays in FP32's range too
        acc += sum.wide();
        sum = Compensated();
      }
    } else {
#pragma unroll
      for (int c = 0; c < 16; ++c) acc += (double)x[c] * x[c];
    }
    uint4* dst = reinterpret_cast<uint4*>(g + p * 16);
    dst[0] = reinterpret_cast<const uint4*>(o)[0];
    dst[1] = reinterpret_cast<const uint4*>(o)[1];
  }
  acc += sum.wide();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += red[w];
    part[blockIdx.x] = s * inv_n;
  }
}

}  // namespace learn
}  // namespace msp
