// device_functions.cu -- single device functions and kernels of the library on given operands, for
// test_gpu_device_functions.py (compiled there against csrc/).
#include "msp_fft.cuh"
#include "msp_loss.cuh"

using namespace msp;

extern "C" int run_loss(const float* pre, const float* target, int L, size_t P, float inv_sd, void* g, double* part, int blocks) {
  learn::loss_kernel<<<blocks, 256>>>(pre, target, L, P, inv_sd, (__nv_bfloat16*)g, part);
  return (int)cudaDeviceSynchronize();
}

// out[2 i], out[2 i + 1]: the factor and the loss term of operands i, through the choice that the kernels make (general 0)
// or the general form (1)
__global__ void residual_of(const float* a2, const float* I, float zthr2, int n, int general, float* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float l = 0.f, f;
  if (general || !residual_in_range(a2[i], I[i])) f = residual_exact(a2[i], I[i], zthr2, l);
  else f = residual_fast(a2[i], I[i], zthr2, l);
  out[2 * i] = f;
  out[2 * i + 1] = l;
}
extern "C" int run_residual(const float* a2, const float* I, float zthr2, int n, int general, float* out) {
  residual_of<<<(n + 255) / 256, 256>>>(a2, I, zthr2, n, general, out);
  return (int)cudaDeviceSynchronize();
}
