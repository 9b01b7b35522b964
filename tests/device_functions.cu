// device_functions.cu -- single device functions and kernels of the library on given operands, for
// test_gpu_device_functions.py (compiled there against csrc/).
#include "msp_fft.cuh"
#include "msp_loss.cuh"

using namespace msp;

extern "C" int run_loss(const float* pre, const float* target, int L, size_t P, float inv_sd, void* g, double* part, int blocks) {
  learn::loss_kernel<<<blocks, 256>>>(pre, target, L, P, inv_sd, (__nv_bfloat16*)g, part);
  return (int)cudaDeviceSynchronize();
}
