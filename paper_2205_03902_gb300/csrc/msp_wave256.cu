// msp_wave256.cu -- the fused per-position kernel of W = 256.
#include "msp_wave.cuh"

namespace msp {

template cudaError_t launch_wave<256>(int mode, const PosParams& p, int grid, cudaStream_t st);
template cudaError_t launch_again<256>(int mode, const PosParams& p, int grid, cudaStream_t st);
template int wave_slots<256>(int sms);

}  // namespace msp
