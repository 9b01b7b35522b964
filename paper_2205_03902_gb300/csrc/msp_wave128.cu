// msp_wave128.cu -- the fused per-position kernel of W = 128.
#include "msp_wave.cuh"

namespace msp {

template cudaError_t launch_wave<128>(int mode, const PosParams& p, int grid, cudaStream_t st);
template cudaError_t launch_again<128>(int mode, const PosParams& p, int grid, cudaStream_t st);
template int wave_slots<128>(int sms);

}  // namespace msp
