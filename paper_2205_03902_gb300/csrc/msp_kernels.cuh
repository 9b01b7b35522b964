// msp_kernels.cuh -- kernel parameter blocks and launch helpers shared by the
// translation units of libmsp.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace msp {

enum Mode { MODE_FORWARD = 0, MODE_LOSS_GRAD = 1, MODE_LAYER = 2, MODE_PROBE = 3 };

// Everything the fused per-position kernel reads or writes.
struct PosParams {
  const float2* probe;     // [W][W]
  const float2* T;         // [L][Ny][Nx] slice transmissions exp(i sigma V)
  const float2* h1;        // [W] separable propagator factor exp(-i pi dz lambda q_k^2) / W
  const int2* pos;         // [S] window top-left (y, x)
  const float* I_meas;     // [S][W][W]
  float* I_out;            // [S][W][W]                (forward)
  float2* stash;           // [G][Ls][W][W] exit waves kept for the adjoint
  float* wgrad;            // [S][Lg][W][W] per-position window gradients (float2 in transmission mode)
  float* willum;           // [S][W][W] per-position |psi_in,l|^2 (layer step)
  float* dVred;            // [L][Ny][Nx] (loss and gradients) or [Ny][Nx] (layer step), float2 in
                           // transmission mode, zeroed: when set, the kernel adds every window
                           // gradient into it with reductions in L2 instead of writing wgrad (the
                           // order of the additions is not fixed)
  float* illumred;         // [Ny][Nx], zeroed: the layer step's |psi_in,l|^2 likewise, instead of willum
  float2* dprobe_part;     // [G][W][W] per-CTA probe-gradient partial sums
  double* loss_part;       // [S] per-position loss ([S][4], one per CTA, for W = 256)
  uint8_t* again;          // [S] 1: the position is left to the second launch (W = 128, 256; not forward)
  int* again_any;          // whether there is such a position
  const double* zthr2;     // [1] squared far-field amplitude that counts as zero
  int* err;                // error flags
  int L, Ny, Nx, S;
  int layer;               // slice of a layer step
  int want_dprobe;
  int loss_only;           // loss-and-gradient pass with neither gradient wanted: forward and loss only
  int cplx;                // transmission mode: T is the caller's complex slices, gradients complex
  float two_sigma;
};

// Programmatic dependent launch: a kernel of a pass is set up and its prologue runs while its predecessor in
// the stream drains; it reads and writes nothing of the pass before wait_for_predecessor(), which returns once
// the predecessor has completed (and so, each kernel waiting in turn, everything before it).  Without the
// launch attribute the wait does nothing.  The predecessor gives no earlier signal: with one
// (griddepcontrol.launch_dependents at its start) the next kernel's CTAs were placed around those still running and
// shared SMs that a later placement leaves to one each (the plain method at W = 64, 64 positions, ten passes: 311 us with it,
// 235 us without, 314 us with ordinary launches).
__device__ __forceinline__ void wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename... P, typename... A>
inline cudaError_t launch_following(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cluster,
                                    A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Launches a fused per-position kernel K on `grid` position slots.
template <typename K>
cudaError_t launch_position_as(const PosParams& p, int grid, cudaStream_t st) {
  static bool attr_done[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 64 && !attr_done[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(K::fn(), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)K::SMEM);
    if (e != cudaSuccess) return e;
    attr_done[dev] = true;
  }
  return launch_following(K::fn(), dim3(grid * K::CLUSTER), dim3(K::NT), K::SMEM, st, K::CLUSTER, p);
}

// An FP64 sum of FP32 values without the FP64 pipe, which converts and adds about one value per cycle and SM: three
// FP32 terms, the sum, its rounding errors (Knuth's two-sum) and theirs (cascaded, Klein 2006), about 72 bits before the one
// rounding to FP64. A sum that leaves FP32's range is not finite, and the caller takes it again in FP64.
struct Compensated {
  float s = 0.f, e = 0.f, ee = 0.f;
  // x + v in x, returns the rounding error; the intrinsics are never fused with the product that v may be
  static __device__ __forceinline__ float two_sum(float& x, float v) {
    const float t = __fadd_rn(x, v), b = __fsub_rn(t, x);
    const float r = __fadd_rn(__fsub_rn(x, __fsub_rn(t, b)), __fsub_rn(v, b));
    x = t;
    return r;
  }
  __device__ __forceinline__ void add_error(float v) { ee += two_sum(e, v); }
  __device__ __forceinline__ void add(float v) { add_error(two_sum(s, v)); }
  __device__ __forceinline__ void add(const Compensated& c) {
    add(c.s);
    add_error(c.e);
    ee += c.ee;
  }
  // where s is not finite, its errors are NaN
  __device__ __forceinline__ double wide() const { return ee == ee ? (double)s + ((double)e + (double)ee) : (double)s; }
};

// Workspace carve-up (all offsets 256-byte aligned).
struct Workspace {
  int* err;                // [2] window error; whether any `again` is set
  double* scal;            // [16] scalars: 0 loss, 1 mu, 2 max illum, 3 sum I, 5 zero-rule threshold^2
  double* red;             // [kRedSlots] block partials of FP64 reductions, or (as floats) per-tile maxima
  float2* h1;              // [W]
  float2* T;
  float2* stash;
  float* wgrad;
  float* willum;
  float2* dprobe_part;
  float2* dprobe_sum;      // [W][W]
  double* loss_part;       // [S], or [S][4]
  uint8_t* again;          // [S] positions left to the second launch of a pass
  float* map0;             // [Ny][Nx] layer gradient map
  float* map1;             // [Ny][Nx] illumination map
  char* precise;           // the precise-forward mode's buffers (NULL in the FP32 mode)
  size_t bytes;
};

// Inputs of the batched modes (FP64 forward, split-BF16 DFT) beyond the fused kernel's parameters.
struct PreciseIn {
  const float* V;        // FP32 potentials (potential mode) or NULL
  const float2* X;       // the caller's complex slices (transmission mode) or NULL
  double sigma;          // interaction constant
  double dzlam, dq;      // dz lambda and the reciprocal pixel 1 / (W pixel) of the propagator
  char* extra;           // the batched modes' workspace segment
  int sms;               // SMs of the device (grid sizes of the element-wise kernels)
  int precision;         // MSP_PRECISION_FP64_FORWARD or MSP_PRECISION_BF16X3_DFT
  int wait_limit;        // poll bound of the tensor-core waits
};

constexpr int kRedSlots = 8192;

// Zero rule of the amplitude-flow gradient (Sec. 3.2: Qz/|Qz| := 0 where Qz = 0),
// resolved at the arithmetic's resolution: a far-field value counts as zero when
// |Psi_k| <= kZeroRuleTau * ||p||_2, the probe norm being the RMS far-field amplitude
// of every pattern of pure-phase slices (Parseval).
constexpr double kZeroRuleTau = 1e-5;

}  // namespace msp
