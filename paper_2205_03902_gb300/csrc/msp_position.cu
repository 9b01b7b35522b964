// msp_position.cu -- the fused per-position multislice forward / adjoint kernels: W = 64 here, W = 128 and 256 in
// msp_wave.cuh.
//
// One CTA (W = 256: a cluster of four) owns one scan position at a time (persistent grid, slot g takes the
// positions g, g + slots, ...) and runs the whole of it: every slice's
// transmit (Sec. 2.1, E_m = V_z(E_{m-1}) o X_m), Fresnel propagation F^-1(H o F .), the
// far-field transform F(E_M), the amplitude-flow residual (Sec. 3.2) and the adjoint
// recursion chi_{m-1} = G^H (conj(X_m) o chi_m) (Sec. 3.3, the prefix / suffix products R_l
// and S_l applied matrix-free).
//
// The propagator is separable, h(ky, kx) = h1(ky) h1(kx) with
// h1(k) = exp(-i pi dz lambda q_k^2) / W (the 1/W^2 of F^-1 folded in), so it is
// a W-entry shared table.
//
// The only per-slice global traffic is the transmission window (read), the exit
// wave of each slice (written to this CTA's stash slot on the way forward, read
// back on the way down; the slots are reused position after position so they
// stay L2-resident) and the per-position window gradient.  The data each position
// touches once (window gradients, illumination) is stored with the evict-first
// (streaming) cache hint, so that it does not push the stash slots out of L2.
#include "msp_fft.cuh"
#include "msp_kernels.cuh"

namespace msp {

// ----------------------------------------------------------------------------
// W = 64: the wave in shared memory, line transforms by groups of eight threads
// ----------------------------------------------------------------------------
// A propagation is  rows F -> [columns F, x H, columns F^-1] -> rows F^-1: the column transforms and
// the propagator run back to back in registers, and the inverse row transform of one slice, the
// transmit of the next slice and its forward row transform also run back to back in registers.
// Each phase is one read and one write of the wave in shared memory plus the in-line exchange, which
// goes through a small padded buffer that each line group owns next to the wave.
template <int W>
struct Geo {
  static constexpr int NT = 4 * W;        // threads per CTA
  static constexpr int N1 = W / 8;        // values per thread per line
  static constexpr int GROUPS = NT / 8;   // eight-thread line groups
  static constexpr int LPG = W / GROUPS;  // lines per group per pass
};

// Shared-memory offset of element j + 8m of wave row r: (j + 8m) ^ swz(r) flips bits 0-2
// by swz(r) & 7 and bit 3 by swz(r) & 8, i.e. adds +-8 for even / odd m.
template <int W>
struct RowIdx {
  int be, bo;
  __device__ __forceinline__ RowIdx(int r, int j) {
    const int sw = swz(r);
    const int base = r * W + (j ^ (sw & 7));
    be = base + (sw & 8);
    bo = base - (sw & 8);
  }
  __device__ __forceinline__ int operator()(int m) const { return ((m & 1) ? bo : be) + 8 * m; }
};
// Element j + 8m of wave column c: swz depends on the row's low three bits only (= j).
template <int W>
struct ColIdx {
  int b;
  __device__ __forceinline__ ColIdx(int c, int j) : b(j * W + (c ^ swz(j))) {}
  __device__ __forceinline__ int operator()(int m) const { return b + 8 * m * W; }
};

// Dynamic shared memory: the wave, then one exchange buffer per eight-thread line group.
template <int W>
__host__ __device__ constexpr int exchange_floats2() {
  return kXGroup(W / 8);
}
template <int W>
constexpr size_t position_smem_bytes() {
  return ((size_t)W * W + (size_t)(W / 2) * exchange_floats2<W>()) * sizeof(float2);
}

// CPLX: transmission mode (the paper's complex slices o_l).  The stash then holds the wave
// incident on each slice and the window gradient is dL/dconj(o_l) = conj(psi_in,l) o chi_l;
// in potential mode it holds the exit wave and the gradient is 2 sigma Im(conj(E_l) chi_l).
template <int W, int MODE, bool CPLX = false>
__global__ void __launch_bounds__(4 * W, 1) position_kernel(const PosParams p) {
  using G = Geo<W>;
  constexpr int N1 = G::N1;
  extern __shared__ float2 sm[];
  __shared__ float2 s_tw[N1 * 8];   // w_W^(j k1) at [k1 * 8 + j]
  __shared__ float2 s_h1[W];        // h1(k) = exp(-i pi dz lambda q_k^2) / W
  __shared__ float red[G::NT / 32];

  const int tid = threadIdx.x;
  const int j = tid & 7;
  const int grp = tid >> 3;
  const size_t WW = (size_t)W * W;
  const size_t plane = (size_t)p.Ny * p.Nx;
  float2* xb = sm + W * W + grp * exchange_floats2<W>();   // this group's exchange buffer

  if (tid < N1 * 8) {
    const int k1 = tid >> 3, jj = tid & 7;
    s_tw[tid] = twiddle<W>((jj * k1) % W);
  }
  wait_for_predecessor();
  if (tid < W) s_h1[tid] = p.h1[tid];
  __syncthreads();
  const RegisterTwiddles<W, 8> tw(s_tw, j);

  const int L = p.L;
  const float zthr2 = (MODE == MODE_FORWARD) ? 0.f : (float)p.zthr2[0];
  const bool need_stash = (MODE == MODE_LOSS_GRAD && !p.loss_only) || (MODE == MODE_LAYER);
  const int lowest = (MODE == MODE_LAYER) ? p.layer : 0;
  bool first_dprobe = true;
  for (int s = blockIdx.x; s < p.S; s += gridDim.x) {
    const int2 ps = p.pos[s];
    const int y0 = ps.x, x0 = ps.y;
    const bool ok = (y0 >= 0) && (x0 >= 0) && (y0 <= p.Ny - W) && (x0 <= p.Nx - W);
    if (!ok) {
      if (tid == 0) atomicMax(p.err, 1);
      // outputs of a skipped position are zero
      if (MODE == MODE_FORWARD) {
        for (size_t i = tid; i < WW; i += G::NT) p.I_out[s * WW + i] = 0.f;
      } else {
        if (tid == 0) p.loss_part[s] = 0.0;
        constexpr int CW = CPLX ? 2 : 1;
        if (MODE == MODE_LOSS_GRAD && !p.dVred)
          for (size_t i = tid; i < CW * WW * L; i += G::NT) p.wgrad[CW * s * WW * L + i] = 0.f;
        if (MODE == MODE_LAYER && !p.dVred) {
          for (size_t i = tid; i < CW * WW; i += G::NT) p.wgrad[CW * s * WW + i] = 0.f;
          for (size_t i = tid; i < WW; i += G::NT) p.willum[s * WW + i] = 0.f;
        }
      }
      continue;  // uniform across the CTA
    }
    const size_t win0 = (size_t)y0 * p.Nx + x0;
    float2* stash = p.stash + (size_t)blockIdx.x * (MODE == MODE_LOSS_GRAD ? L : 1) * WW;

    // ---------------- forward: slice 0, rows ----------------
#pragma unroll 1
    for (int it = 0; it < G::LPG; ++it) {
      const int r = grp + G::GROUPS * it;
      float2 v[N1];
      const float2* T0 = p.T + win0 + (size_t)r * p.Nx;
#pragma unroll
      for (int m = 0; m < N1; ++m) v[m] = p.probe[r * W + j + 8 * m];
      const bool keep0 = need_stash && (MODE == MODE_LOSS_GRAD || p.layer == 0);
      if (CPLX && keep0) {
#pragma unroll
        for (int m = 0; m < N1; ++m) stash[r * W + j + 8 * m] = v[m];   // incident wave
      }
#pragma unroll
      for (int m = 0; m < N1; ++m) v[m] = cmul(v[m], T0[j + 8 * m]);
      if (!CPLX && keep0) {
#pragma unroll
        for (int m = 0; m < N1; ++m) stash[r * W + j + 8 * m] = v[m];   // exit wave
      }
      line_fft_t<W, false>(v, tw, xb, j);
#pragma unroll
      for (int m = 0; m < N1; ++m) sm[RowIdx<W>(r, j)(m)] = v[m];
    }
    __syncthreads();

    float lsum = 0.f;
#pragma unroll 1
    for (int l = 0; l < L; ++l) {
      if (l < L - 1) {
        // columns: F, x H / W^2, F^-1 (unnormalised)
#pragma unroll 1
        for (int it = 0; it < G::LPG; ++it) {
          const int c = grp + G::GROUPS * it;
          const ColIdx<W> ca(c, j);
          float2 v[N1];
#pragma unroll
          for (int m = 0; m < N1; ++m) v[m] = sm[ca(m)];
          line_fft_t<W, false>(v, tw, xb, j);
          const float2 hx = s_h1[c];
#pragma unroll
          for (int m = 0; m < N1; ++m) v[m] = cmul(v[m], cmul(s_h1[j + 8 * m], hx));
          line_fft_t<W, true>(v, tw, xb, j);
#pragma unroll
          for (int m = 0; m < N1; ++m) sm[ca(m)] = v[m];
        }
        __syncthreads();
        // rows: F^-1, transmit slice l+1, keep the exit wave, F
        const float2* Tl = p.T + (size_t)(l + 1) * plane + win0;
        const bool keep = need_stash && (MODE == MODE_LOSS_GRAD || p.layer == l + 1);
        float2* st = stash + (MODE == MODE_LOSS_GRAD ? (size_t)(l + 1) * WW : 0);
#pragma unroll 1
        for (int it = 0; it < G::LPG; ++it) {
          const int r = grp + G::GROUPS * it;
          const RowIdx<W> ra(r, j);
          float2 t[N1], v[N1];
          const float2* Tr = Tl + (size_t)r * p.Nx;
#pragma unroll
          for (int m = 0; m < N1; ++m) t[m] = Tr[j + 8 * m];     // in flight during the transform
#pragma unroll
          for (int m = 0; m < N1; ++m) v[m] = sm[ra(m)];
          line_fft_t<W, true>(v, tw, xb, j);
          if (CPLX && keep) {
#pragma unroll
            for (int m = 0; m < N1; ++m) st[r * W + j + 8 * m] = v[m];   // incident wave
          }
#pragma unroll
          for (int m = 0; m < N1; ++m) v[m] = cmul(v[m], t[m]);
          if (!CPLX && keep) {
#pragma unroll
            for (int m = 0; m < N1; ++m) st[r * W + j + 8 * m] = v[m];   // exit wave
          }
          line_fft_t<W, false>(v, tw, xb, j);
#pragma unroll
          for (int m = 0; m < N1; ++m) sm[ra(m)] = v[m];
        }
        __syncthreads();
      } else {
        // far field Psi = F(E_L): finish with the column transforms
#pragma unroll 1
        for (int it = 0; it < G::LPG; ++it) {
          const int c = grp + G::GROUPS * it;
          const ColIdx<W> ca(c, j);
          float2 v[N1];
          float im[N1];
          if (MODE != MODE_FORWARD) {
            const float* ip = p.I_meas + s * WW + c;
#pragma unroll
            for (int m = 0; m < N1; ++m) im[m] = __ldcs(ip + (j + 8 * m) * W);   // read once: evict first; in flight during the transform
          }
#pragma unroll
          for (int m = 0; m < N1; ++m) v[m] = sm[ca(m)];
          line_fft_t<W, false>(v, tw, xb, j);
          if (MODE == MODE_FORWARD) {
            float* out = p.I_out + s * WW + c;
#pragma unroll
            for (int m = 0; m < N1; ++m) out[(j + 8 * m) * W] = fmaf(v[m].x, v[m].x, v[m].y * v[m].y);
          } else {
            // amplitude-flow residual R = Psi - sqrt(I) Psi / |Psi| (fraction 0 where Psi counts as 0)
            residual(v, im, zthr2, lsum);
            // chi = F^H R: inverse column transforms now, rows below
            if (!p.loss_only) {
              line_fft_t<W, true>(v, tw, xb, j);
#pragma unroll
              for (int m = 0; m < N1; ++m) sm[ca(m)] = v[m];
            }
          }
        }
        if (MODE != MODE_FORWARD) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
          if ((tid & 31) == 0) red[tid >> 5] = lsum;
        }
        __syncthreads();
        if (MODE != MODE_FORWARD && tid == 0) {
          double acc = 0.0;
#pragma unroll 1
          for (int w = 0; w < G::NT / 32; ++w) acc += (double)red[w];
          p.loss_part[s] = acc;
        }
      }
    }
    if (MODE == MODE_FORWARD || p.loss_only) {
      __syncthreads();
      continue;
    }

    // ---------------- adjoint: slices L-1 .. lowest ----------------
#pragma unroll 1
    for (int l = L - 1; l >= lowest; --l) {
      const bool grad_here = (MODE == MODE_LOSS_GRAD) || (MODE == MODE_LAYER && l == p.layer);
      const bool go_on = (l > lowest) || (l == 0 && MODE != MODE_LAYER && p.want_dprobe);
      const float2* Tl = p.T + (size_t)l * plane + win0;
      const float2* st = stash + (MODE == MODE_LOSS_GRAD ? (size_t)l * WW : 0);
      // window gradients: [S][L][W][W] (LOSS_GRAD) or [S][W][W] (LAYER), float2 in transmission mode
      float* wg = p.wgrad + (CPLX ? 2 : 1) * (MODE == MODE_LOSS_GRAD ? ((size_t)s * L + l) * WW : (size_t)s * WW);
#pragma unroll 1
      for (int it = 0; it < G::LPG; ++it) {
        const int r = grp + G::GROUPS * it;
        const RowIdx<W> ra(r, j);
        float2 e[N1], v[N1];
        if (grad_here) {
#pragma unroll
          for (int m = 0; m < N1; ++m) e[m] = st[r * W + j + 8 * m];   // in flight during the transform
        }
#pragma unroll
        for (int m = 0; m < N1; ++m) v[m] = sm[ra(m)];
        line_fft_t<W, true>(v, tw, xb, j);   // v = chi_l (row r)
        if (grad_here) {
          // object-frame offset of this row's first element (the layer step's map is one slice)
          const size_t o = (MODE == MODE_LOSS_GRAD ? (size_t)l * plane : 0) + win0 + (size_t)r * p.Nx + j;
          if (p.dVred) {
            // added into the object-frame gradient at once (reductions in L2)
            if (CPLX) {
#pragma unroll
              for (int m = 0; m < N1; ++m) atomicAdd(reinterpret_cast<float2*>(p.dVred) + o + 8 * m, cmulc(v[m], e[m]));
            } else {
#pragma unroll
              for (int m = 0; m < N1; ++m) atomicAdd(p.dVred + o + 8 * m, p.two_sigma * fmaf(e[m].x, v[m].y, -e[m].y * v[m].x));
            }
          } else if (CPLX) {
            // dL/dconj(o_l) on the window: conj(psi_in,l) o chi_l
            float2* wg2 = reinterpret_cast<float2*>(wg) + r * W + j;
#pragma unroll
            for (int m = 0; m < N1; ++m) __stcs(wg2 + 8 * m, cmulc(v[m], e[m]));
          } else {
            // dL/dV_l on the window: 2 sigma Im(conj(E_l) chi_l)
#pragma unroll
            for (int m = 0; m < N1; ++m) __stcs(wg + r * W + j + 8 * m, p.two_sigma * fmaf(e[m].x, v[m].y, -e[m].y * v[m].x));
          }
          if (MODE == MODE_LAYER) {   // |psi_in,l|^2 (= |E_l|^2 for unimodular slices)
            if (p.illumred) {
#pragma unroll
              for (int m = 0; m < N1; ++m) atomicAdd(p.illumred + o + 8 * m, fmaf(e[m].x, e[m].x, e[m].y * e[m].y));
            } else {
#pragma unroll
              for (int m = 0; m < N1; ++m) __stcs(p.willum + s * WW + r * W + j + 8 * m, fmaf(e[m].x, e[m].x, e[m].y * e[m].y));
            }
          }
        }
        if (go_on) {
          const float2* Tr = Tl + (size_t)r * p.Nx;
#pragma unroll
          for (int m = 0; m < N1; ++m) v[m] = cmulc(v[m], Tr[j + 8 * m]);   // conj(X_l) o chi_l
          if (l == 0) {
            float2* dp = p.dprobe_part + (size_t)blockIdx.x * WW + r * W;
            if (first_dprobe) {
#pragma unroll
              for (int m = 0; m < N1; ++m) dp[j + 8 * m] = v[m];
            } else {
#pragma unroll
              for (int m = 0; m < N1; ++m) dp[j + 8 * m] = cadd(dp[j + 8 * m], v[m]);
            }
          } else {
            line_fft_t<W, false>(v, tw, xb, j);
#pragma unroll
            for (int m = 0; m < N1; ++m) sm[ra(m)] = v[m];
          }
        }
      }
      if (l == 0 && go_on) first_dprobe = false;
      if (!go_on || l == 0) break;
      __syncthreads();
      // columns of G^H: F, x conj(H) / W^2, F^-1
#pragma unroll 1
      for (int it = 0; it < G::LPG; ++it) {
        const int c = grp + G::GROUPS * it;
        const ColIdx<W> ca(c, j);
        float2 v[N1];
#pragma unroll
        for (int m = 0; m < N1; ++m) v[m] = sm[ca(m)];
        line_fft_t<W, false>(v, tw, xb, j);
        const float2 hx = s_h1[c];
#pragma unroll
        for (int m = 0; m < N1; ++m) v[m] = cmulc(v[m], cmul(s_h1[j + 8 * m], hx));
        line_fft_t<W, true>(v, tw, xb, j);
#pragma unroll
        for (int m = 0; m < N1; ++m) sm[ca(m)] = v[m];
      }
      __syncthreads();
    }
    __syncthreads();
  }

  // a CTA whose every position was skipped still owns a (zero) probe partial
  if ((MODE == MODE_LOSS_GRAD || MODE == MODE_PROBE) && p.want_dprobe && first_dprobe) {
    float2* dp = p.dprobe_part + (size_t)blockIdx.x * WW;
    for (size_t i = tid; i < WW; i += G::NT) dp[i] = make_float2(0.f, 0.f);
  }
}

// ----------------------------------------------------------------------------
// launch helpers
// ----------------------------------------------------------------------------
template <int MODE, bool CPLX>
struct Kernel64 {
  static constexpr int NT = Geo<64>::NT, CLUSTER = 1;
  static constexpr size_t SMEM = position_smem_bytes<64>();
  static void (*fn())(const PosParams) { return position_kernel<64, MODE, CPLX>; }
};

template <bool CPLX>
static cudaError_t launch_64(int mode, const PosParams& p, int grid, cudaStream_t st) {
  switch (mode) {
    case MODE_FORWARD: return launch_position_as<Kernel64<MODE_FORWARD, CPLX>>(p, grid, st);
    case MODE_LOSS_GRAD: return launch_position_as<Kernel64<MODE_LOSS_GRAD, CPLX>>(p, grid, st);
    case MODE_LAYER: return launch_position_as<Kernel64<MODE_LAYER, CPLX>>(p, grid, st);
    default: return launch_position_as<Kernel64<MODE_PROBE, CPLX>>(p, grid, st);
  }
}

template <int W>
cudaError_t launch_wave(int mode, const PosParams& p, int grid, cudaStream_t st);
template <int W>
cudaError_t launch_again(int mode, const PosParams& p, int grid, cudaStream_t st);
template <int W>
int wave_slots(int sms);

// `grid` counts position slots: CTAs for W = 64 / 128, four-CTA clusters for W = 256.
cudaError_t launch_position_kernel(int win, int mode, const PosParams& p, int grid, cudaStream_t st) {
  if (win == 128) return launch_wave<128>(mode, p, grid, st);
  if (win == 256) return launch_wave<256>(mode, p, grid, st);
  // the forward model reads the slices the same way in both parametrisations
  return p.cplx && mode != MODE_FORWARD ? launch_64<true>(mode, p, grid, st) : launch_64<false>(mode, p, grid, st);
}

// Whether a pass may leave positions to a second launch (msp_wave.cuh), which has to follow it.
bool position_kernel_leaves_positions(int win, int mode, const PosParams& p) {
  return win != 64 && mode != MODE_FORWARD && !p.loss_only;
}
cudaError_t launch_position_again(int win, int mode, const PosParams& p, int grid, cudaStream_t st) {
  return win == 128 ? launch_again<128>(mode, p, grid, st) : launch_again<256>(mode, p, grid, st);
}

// Positions the fused kernel processes at once on the current device (its persistent grid): resident CTAs for
// W = 64 / 128, resident four-CTA clusters for W = 256. Of the gradient pass, for every mode: the workspace holds a
// stash slot and a probe partial for each. (At W = 64 a forward or probe pass alone would fit three CTAs to an SM, not two.)
int position_slots(int win) {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (win == 128) return wave_slots<128>(sms);
  if (win == 256) return wave_slots<256>(sms);
  using K = Kernel64<MODE_LOSS_GRAD, false>;
  int n = 0;
  cudaFuncSetAttribute(K::fn(), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)K::SMEM);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, K::fn(), K::NT, K::SMEM);
  return sms * (n < 1 ? 1 : n);
}

}  // namespace msp
