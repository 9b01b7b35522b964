// msp_wave.cuh -- the fused per-position kernel of W = 128 and W = 256, its launches and its grid; msp_wave128.cu and
// msp_wave256.cu compile one window size each.  The outline of a pass is in msp_position.cu.
#pragma once
#include <type_traits>

#include "msp_fft.cuh"
#include "msp_kernels.cuh"
#include "msp_tc.cuh"

namespace msp {

// ----------------------------------------------------------------------------
// W = 128, 256: the wave in registers, two values per packed instruction
// ----------------------------------------------------------------------------
// 512 threads hold the wave (W = 256: four CTAs of 512), 32 complex values each; shared memory only carries it
// from one pass to the next.  The 2-D transform is split over the two axes together (four-step Cooley-Tukey per
// axis, spectrum index k1 + N1 k2): W = 128 row n = 16 n1 + n2 and column n = 32 n1 + n2, W = 256 row
// n = 64 n1 + n2 and column n = 32 n1 + n2.
//   pass A   the 8- and 4-point transforms of the two axes over their n1.  The warp (with the CTA, W = 256) is the
//            row's n2, the lane the column's n2: every global access (transmission window, window gradients) is
//            a run of 32 consecutive elements of a row;
//   pass B   the 32-point column transform over the column's n2, one row of 32 values per thread;
//   pass C   the row transform over the row's n2 of two columns per thread, the propagator (or the far field and
//            its residual), and the inverse row transform.  W = 128: 16 points.  W = 256: 64 points, 16 over
//            the warps and four over the CTAs of the cluster; the latter go through distributed shared memory in
//            16-byte accesses of consecutive addresses, between two cluster barriers.
// The inverse runs B, A.  A row's n2 stays with its warp from B through A to B, so these exchanges need warp
// synchronisation only, within the warp's own region; the CTA meets at the two sides of pass C.  Every pass
// writes back to the addresses that it read.  Spectra stay in the order of the split: the propagator and
// the patterns are indexed by k, and the inverse consumes the same order.
//
// Against line transforms by thread groups with an exchange inside each (the form of W = 64), a propagation at
// W = 128 moves the wave through shared memory four times in and out instead of six, and packed arithmetic
// needs 320 thousand warp instructions per position (L = 4) instead of 441.  What bounds it: the L1 data
// pipe (61 %), the FP32 pipe (51 %) and issue (44 %) together, with the warps of a position in step between
// two barriers.  Loss and gradients, W = 128, L = 4, 1024 positions: 0.709 -> 0.598 ms; forward model
// 0.302 -> 0.251 ms.  W = 256 against rows of the wave per CTA and columns read across the cluster in 8-byte accesses
// 2 KB apart (L = 16, 2304 positions, the whole call): 55.5 -> 44.9 ms.  It issues in 27 % of the cycles; its warps wait
// for loads from other CTAs' shared memory and the stash (long scoreboard 2.2 of 14.6 cycles per issue, queue for
// them 2.1), for shared memory (MIO 1.7, short scoreboard 1.4) and at the CTA's and the cluster's barriers (1.2 and 0.9).
namespace wave {
constexpr int NT = 512, V = 32;     // threads per CTA, values per thread
constexpr int CL = 32, RC = 16;     // column n2 extent (lanes), rows' n2 per CTA (warps)
constexpr int XS = CL + 2;          // row stride of a region (float2): 16-byte accesses of rows are conflict-free
constexpr int REGION = V * XS;
constexpr float kBand = 0.1f;       // half width of the band around the zero rule's threshold in |Psi|^2, times sqrt(L)
constexpr float kJump = 2e-6f;      // the least change of all residuals' norm that a decision is taken again for
constexpr int TBUF = 16;            // transmission values per thread that are fetched a pass ahead
constexpr size_t SMEM = ((size_t)RC * REGION + (size_t)TBUF * NT) * sizeof(float2);

// 16-byte accesses to the shared memory of a CTA of this cluster, by shared::cluster address
__device__ __forceinline__ uint32_t cluster_addr(const void* local, int rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(tc::smem_u32(local)), "r"(rank));
  return a;
}
__device__ __forceinline__ C2 cluster_load(uint32_t a) {
  C2 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.re.x), "=f"(v.re.y), "=f"(v.im.x), "=f"(v.im.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_store(uint32_t a, const C2& v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.re.x), "f"(v.re.y), "f"(v.im.x), "f"(v.im.y) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ int cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}

__device__ __forceinline__ void fetch8(float2* dst, const float2* src) {   // 8 bytes, asynchronously
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void fetch4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void fetch_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void fetch_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Half a slice of a thread's values (16 complex) in its own TMEM lane.
__device__ __forceinline__ void tmem_store(uint32_t addr, const C2 (&v)[8]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(addr),
      "f"(v[0].re.x), "f"(v[0].re.y), "f"(v[0].im.x), "f"(v[0].im.y), "f"(v[1].re.x), "f"(v[1].re.y), "f"(v[1].im.x),
      "f"(v[1].im.y), "f"(v[2].re.x), "f"(v[2].re.y), "f"(v[2].im.x), "f"(v[2].im.y), "f"(v[3].re.x), "f"(v[3].re.y),
      "f"(v[3].im.x), "f"(v[3].im.y), "f"(v[4].re.x), "f"(v[4].re.y), "f"(v[4].im.x), "f"(v[4].im.y), "f"(v[5].re.x),
      "f"(v[5].re.y), "f"(v[5].im.x), "f"(v[5].im.y), "f"(v[6].re.x), "f"(v[6].re.y), "f"(v[6].im.x), "f"(v[6].im.y),
      "f"(v[7].re.x), "f"(v[7].re.y), "f"(v[7].im.x), "f"(v[7].im.y)
      : "memory");
}
__device__ __forceinline__ C2 tmem_c2(const uint32_t* r) {
  return {make_float2(__uint_as_float(r[0]), __uint_as_float(r[1])), make_float2(__uint_as_float(r[2]), __uint_as_float(r[3]))};
}
// four values of each column of the half slice at `addr`
__device__ __forceinline__ void tmem_load(uint32_t addr, C2 (&v)[4]) {
  uint32_t r[16];
  tc::tmem_ld16(addr, r);
  tc::tmem_wait_ld();
  tc::tmem_ready(r);
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = tmem_c2(r + 4 * i);
}
// A value that the compiler has to take as new here: what is derived from it is derived again instead of
// being kept in registers across the passes.
__device__ __forceinline__ uint32_t anew(uint32_t a) {
  asm volatile("" : "+r"(a));
  return a;
}
// v w and v conj(w), w as (re, re, im, im)
__device__ __forceinline__ C2 rotate(const C2& v, const float4& w) {
  const float2 wx = make_float2(w.x, w.y), wy = make_float2(w.z, w.w);
  return {fma2(v.re, wx, neg2(mul2(v.im, wy))), fma2(v.re, wy, mul2(v.im, wx))};
}
__device__ __forceinline__ C2 rotate_back(const C2& v, const float4& w) {
  const float2 wx = make_float2(w.x, w.y), wy = make_float2(w.z, w.w);
  return {fma2(v.re, wx, mul2(v.im, wy)), fma2(v.im, wx, neg2(mul2(v.re, wy)))};
}
// a & b, tested anew at each use
__device__ __forceinline__ bool word(uint32_t a, uint32_t b) {
  return (anew(a) & b) != 0;
}

// The zero rule decides by |Psi| > tau ||p||, and R jumps by sqrt(I) there. Two forward models that round differently decide
// a value near the threshold either way: this kernel and the line transforms differ by 1.3 % of it times sqrt(L)
// (rms, W = 128 and 256, L = 1 to 16). Where counts were measured, one such decision moves dV by up to 4.5e-5 of its norm
// (W = 128, L = 4, 1024 positions: two inputs of forty), twenty times what rounding does. So a pass leaves a position with
// a value within the band (3.9 times that rms) and a jump above kJump of the far fields' norm sqrt(S) W ||p|| to
// a second launch, which takes the decisions of the whole position from the line transforms, the arithmetic of W = 64:
// they then depend on the inputs and not on the kernel. Of the decisions that differ 0.5 % lie outside the band.
// At W = 128, L = 4, 1024 positions one pass in three has such a position. Without one the second launch costs 2.2 us
// (of 680), with one or two 155 us; at W = 256, L = 16 1.1 ms (of 44.6). Slower: the decisions within the pass (the line
// transforms' code takes registers from all of it: 675 -> 715 to 812 us); every position run to its end there and only the
// difference of the residuals run again (the pass itself 680 -> 686 to 705 us, 65 us saved where no decision differs).
//
// Which of this thread's far-field values count as nonzero by that arithmetic: bit 2 k + e for value k of column
// kc + CH e (wave_kernel's pass C).  The forward model once more, every line by a group of 8 (W = 128) or 16 threads,
// the wave in `sm` (W W / RANKS values per CTA), exchanges in the places of the fetched transmissions behind it.  Called by
// every thread of the CTA (cluster), when nothing else needs these; they are free again on return.
template <int W>
__device__ __noinline__ uint32_t counted_by_lines(const float2* __restrict__ probe, const float2* __restrict__ T, size_t plane,
                                                  int Nx, int L, float2* sm, const float2* s_w, const float2* s_h1, float zthr2,
                                                  int rank, int k1r, int kc) {
  constexpr int RANKS = W == 256 ? 4 : 1, RW = W / RANKS;          // lines per CTA and direction
  constexpr int TL = W == 128 ? 8 : 16, N1 = W / TL, GROUPS = NT / TL;
  constexpr int RH = W == 128 ? 8 : 4, CH = W / CL;
  const int j = threadIdx.x % TL, grp = threadIdx.x / TL, odd = W == 128 ? grp & 1 : 0;
  float2* const xb = sm + RC * REGION + grp * W;
  static_assert(GROUPS * W <= TBUF * NT, "the groups' exchanges fit");
  RegisterTwiddles<W, TL> tw;
#pragma unroll
  for (int k = 1; k < 8; ++k) tw.r[k] = s_w[k * j];
  tw.w8 = s_w[8 * j];
  // value (r, c): row r % RW of CTA r / RW; the permutation spreads rows and columns over the banks
  auto at = [](int r, int c) { return (r % RW) * W + (c ^ (W == 128 ? swz(r) : r & 15)); };
  auto load = [&](int r, int c) {
    if constexpr (RANKS == 1) return sm[at(r, c)];
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(cluster_addr(sm + at(r, c), r / RW)) : "memory");
    return v;
  };
  auto store = [&](int r, int c, float2 v) {
    if constexpr (RANKS == 1) sm[at(r, c)] = v;
    else asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(cluster_addr(sm + at(r, c), r / RW)), "f"(v.x), "f"(v.y) : "memory");
  };
  auto sync = [] {
    if constexpr (RANKS == 1) __syncthreads();
    else cluster_sync();
  };
#pragma unroll 1
  for (int l = 0; l < L; ++l) {
#pragma unroll 1
    for (int r = rank * RW + grp; r < (rank + 1) * RW; r += GROUPS) {
      float2 v[N1], t[N1];
      const float2* Tr = T + l * plane + (size_t)r * Nx + j;
#pragma unroll
      for (int m = 0; m < N1; ++m) t[m] = Tr[TL * m];   // in flight during the transform
      if (l == 0) {
#pragma unroll
        for (int m = 0; m < N1; ++m) v[m] = probe[r * W + j + TL * m];
      } else {
#pragma unroll
        for (int m = 0; m < N1; ++m) v[m] = sm[at(r, j + TL * m)];
        line_fft_permuted<W, TL, true>(v, tw, xb, j, odd);
      }
#pragma unroll
      for (int m = 0; m < N1; ++m) v[m] = cmul(v[m], t[m]);
      line_fft_permuted<W, TL, false>(v, tw, xb, j, odd);
#pragma unroll
      for (int m = 0; m < N1; ++m) sm[at(r, j + TL * m)] = v[m];
    }
    sync();
#pragma unroll 1
    for (int c = rank * RW + grp; c < (rank + 1) * RW; c += GROUPS) {
      float2 v[N1];
#pragma unroll
      for (int m = 0; m < N1; ++m) v[m] = load(j + TL * m, c);
      line_fft_permuted<W, TL, false>(v, tw, xb, j, odd);
      if (l < L - 1) {
        const float2 hx = s_h1[c];
#pragma unroll
        for (int m = 0; m < N1; ++m) v[m] = cmul(v[m], cmul(s_h1[j + TL * m], hx));
        line_fft_permuted<W, TL, true>(v, tw, xb, j, odd);
      } else {
#pragma unroll
        for (int m = 0; m < N1; ++m) v[m].x = fmaf(v[m].x, v[m].x, v[m].y * v[m].y);
      }
#pragma unroll
      for (int m = 0; m < N1; ++m) store(j + TL * m, c, v[m]);
    }
    sync();
  }
  uint32_t counted = 0;
#pragma unroll 1
  for (int k = 0; k < 16; ++k) {
    const int r = W == 128 ? k1r + RH * k : k1r + RH * (4 * rank + (k >> 2) + 16 * (k & 3));
#pragma unroll
    for (int e = 0; e < 2; ++e) counted |= (uint32_t)(load(r, kc + CH * e).x > zthr2) << (2 * k + e);
  }
  sync();
  return counted;
}
}  // namespace wave

// AGAIN: the positions that the pass marked (p.again), with their zero-rule decisions from the line transforms. Usually there
// is none and the launch ends at once.
template <int W, int MODE, bool CPLX, bool AGAIN>
__global__ void __launch_bounds__(512, 1) wave_kernel(const PosParams p) {
  using namespace wave;
  constexpr bool kCluster = W == 256;
  constexpr int RANKS = kCluster ? 4 : 1;           // CTAs per position
  constexpr int RH = W == 128 ? 8 : 4, CH = W / CL;  // n1 extents
  constexpr int RL = W / RH;                        // rows' n2 extent: 16 warps, or 16 warps x 4 CTAs
  extern __shared__ float4 sm4[];
  float2* sm = reinterpret_cast<float2*>(sm4);
  __shared__ float2 s_w[W];     // w_W^k
  __shared__ float4 s_wd[W];    // the same, (re, re, im, im)
  __shared__ float4 s_wl[kCluster ? 8 * CL : 1];   // w_W^(lane k) at [k 32 + lane], likewise
  __shared__ float2 s_h1[W];    // h1(k) = exp(-i pi dz lambda q_k^2) / W
  __shared__ float4 s_hd[W];    // the same, (re, re, im, im)
  __shared__ float red[NT / 32];
  __shared__ float s_zthr2;
  __shared__ uint32_t s_near[2];   // whether a value of the j-th position lies within the band, in s_near[j & 1]
  __shared__ int2 s_pos[2];     // window origins of this CTA's positions, the j-th one in s_pos[j & 1]
  __shared__ uint32_t s_tmem;

  const int tid = threadIdx.x, lane = tid & 31, warp = (int)anew(tid >> 5);
  const int rank = kCluster ? cluster_rank() : 0;
  const int slot = blockIdx.x / RANKS, slots = gridDim.x / RANKS;   // position slots
  constexpr size_t WW = (size_t)W * W;
  const size_t plane = (size_t)p.Ny * p.Nx;

  if (tid < W) {
    const float2 w = twiddle<W>(tid);
    s_w[tid] = w;
    s_wd[tid] = make_float4(w.x, w.x, w.y, w.y);
  }
  if (kCluster && tid < 8 * CL) {
    const float2 w = twiddle<W>((tid / CL) * (tid % CL));
    s_wl[tid] = make_float4(w.x, w.x, w.y, w.y);
  }
  constexpr bool kStash = MODE == MODE_LOSS_GRAD || MODE == MODE_LAYER;
  wait_for_predecessor();
  if (AGAIN && p.again_any[0] == 0) return;
  if (tid < W) {
    const float2 h = p.h1[tid];
    s_h1[tid] = h;
    s_hd[tid] = make_float4(h.x, h.x, h.y, h.y);
  }
  uint32_t tm = 0;   // this thread's TMEM lane and its warp's first column
  if constexpr (kStash) {
    if (tid < 32) tc::tmem_alloc(&s_tmem, 512);
    tc::fence_before();
  }
  if (MODE != MODE_FORWARD && tid == 0) s_zthr2 = (float)p.zthr2[0];
  if (tid < 2) {
    s_near[tid] = 0;
    const int sp = slot + tid * slots;
    s_pos[tid] = !AGAIN && sp < p.S ? p.pos[sp] : make_int2(-1, -1);
  }
  __syncthreads();
  if constexpr (kStash) {
    tc::fence_after();
    tm = s_tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(128 * (warp >> 2));
  }

  // passes A and B: the row's n2 is the warp (W = 256: 4 warp + rank), in A the column's n2 the lane
  float2* const sa = sm + warp * REGION + lane;           // A: value a at sa[a XS]
  float2* const sb = sm + warp * REGION + lane * XS;      // B: this thread's row
  float2* const tb = sm + RC * REGION + tid;              // fetched transmissions: value i at tb[i NT]
  const int n2 = kCluster ? 4 * warp + rank : warp;
  const int rc = n2 * W + lane;                           // window offset of value (0, 0) in pass A
  // Value (u, k, e) of pass A, half u, element k of the eight-point transform, e of the pair: W = 128 row n1 = k,
  // column n1 = 2 u + e; W = 256 row n1 = 2 u + e, column n1 = k.  Steps of k and e in the window:
  constexpr int KW = W == 128 ? RL * W : CL, EW = W == 128 ? CL : RL * W;
  // pass C: slot a = 4 k + t of the spectra k of the eight-point and t of the four-point transforms, columns
  // kc and kc + CH
  const int sk = warp & 7, st4 = lane >> 3, xp = (lane & 7) + 8 * (warp >> 3);
  const int k1r = W == 128 ? sk : st4, k1c = W == 128 ? st4 : sk;
  float2* const sc = sm + (4 * sk + st4) * XS + 2 * xp;   // C: row n2 at sc[n2 REGION]
  const int kc = k1c + CH * 2 * xp;
  // the row k = 4 i + j of a thread's 16 far-field values of a column: k2 = k, or (W = 256) k2 = 4 rank + i + 16 j
  auto far_row = [&](int k) { return W == 128 ? k1r + RH * k : k1r + RH * (4 * rank + (k >> 2) + 16 * (k & 3)); };

  const int L = p.L;
  const bool need_stash = (MODE == MODE_LOSS_GRAD && !p.loss_only) || (MODE == MODE_LAYER);
  const int lowest = (MODE == MODE_LAYER) ? p.layer : 0;
  // TMEM slot (32 columns) of half h of slice l, or -1 for the global stash: there is room for four halves
  auto half_slot = [&](int l, int h) -> int {
    if (MODE == MODE_LAYER) return h;
    if (L <= 2) return 2 * l + h;
    return (h == 0 && l >= L - 4) ? l - (L > 4 ? L - 4 : 0) : -1;
  };
  // keeps the exit (or incident) wave of half h of slice l for the adjoint; the thread that wrote it reads it
  // back, so the pairs are kept as they are, 16 bytes per lane
  auto keep_half = [&](int l, int h, float4* st, const C2 (&q)[8]) {
    const int sl = half_slot(l, h);
    if (sl >= 0) {
      tmem_store(tm + 32u * sl, q);
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) st[(8 * h + i) * NT + tid] = make_float4(q[i].re.x, q[i].re.y, q[i].im.x, q[i].im.y);
    }
  };

  // forward pass A behind the eight-point transforms: v[half][k1] -> shared memory
  auto a_out = [&](const C2 (&v)[2][8]) {
    const uint32_t m = anew(W == 128 ? lane : n2);
    const float2 w1 = s_w[m], w2 = s_w[2 * m], w3 = s_w[3 * m];   // twiddles w_W^(n2 k1) of the four-point axis
#pragma unroll
    for (int h = 0; h < 8; ++h) {
      C2 a = v[0][h], b = v[1][h];
      if (h) {   // twiddle of the eight-point axis
        const float4 w = W == 128 ? s_wd[warp * h] : s_wl[CL * h + lane];
        a = rotate(a, w);
        b = rotate(b, w);
      }
      // four-point transform: (E, O) sums and differences in pairs, then scalars
      const C2 s = add(a, b), d = sub(a, b);
      const float2 y0 = make_float2(s.re.x + s.re.y, s.im.x + s.im.y);
      const float2 y2 = make_float2(s.re.x - s.re.y, s.im.x - s.im.y);
      const float2 y1 = make_float2(d.re.x + d.im.y, d.im.x - d.re.y);
      const float2 y3 = make_float2(d.re.x - d.im.y, d.im.x + d.re.y);
      sa[(h * 4 + 0) * XS] = y0;
      sa[(h * 4 + 1) * XS] = cmul(y1, w1);
      sa[(h * 4 + 2) * XS] = cmul(y2, w2);
      sa[(h * 4 + 3) * XS] = cmul(y3, w3);
    }
  };
  // inverse pass A up to the eight-point transforms: shared memory -> v[half][k1]
  auto a_in = [&](C2 (&v)[2][8]) {
    const uint32_t m = anew(W == 128 ? lane : n2);
    const float2 w1 = s_w[m], w2 = s_w[2 * m], w3 = s_w[3 * m];
#pragma unroll
    for (int h = 0; h < 8; ++h) {
      const float2 t0 = sa[(h * 4 + 0) * XS];
      const float2 t1 = cmulc(sa[(h * 4 + 1) * XS], w1);
      const float2 t2 = cmulc(sa[(h * 4 + 2) * XS], w2);
      const float2 t3 = cmulc(sa[(h * 4 + 3) * XS], w3);
      // (E0, E1) and (O0, i O1)
      const C2 e = {make_float2(t0.x + t2.x, t0.x - t2.x), make_float2(t0.y + t2.y, t0.y - t2.y)};
      const C2 o = {make_float2(t1.x + t3.x, t3.y - t1.y), make_float2(t1.y + t3.y, t1.x - t3.x)};
      C2 a = add(e, o), b = sub(e, o);
      if (h) {
        const float4 w = W == 128 ? s_wd[warp * h] : s_wl[CL * h + lane];
        a = rotate_back(a, w);
        b = rotate_back(b, w);
      }
      v[0][h] = a;
      v[1][h] = b;
    }
  };

  // q o X of half u of a window (q o conj(X) on the way back)
  auto transmit = [&](auto conj, int u, C2 (&q)[8]) {
#pragma unroll
    for (int h = 0; h < 8; ++h) {
      const float2 x0 = u == 0 ? tb[(2 * h) * NT] : sa[(2 * h) * XS], x1 = u == 0 ? tb[(2 * h + 1) * NT] : sa[(2 * h + 1) * XS];
      const float2 q0 = make_float2(q[h].re.x, q[h].im.x), q1 = make_float2(q[h].re.y, q[h].im.y);
      const float2 y0 = conj.value ? cmulc(q0, x0) : cmul(q0, x0), y1 = conj.value ? cmulc(q1, x1) : cmul(q1, x1);
      q[h] = {make_float2(y0.x, y1.x), make_float2(y0.y, y1.y)};
    }
  };
  constexpr std::false_type kPlain{};
  constexpr std::true_type kConj{};

  constexpr uint32_t kForward = 1, kKeep = 2, kGrad = 4, kGoOn = 8, kPropagate = 16;   // words of a pass
  // The object offset of a window's origin (a plane holds at most 4e9 values), or kNoWindow.
  constexpr uint32_t kNoWindow = 0xffffffffu;
  auto window = [&](uint32_t j) {
    const int2 ps = s_pos[j & 1];
    const bool ok = ps.x >= 0 && ps.y >= 0 && ps.x <= p.Ny - W && ps.y <= p.Nx - W;
    return ok ? (uint32_t)ps.x * (uint32_t)p.Nx + (uint32_t)ps.y : kNoWindow;
  };
  // Transmission windows arrive asynchronously: the first half of a slice's in tb,
  // fetched a pass ahead; the second half in this thread's slots of the wave, which are free between
  // a_in and a_out.  Each thread fetches what it uses itself, so no other synchronisation is needed.
  auto fetch_first = [&](const float2* T) {
    const size_t hstep = (size_t)RL * anew(p.Nx), ko = W == 128 ? hstep : CL, eo = W == 128 ? CL : hstep;
#pragma unroll
    for (int h = 0; h < 8; ++h) {
      fetch8(tb + (2 * h) * NT, T + h * ko);
      fetch8(tb + (2 * h + 1) * NT, T + h * ko + eo);
    }
  };
  auto fetch_second = [&](const float2* T) {
    const size_t hstep = (size_t)RL * anew(p.Nx), ko = W == 128 ? hstep : CL, eo = W == 128 ? CL : hstep;
#pragma unroll
    for (int h = 0; h < 8; ++h) {
      fetch8(sa + (2 * h) * XS, T + h * ko + 2 * eo);
      fetch8(sa + (2 * h + 1) * XS, T + h * ko + 3 * eo);
    }
  };

  // the window gradient of values 4 i .. 4 i + 3 of half u of slice l from chi_l = q and the stashed wave e
  auto gradient = [&](int s, int l, int u, int i, uint32_t oc, const C2* q, const C2 (&e)[4]) {
    // window gradients: [S][L][W][W] (LOSS_GRAD) or [S][W][W] (LAYER), float2 in transmission mode
    const size_t wo = (MODE == MODE_LOSS_GRAD ? ((size_t)s * L + l) * WW : (size_t)s * WW) + rc + KW * 4 * i + 2 * EW * u;
    // object-frame offset (the layer step's map is one slice)
    const size_t hstep = (size_t)RL * anew(p.Nx), ko = W == 128 ? hstep : CL, eo = W == 128 ? CL : hstep;
    const size_t om = (MODE == MODE_LOSS_GRAD ? (size_t)l * plane : 0) + oc + 4 * i * ko + 2 * u * eo;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      if (CPLX) {   // dL/dconj(o_l) on the window: conj(psi_in,l) o chi_l
        const float2 a = cmulc(make_float2(q[h].re.x, q[h].im.x), make_float2(e[h].re.x, e[h].im.x));
        const float2 b = cmulc(make_float2(q[h].re.y, q[h].im.y), make_float2(e[h].re.y, e[h].im.y));
        if (p.dVred) {   // reductions in L2
          atomicAdd(reinterpret_cast<float2*>(p.dVred) + om + h * ko, a);
          atomicAdd(reinterpret_cast<float2*>(p.dVred) + om + h * ko + eo, b);
        } else {
          __stcs(reinterpret_cast<float2*>(p.wgrad) + wo + KW * h, a);
          __stcs(reinterpret_cast<float2*>(p.wgrad) + wo + KW * h + EW, b);
        }
      } else {      // dL/dV_l on the window: 2 sigma Im(conj(E_l) chi_l)
        const float2 d = mul2(make_float2(p.two_sigma, p.two_sigma), fma2(e[h].re, q[h].im, neg2(mul2(e[h].im, q[h].re))));
        if (p.dVred) {
          atomicAdd(p.dVred + om + h * ko, d.x);
          atomicAdd(p.dVred + om + h * ko + eo, d.y);
        } else {
          __stcs(p.wgrad + wo + KW * h, d.x);
          __stcs(p.wgrad + wo + KW * h + EW, d.y);
        }
      }
      if (MODE == MODE_LAYER) {   // |psi_in,l|^2 (= |E_l|^2 for unimodular slices)
        const float2 d = fma2(e[h].re, e[h].re, mul2(e[h].im, e[h].im));
        if (p.illumred) {
          atomicAdd(p.illumred + om + h * ko, d.x);
          atomicAdd(p.illumred + om + h * ko + eo, d.y);
        } else {
          __stcs(p.willum + wo + KW * h, d.x);
          __stcs(p.willum + wo + KW * h + EW, d.y);
        }
      }
    }
  };

  // State carried from position to position: the lowest bit, the parity of the position's number in this CTA;
  // kFetched, slice 0 of the coming position is under way; kSummed, this CTA's probe-gradient partial has been
  // written.  Like the words of a pass it is tested where it is used: flags that live across a pass cost
  // registers, and the few that do not fit go to local memory at L2 latency (measured: 722 bytes of spills
  // made the loss-and-gradient pass 1.16 times as long as 230 bytes).
  constexpr uint32_t kFetched = 2, kSummed = 4;
  uint32_t state = AGAIN ? kSummed : 0u;
  auto fetch_next_first = [&]() {
    const uint32_t at = window(state + 1);
    if (at != kNoWindow) fetch_first(p.T + (at + (uint32_t)n2 * (uint32_t)p.Nx + (uint32_t)lane));
  };
  auto fetch_next_second = [&]() {
    const uint32_t at = window(state + 1);
    if (at != kNoWindow) fetch_second(p.T + (at + (uint32_t)n2 * (uint32_t)p.Nx + (uint32_t)lane));
  };
  // the origin after the next one into this position's slot; tid 0 waits for it in its next slice 0, and the
  // barriers that follow there show it to the others
  auto fetch_origin = [&](int s) {
    const int sp = s + 2 * slots;
    if (tid == 0 && sp < p.S) fetch8(reinterpret_cast<float2*>(&s_pos[state & 1]), reinterpret_cast<const float2*>(p.pos + sp));
    if (tid == 0 && sp >= p.S) s_pos[state & 1] = make_int2(-1, -1);
  };
  for (int s = slot; s < p.S; s += slots, state ^= 1) {
    uint32_t counted = 0;   // AGAIN: the decisions, bit 2 k + e for value k of column e of pass C
    if constexpr (AGAIN) {
      if (!p.again[s]) continue;
      const int2 ps = p.pos[s];   // the slots of the origins stay empty: nothing is fetched for a coming position
      __syncthreads();
      if (tid == 0) s_pos[state & 1] = ps;
      __syncthreads();
    }
    const uint32_t at = window(state);
    if (!AGAIN && at == kNoWindow) {
      if (tid == 0) atomicMax(p.err, 1);
      // outputs of a skipped position are zero; each CTA writes its share
      auto zero = [&](auto* a, size_t n) {
        for (size_t i = n / RANKS * rank + tid; i < n / RANKS * (rank + 1); i += NT) a[i] = 0.f;
      };
      constexpr int CW = CPLX ? 2 : 1;
      if (MODE == MODE_FORWARD) zero(p.I_out + s * WW, WW);
      if (MODE != MODE_FORWARD && tid == 0) {
        p.loss_part[s * RANKS + rank] = 0.0;
        if (rank == 0) p.again[s] = 0;
      }
      if (MODE == MODE_LOSS_GRAD && !p.dVred && !p.loss_only) zero(p.wgrad + CW * s * WW * L, CW * WW * L);
      if (MODE == MODE_LAYER && !p.dVred) {
        zero(p.wgrad + CW * s * WW, CW * WW);
        zero(p.willum + s * WW, WW);
      }
      state &= ~kFetched;
      __syncthreads();   // every thread has read this position's slot
      fetch_origin(s);
      fetch_commit();
      fetch_wait<0>();
      __syncthreads();
      continue;  // uniform across the CTA
    }
    const uint32_t oc = at + (uint32_t)n2 * (uint32_t)p.Nx + (uint32_t)lane;   // object offset of this thread's value (0, 0)
    float4* stash = reinterpret_cast<float4*>(p.stash + (size_t)slot * (MODE == MODE_LOSS_GRAD ? L : 1) * WW) + rank * (WW / 2 / RANKS);
    const bool forward_only = MODE == MODE_FORWARD || p.loss_only;
    if constexpr (AGAIN) counted = counted_by_lines<W>(p.probe, p.T + at, plane, p.Nx, L, sm, s_w, s_h1, s_zthr2, rank, k1r, kc);
    // what the buffer tb receives after slice l's pass on the way forward: the next slice's window, or this
    // thread's values of the measured pattern, or slice 0 of the next position
    auto fetch_after = [&](int l) {
      if (l + 1 < L) {
        fetch_first(p.T + (size_t)(l + 1) * plane + oc);
      } else if (MODE != MODE_FORWARD) {
        const float* I = p.I_meas + s * WW + kc;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          fetch4(&tb[k * NT].x, I + far_row(k) * W);
          fetch4(&tb[k * NT].y, I + far_row(k) * W + CH);
        }
      } else if (L > 1) {   // with one slice the next origin is not known yet
        fetch_next_first();
      }
      fetch_commit();
    };

    C2 v[2][8];
    {   // slice 0: probe o X_0, forward pass A
      const bool keep = need_stash && (MODE == MODE_LOSS_GRAD || p.layer == 0);
      if (!word(state, kFetched)) {
        fetch_first(p.T + oc);
        fetch_second(p.T + oc);
        fetch_commit();
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        C2 q[8];
#pragma unroll
        for (int h = 0; h < 8; ++h) {
          const float2 a = p.probe[rc + KW * h + EW * 2 * u], b = p.probe[rc + KW * h + EW * (2 * u + 1)];
          q[h] = {make_float2(a.x, b.x), make_float2(a.y, b.y)};
        }
        if (CPLX && keep) keep_half(0, u, stash, q);   // incident wave
        if (u == 0) fetch_wait<0>();
        transmit(kPlain, u, q);
        if (u == 0) fetch_after(0);
        if (!CPLX && keep) keep_half(0, u, stash, q);  // exit wave
        fft<8, 1, false>(q, v[u]);
      }
      if constexpr (kStash) tc::tmem_wait_st();
      a_out(v);
    }

    // step st < L - 1: propagate slice st to st + 1 and transmit; st = L - 1: far field, residual and the
    // adjoint of slice L - 1; st >= L: back-propagate to slice l = 2 L - 2 - st and its adjoint
#pragma unroll 1
    for (int st = 0;; ++st) {
      __syncwarp();
      {   // ---------------- pass B ----------------
        float4* q = reinterpret_cast<float4*>(sb);
        float2 x[32];
        C2 X[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float4 f = q[i];
          x[2 * i] = make_float2(f.x, f.y);
          x[2 * i + 1] = make_float2(f.z, f.w);
        }
        fft32_dif(x, X);
#pragma unroll
        for (int i = 0; i < 16; ++i) q[i] = make_float4(X[i].re.x, X[i].re.y, X[i].im.x, X[i].im.y);
      }
      // ---------------- pass C ----------------
      {
        if (MODE != MODE_FORWARD && st == L - 1) fetch_wait<0>();   // the pattern
        __syncthreads();
        C2 x[16], X[16];
#pragma unroll
        for (int n = 0; n < RC; ++n) {
          const float4 f = *reinterpret_cast<const float4*>(sc + n * REGION);
          x[n] = {make_float2(f.x, f.y), make_float2(f.z, f.w)};
        }
        fft<16, 1, false>(x, X);
        // W = 256: the row transform's n2 = 4 n21 + n22 reaches over the CTAs (n22).  The 16-point transforms over
        // n21 are local; then each CTA takes four of the sixteen k21 through the four-point transforms over n22 and
        // back, reading and writing the four CTAs' shared memory.
        uint32_t far[RANKS] = {};   // this thread's pair of row k21 = 4 rank of the other CTAs' regions
        if constexpr (kCluster) {
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            if (k) X[k] = rotate(X[k], s_wd[4 * rank * k]);
            *reinterpret_cast<float4*>(sc + k * REGION) = make_float4(X[k].re.x, X[k].re.y, X[k].im.x, X[k].im.y);
          }
#pragma unroll
          for (int r = 0; r < RANKS; ++r) far[r] = cluster_addr(sc + 4 * rank * REGION, r);
          cluster_sync();
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int r = 0; r < RANKS; ++r) x[4 * i + r] = cluster_load(far[r] + i * REGION * (uint32_t)sizeof(float2));
#pragma unroll
          for (int i = 0; i < 4; ++i) fft<4, 1, false>(x + 4 * i, X + 4 * i);
        }
        if (st != L - 1) {   // x H / W^2 (conjugated on the way back)
          const float sg = st < L ? 1.f : -1.f;
          const uint32_t c = anew(kc);
          const float2 h0 = s_h1[c], h1 = s_h1[c + CH];
          const float2 hcr = make_float2(h0.x, h1.x), hcn = make_float2(-h0.y, -h1.y);
          const float2 hcrs = make_float2(sg * h0.x, sg * h1.x), hcis = make_float2(sg * h0.y, sg * h1.y);
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            const float4 h = s_hd[far_row(k)];
            const float2 hx = make_float2(h.x, h.y), hy = make_float2(h.z, h.w);
            const float2 pr = fma2(hx, hcr, mul2(hy, hcn)), pi = fma2(hx, hcis, mul2(hy, hcrs));
            X[k] = {fma2(X[k].re, pr, neg2(mul2(X[k].im, pi))), fma2(X[k].re, pi, mul2(X[k].im, pr))};
          }
        } else if (MODE == MODE_FORWARD) {   // far field Psi
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            const float2 a2 = fma2(X[k].re, X[k].re, mul2(X[k].im, X[k].im));
            float* out = p.I_out + s * WW + far_row(k) * W + kc;
            out[0] = a2.x;
            out[CH] = a2.y;
          }
        } else {   // far field, residual R = Psi - sqrt(I) Psi / |Psi|
          const float zthr2 = s_zthr2, band = kBand * sqrtf((float)L) * zthr2;
          const float least = (kJump / (float)kZeroRuleTau) * (kJump / (float)kZeroRuleTau) * (float)p.S * (float)WW * zthr2;
          float lsum = 0.f;
          bool in_range = true, near = false;
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            const float2 a2 = fma2(X[k].re, X[k].re, mul2(X[k].im, X[k].im));
            in_range = in_range && residual_in_range(a2.x, tb[k * NT].x) && residual_in_range(a2.y, tb[k * NT].y);
          }
          auto look = [&](float a2, float I) { near = near || (fabsf(a2 - zthr2) <= band && !(fabsf(I) <= least)); };
          // the threshold of value 2 k + e
          auto threshold = [&](int i) { return !AGAIN ? zthr2 : (counted >> i) & 1 ? 0.f : INFINITY; };
          if (in_range) {
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              const float2 a2 = fma2(X[k].re, X[k].re, mul2(X[k].im, X[k].im));
              const float2 im = tb[k * NT];
              const float2 f = make_float2(residual_fast(a2.x, im.x, threshold(2 * k), lsum), residual_fast(a2.y, im.y, threshold(2 * k + 1), lsum));
              look(a2.x, im.x);
              look(a2.y, im.y);
              X[k] = {mul2(X[k].re, f), mul2(X[k].im, f)};
            }
          } else if (kCluster) {   // the slots of the wave are still being read by the other CTAs
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              const float2 a2 = fma2(X[k].re, X[k].re, mul2(X[k].im, X[k].im));
              const float2 im = tb[k * NT];
              const float2 f = make_float2(residual_exact(a2.x, im.x, threshold(2 * k), lsum), residual_exact(a2.y, im.y, threshold(2 * k + 1), lsum));
              look(a2.x, im.x);
              look(a2.y, im.y);
              X[k] = {mul2(X[k].re, f), mul2(X[k].im, f)};
            }
          } else {   // through this thread's slots of the wave, to keep the rare path short
#pragma unroll
            for (int k = 0; k < 16; ++k)
              *reinterpret_cast<float4*>(sc + k * REGION) = make_float4(X[k].re.x, X[k].re.y, X[k].im.x, X[k].im.y);
#pragma unroll 1
            for (int k = 0; k < 16; ++k) {
              float4& f = *reinterpret_cast<float4*>(sc + k * REGION);
              const float2 im = tb[k * NT];
              look(fmaf(f.x, f.x, f.z * f.z), im.x);
              look(fmaf(f.y, f.y, f.w * f.w), im.y);
              const float fx = residual_exact(fmaf(f.x, f.x, f.z * f.z), im.x, threshold(2 * k), lsum);
              const float fy = residual_exact(fmaf(f.y, f.y, f.w * f.w), im.y, threshold(2 * k + 1), lsum);
              f = make_float4(f.x * fx, f.y * fy, f.z * fx, f.w * fy);
            }
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              const float4 f = *reinterpret_cast<const float4*>(sc + k * REGION);
              X[k] = {make_float2(f.x, f.y), make_float2(f.z, f.w)};
            }
          }
          if (!AGAIN && near && !p.loss_only) {   // the position is left to the launch that decides
            if constexpr (kCluster) {
              for (int r = 0; r < RANKS; ++r)
                asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(&s_near[state & 1], r)), "r"(1) : "memory");
            } else {
              s_near[state & 1] = 1;
            }
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
          if (lane == 0) red[warp] = lsum;
        }
        if (st != L - 1 || !forward_only) {
          if constexpr (kCluster) {
#pragma unroll
            for (int i = 0; i < 4; ++i) fft<4, 1, true>(X + 4 * i, x + 4 * i);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int r = 0; r < RANKS; ++r) cluster_store(far[r] + i * REGION * (uint32_t)sizeof(float2), x[4 * i + r]);
            cluster_sync();
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              const float4 f = *reinterpret_cast<const float4*>(sc + k * REGION);
              X[k] = {make_float2(f.x, f.y), make_float2(f.z, f.w)};
              if (k) X[k] = rotate_back(X[k], s_wd[4 * rank * k]);
            }
          }
          fft<16, 1, true>(X, x);
#pragma unroll
          for (int n = 0; n < RC; ++n)
            *reinterpret_cast<float4*>(sc + n * REGION) = make_float4(x[n].re.x, x[n].re.y, x[n].im.x, x[n].im.y);
        }
      }
      if (kCluster && st == L - 1 && forward_only) cluster_sync();   // the other CTAs have read this one's regions
      else __syncthreads();
      if (st == L - 1) {
        bool ends = forward_only;   // no adjoint
        if (!AGAIN && MODE != MODE_FORWARD) {
          const uint32_t left = s_near[state & 1];
          ends = ends || left;
          if (tid == 0) {
            s_near[~state & 1] = 0;   // the coming position's; nobody looks at it before another barrier
            if (rank == 0) {
              p.again[s] = left;
              if (left) p.again_any[0] = 1;
            }
          }
        }
        // the pattern has been read: the buffer takes the last slice's window again, or the next position's first
        if (MODE != MODE_FORWARD) {
          if (!ends) fetch_first(p.T + (size_t)(L - 1) * plane + oc);
          else fetch_next_first();
        }
        if (MODE == MODE_FORWARD && L == 1) fetch_next_first();
        if (ends) fetch_next_second();
        state = (state & ~kFetched) | (window(state + 1) != kNoWindow ? kFetched : 0u);
        if (AGAIN) {
          if (tid == 0) s_pos[state & 1] = make_int2(-1, -1);
        } else {
          fetch_origin(s);
        }
        fetch_commit();
        if (MODE == MODE_FORWARD) break;
        if (!AGAIN && tid == 0) {   // the pass itself has summed the loss
          double acc = 0.0;
#pragma unroll 1
          for (int w = 0; w < NT / 32; ++w) acc += (double)red[w];
          p.loss_part[s * RANKS + rank] = acc;
        }
        if (ends) break;
      }
      {   // ---------------- inverse pass B ----------------
        float4* q = reinterpret_cast<float4*>(sb);
        float2 x[32];
        C2 X[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float4 f = q[i];
          X[i] = {make_float2(f.x, f.y), make_float2(f.z, f.w)};
        }
        ifft32_dit(X, x);
#pragma unroll
        for (int i = 0; i < 16; ++i) q[i] = make_float4(x[2 * i].x, x[2 * i].y, x[2 * i + 1].x, x[2 * i + 1].y);
      }
      __syncwarp();
      a_in(v);
      const int l = st < L - 1 ? st + 1 : 2 * L - 2 - st;
      uint32_t f = 0;   // what this pass does
      if (st < L - 1) {
        f = kForward | kGoOn;
        if (need_stash && (MODE == MODE_LOSS_GRAD || p.layer == l)) f |= kKeep;
      } else {
        if (MODE == MODE_LOSS_GRAD || (MODE == MODE_LAYER && l == p.layer)) f |= kGrad;
        if (l > lowest || (l == 0 && MODE != MODE_LAYER && p.want_dprobe)) f |= kGoOn;
        if (l > 0) f |= kPropagate;
      }
      const float2* T = p.T + (size_t)l * plane + oc;
      if (word(f, kGoOn)) fetch_second(T);
      float4* sl = stash + (MODE == MODE_LOSS_GRAD ? (size_t)l * (WW / 2) : 0);
      fetch_commit();
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        C2 q[8];
        fft<8, 1, true>(v[u], q);   // the incident wave of slice l, or chi_l
        if (word(f, kGrad)) {
          const int hs = half_slot(l, u);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            C2 e[4];
            if (hs >= 0) {
              tmem_load(tm + 32u * hs + 16u * i, e);
            } else {
#pragma unroll
              for (int h = 0; h < 4; ++h) {
                const float4 f = sl[(8 * u + 4 * i + h) * NT + tid];
                e[h] = {make_float2(f.x, f.y), make_float2(f.z, f.w)};
              }
            }
            gradient(s, l, u, i, oc, q + 4 * i, e);
          }
        }
        if (CPLX && word(f, kKeep)) keep_half(l, u, sl, q);    // incident wave
        fetch_wait<1>();
        if (word(f, kForward)) transmit(kPlain, u, q);
        else if (word(f, kGoOn)) transmit(kConj, u, q);        // conj(X_l) o chi_l
        if (u == 0) {
          if (word(f, kForward)) fetch_after(l);
          else {
            if (l > lowest) fetch_first(p.T + (size_t)(l - 1) * plane + oc);
            else fetch_next_first();
            fetch_commit();
          }
        }
        if (!CPLX && word(f, kKeep)) keep_half(l, u, sl, q);   // exit wave
        if (word(f, kForward | kPropagate)) {
          fft<8, 1, false>(q, v[u]);
        } else if (word(f, kGoOn)) {
          // this CTA's probe-gradient partial: only this thread ever adds to these values, one position
          // after another, so the order of the sums is fixed
          float2* dp = p.dprobe_part + (size_t)slot * WW + rc + EW * 2 * u;
#pragma unroll
          for (int h = 0; h < 8; ++h) {
            const float2 a = make_float2(q[h].re.x, q[h].im.x), b = make_float2(q[h].re.y, q[h].im.y);
            float2* d = dp + KW * h;
            if (!word(state, kSummed)) {
              d[0] = a;
              d[EW] = b;
            } else {   // (a reduction in L2 would flush subnormal sums)
              d[0] = cadd(d[0], a);
              d[EW] = cadd(d[EW], b);
            }
          }
        }
      }
      if constexpr (kStash) tc::tmem_wait_st();
      if (!word(f, kForward) && l == 0 && word(f, kGoOn)) state |= kSummed;
      if (!word(f, kForward) && (l == 0 || !word(f, kGoOn))) {
        fetch_next_second();
        fetch_commit();
        break;
      }
      a_out(v);
    }
  }

  // a CTA whose every position was skipped still owns a (zero) probe partial
  if ((MODE == MODE_LOSS_GRAD || MODE == MODE_PROBE) && p.want_dprobe && !(state & kSummed)) {
    float2* dp = p.dprobe_part + (size_t)slot * WW;
    for (size_t i = WW / RANKS * rank + tid; i < WW / RANKS * (rank + 1); i += NT) dp[i] = make_float2(0.f, 0.f);
  }
  if constexpr (kStash) {
    tc::fence_before();
    __syncthreads();
    if (tid < 32) {
      tc::fence_after();
      tc::tmem_dealloc(s_tmem, 512);
    }
  }
}

// ----------------------------------------------------------------------------
// launch helpers
// ----------------------------------------------------------------------------
template <int W, int MODE, bool CPLX, bool AGAIN = false>
struct WaveKernel {
  static constexpr int NT = wave::NT, CLUSTER = W == 256 ? 4 : 1;
  static constexpr size_t SMEM = wave::SMEM;
  static void (*fn())(const PosParams) { return wave_kernel<W, MODE, CPLX, AGAIN>; }
};

template <int W, bool CPLX>
static cudaError_t launch_wave_of(int mode, const PosParams& p, int grid, cudaStream_t st) {
  switch (mode) {
    case MODE_FORWARD: return launch_position_as<WaveKernel<W, MODE_FORWARD, CPLX>>(p, grid, st);
    case MODE_LOSS_GRAD: return launch_position_as<WaveKernel<W, MODE_LOSS_GRAD, CPLX>>(p, grid, st);
    case MODE_LAYER: return launch_position_as<WaveKernel<W, MODE_LAYER, CPLX>>(p, grid, st);
    default: return launch_position_as<WaveKernel<W, MODE_PROBE, CPLX>>(p, grid, st);
  }
}
template <int W>
cudaError_t launch_wave(int mode, const PosParams& p, int grid, cudaStream_t st) {
  // the forward model reads the slices the same way in both parametrisations
  if (p.cplx && mode != MODE_FORWARD) return launch_wave_of<W, true>(mode, p, grid, st);
  return launch_wave_of<W, false>(mode, p, grid, st);
}

// The positions of a pass just launched that it left to the line transforms.
template <int W, bool CPLX>
static cudaError_t launch_again_of(int mode, const PosParams& p, int grid, cudaStream_t st) {
  switch (mode) {
    case MODE_LOSS_GRAD: return launch_position_as<WaveKernel<W, MODE_LOSS_GRAD, CPLX, true>>(p, grid, st);
    case MODE_LAYER: return launch_position_as<WaveKernel<W, MODE_LAYER, CPLX, true>>(p, grid, st);
    default: return launch_position_as<WaveKernel<W, MODE_PROBE, CPLX, true>>(p, grid, st);
  }
}
template <int W>
cudaError_t launch_again(int mode, const PosParams& p, int grid, cudaStream_t st) {
  return p.cplx ? launch_again_of<W, true>(mode, p, grid, st) : launch_again_of<W, false>(mode, p, grid, st);
}

// Positions that are resident at once on this device: one per CTA of 512 threads (W = 128), or per four-CTA cluster.
template <int W>
int wave_slots(int sms) {
  using K = WaveKernel<W, MODE_LOSS_GRAD, false>;
  cudaFuncSetAttribute(K::fn(), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)K::SMEM);
  int n = 0;
  if constexpr (K::CLUSTER == 1) {
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, K::fn(), K::NT, K::SMEM);
    return sms * (n < 1 ? 1 : n);
  } else {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(K::CLUSTER);
    cfg.blockDim = dim3(K::NT);
    cfg.dynamicSmemBytes = K::SMEM;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = K::CLUSTER;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, K::fn(), &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    return n < 1 ? 1 : n;
  }
}

}  // namespace msp
