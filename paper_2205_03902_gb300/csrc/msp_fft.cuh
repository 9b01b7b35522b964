// msp_fft.cuh -- 2-D FFT building blocks for sm_103a: line transforms by groups of eight threads (W = 64),
// small transforms in registers (W = 128, 256), and the residual of the far field.
//
// The Fourier operator F of the multislice model (Sec. 2.1 / 2.2) is the
// unnormalised 2-D DFT of a W x W wave.  A W-point line transform by a group is split
// W = N1 * 8 (four-step Cooley-Tukey): eight threads share one line, thread j
// holds the line elements j, j+8, j+16, ...  (N1 complex values in registers),
//   step A: an N1-point DFT in registers over those elements,
//   step B: twiddle by w_W^(j k1),
//   exchange through a small shared buffer private to the group (warp-synchronous),
//   step C: N1/8 eight-point DFTs in registers.
// The output indices k1 + N1 k2 held by thread j are again exactly the set
// {j + 8m}, so every line transform starts and ends with the same thread/index
// ownership and consecutive passes need no re-distribution beyond the row <->
// column transpose through shared memory.
//
// There the inverse transform is conj(F(conj(x))) (unnormalised); negations fold into
// the arithmetic, so one forward kernel of small DFTs serves both directions.
//
// Shared-memory layout of the W = 64 wave: element (r, c) lives at r*W + (c ^ swz(r)),
// swz(r) = ((r & 1) << 3) | (r & 6).  With eight threads per line and four lines
// per warp this makes every row and column access of the wave free of bank
// conflicts for 8-byte elements.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace msp {

// cos(2 pi k / W) and sin(2 pi k / W) at compile time: Taylor series on [0, pi / 4], the rest by symmetry.
constexpr double series(double x, bool sine) {
  double term = sine ? x : 1.0, sum = term;
  for (int n = sine ? 2 : 1; n < 24; n += 2) {
    term = -term * x * x / (n * (n + 1));
    sum += term;
  }
  return sum;
}
constexpr double cos_turn(int k, int w) {
  k %= w;
  if (k < 0) k += w;
  if (k > w / 2) k = w - k;
  if (k > w / 4) return -cos_turn(w / 2 - k, w);
  constexpr double tau = 6.28318530717958647692;
  return 8 * k <= w ? series(tau * k / w, false) : series(tau * (w / 4 - k) / w, true);
}
constexpr double sin_turn(int k, int w) { return cos_turn(k - w / 4, w); }
// w_W^k = exp(-2 pi i k / W), rounded once
template <int W>
struct Twiddles {
  float re[W] = {}, im[W] = {};
  constexpr Twiddles() {
    for (int k = 0; k < W; ++k) {
      re[k] = (float)cos_turn(k, W);
      im[k] = (float)-sin_turn(k, W);
    }
  }
};
// in constant memory: a CTA copies its table at the start instead of evaluating it in double (about 1.3 us of
// every launch at FP64's rate)
static __constant__ Twiddles<64> kTwiddles64;
static __constant__ Twiddles<128> kTwiddles128;
static __constant__ Twiddles<256> kTwiddles256;
template <int W>
__device__ __forceinline__ float2 twiddle(int k) {
  if constexpr (W == 64) return make_float2(kTwiddles64.re[k], kTwiddles64.im[k]);
  else if constexpr (W == 128) return make_float2(kTwiddles128.re[k], kTwiddles128.im[k]);
  else return make_float2(kTwiddles256.re[k], kTwiddles256.im[k]);
}

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// a * conj(b)
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }

// cos(2 pi k / 16) and sin(2 pi k / 16) for k = 0..3 (exact values of the regular 16-gon).
constexpr float kC1 = 0.92387953251128675613f;   // cos(pi/8)
constexpr float kS1 = 0.38268343236508977173f;   // sin(pi/8)
constexpr float kR2 = 0.70710678118654752440f;   // cos(pi/4)

// v * w_16^K with w_16 = exp(-2 pi i / 16); K in [0, 16).  Trivial factors are
// special-cased so that no multiplication by 0 or 1 is issued.
template <int K>
__device__ __forceinline__ float2 tw16(float2 v) {
  constexpr int k = K & 15;
  if constexpr (k == 0) return v;
  else if constexpr (k == 4) return make_float2(v.y, -v.x);           // * (-i)
  else if constexpr (k == 8) return make_float2(-v.x, -v.y);          // * (-1)
  else if constexpr (k == 12) return make_float2(-v.y, v.x);          // * (+i)
  else if constexpr (k == 2) return make_float2(kR2 * (v.x + v.y), kR2 * (v.y - v.x));
  else if constexpr (k == 6) return make_float2(kR2 * (v.y - v.x), -kR2 * (v.x + v.y));
  else if constexpr (k == 10) return make_float2(-kR2 * (v.x + v.y), kR2 * (v.x - v.y));
  else if constexpr (k == 14) return make_float2(kR2 * (v.x - v.y), kR2 * (v.x + v.y));
  else {
    // general: (a + ib)(c - is) with c = cos(2 pi k/16), s = sin(2 pi k/16)
    constexpr float c = (k == 1 || k == 15) ? kC1 : (k == 3 || k == 13) ? kS1 : (k == 5 || k == 11) ? -kS1 : -kC1;
    constexpr float s = (k == 1 || k == 7) ? kS1 : (k == 3 || k == 5) ? kC1 : (k == 9 || k == 15) ? -kS1 : -kC1;
    return make_float2(fmaf(v.x, c, v.y * s), fmaf(v.y, c, -v.x * s));
  }
}

// Radix-2 decimation-in-time butterflies of an N-point DFT, N <= 16.
template <int N, int K>
__device__ __forceinline__ void dit_bfly(const float2* E, const float2* O, float2* X) {
  if constexpr (K < N / 2) {
    const float2 t = tw16<(K * 16) / N>(O[K]);
    X[K] = cadd(E[K], t);
    X[K + N / 2] = csub(E[K], t);
    dit_bfly<N, K + 1>(E, O, X);
  }
}

// X[k] = sum_n x[n*S] w_N^(n k), forward DFT in registers (all indices compile-time).
template <int N, int S>
__device__ __forceinline__ void dft(const float2* x, float2* X) {
  if constexpr (N == 1) {
    X[0] = x[0];
  } else if constexpr (N == 2) {
    X[0] = cadd(x[0], x[S]);
    X[1] = csub(x[0], x[S]);
  } else {
    float2 E[N / 2], O[N / 2];
    dft<N / 2, 2 * S>(x, E);
    dft<N / 2, 2 * S>(x + S, O);
    dit_bfly<N, 0>(E, O, X);
  }
}

__device__ __forceinline__ int swz(int r) { return ((r & 1) << 3) | (r & 6); }

// Twiddles of thread j held in registers: w^(j k) for k < 8, and w^(j k) = w^(8j) w^(j (k - 8))
// for k >= 8 (one extra rounded product).  `t` is the shared table [k1 * T + j].
template <int W, int T = 8>
struct RegisterTwiddles {
  float2 r[8];   // r[0] unused (k1 = 0 is never multiplied); r[k] = w^(j k), k = 1..7
  float2 w8;     // w^(8 j)
  RegisterTwiddles() = default;
  __device__ __forceinline__ RegisterTwiddles(const float2* __restrict__ t, int j) {
#pragma unroll
    for (int k = 1; k < 8; ++k) r[k] = t[k * T + j];
    w8 = (W / T > 8) ? t[8 * T + j] : make_float2(1.f, 0.f);
  }
  template <int K1>
  __device__ __forceinline__ float2 get() const {
    if constexpr (K1 < 8) return r[K1];
    else if constexpr (K1 == 8) return w8;
    else return cmul(w8, r[K1 - 8]);
  }
};

template <int K1, int N1, typename Tw, int STRIDE = 1>
__device__ __forceinline__ void twiddle_store(const float2* y, float2* xw, const Tw& tw) {
  if constexpr (K1 < N1) {
    xw[K1 * STRIDE] = (K1 == 0) ? y[K1] : cmul(y[K1], tw.template get<K1>());
    twiddle_store<K1 + 1, N1, Tw, STRIDE>(y, xw, tw);
  }
}

// Line transform of a W-point line held by eight threads, in place in `v`: on entry v[m] is line element
// j + 8 m, on exit v[m] is spectrum element j + 8 m.  W = 8 N1 (four-step): step A is an N1-point DFT in
// registers over x[8 n1 + j], step B the twiddles w_W^(j k1), then an exchange, then step C, N1/8 eight-point
// DFTs.  `tw.get<k1>()` = w_W^(j k1) (forward sign).  INV selects the unnormalised inverse.
// Exchange layout with the step-A results transposed: row k1 of
// the group's buffer holds Y[0..7][k1] at stride kXRow, so thread j writes Y[j][k1] at
// xb[k1 kXRow + j] (64-bit stores) and reads its step-C operands Y[0..7][k1] for
// k1 = j + 8 mc as four 128-bit loads per row.  With kXRow = 10 and group buffers
// kXGroup(N1) apart (an odd multiple of eight float2) both patterns are conflict-free.
constexpr int kXRow = 10;
__host__ __device__ constexpr int kXGroup(int n1) { return n1 * kXRow + 8; }

template <int W, bool INV, typename Tw>
__device__ __forceinline__ void line_fft_t(float2 (&v)[W / 8], const Tw& tw, float2* xb, int j) {
  constexpr int N1 = W / 8;
  constexpr int NC = N1 / 8;
  float2 y[N1];
  if constexpr (INV) {
#pragma unroll
    for (int m = 0; m < N1; ++m) v[m] = cconj(v[m]);
  }
  dft<N1, 1>(v, y);
  twiddle_store<0, N1, Tw, kXRow>(y, xb + j, tw);
  __syncwarp();
  float2 b[NC][8];
#pragma unroll
  for (int mc = 0; mc < NC; ++mc) {
    const float4* row = reinterpret_cast<const float4*>(xb + (j + 8 * mc) * kXRow);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 f = row[q];
      b[mc][2 * q] = make_float2(f.x, f.y);
      b[mc][2 * q + 1] = make_float2(f.z, f.w);
    }
  }
  __syncwarp();
#pragma unroll
  for (int mc = 0; mc < NC; ++mc) {
    float2 X[8];
    dft<8, 1>(b[mc], X);
#pragma unroll
    for (int k2 = 0; k2 < 8; ++k2) v[mc + NC * k2] = INV ? cconj(X[k2]) : X[k2];
  }
}

// The same transform of a line held by T threads (8 or 16), exchanged through W places at `xb`, in an order that is free of
// bank conflicts within a warp (`odd`: 1 in every second group of eight). Operation for operation line_fft_t, so the results
// have the same bits.
template <int K1, int N1, int T, typename Tw>
__device__ __forceinline__ void twiddle_store_permuted(const float2* y, const Tw& tw, float2* xb, int j, int odd) {
  if constexpr (K1 < N1) {
    xb[(K1 ^ odd) * T + (j ^ (K1 & (T - 1)))] = (K1 == 0) ? y[K1] : cmul(y[K1], tw.template get<K1>());
    twiddle_store_permuted<K1 + 1, N1, T>(y, tw, xb, j, odd);
  }
}
template <int W, int T, bool INV, typename Tw>
__device__ __forceinline__ void line_fft_permuted(float2 (&v)[W / T], const Tw& tw, float2* xb, int j, int odd) {
  constexpr int N1 = W / T;
  constexpr int NC = N1 / T;
  float2 y[N1], b[NC][T];
  if constexpr (INV) {
#pragma unroll
    for (int m = 0; m < N1; ++m) v[m] = cconj(v[m]);
  }
  dft<N1, 1>(v, y);
  twiddle_store_permuted<0, N1, T>(y, tw, xb, j, odd);
  __syncwarp();
#pragma unroll
  for (int mc = 0; mc < NC; ++mc)
#pragma unroll
    for (int n2 = 0; n2 < T; ++n2) b[mc][n2] = xb[((j + T * mc) ^ odd) * T + (n2 ^ j)];
  __syncwarp();   // the places are reused by this group's next transform
#pragma unroll
  for (int mc = 0; mc < NC; ++mc) {
    float2 X[T];
    dft<T, 1>(b[mc], X);
#pragma unroll
    for (int k2 = 0; k2 < T; ++k2) v[mc + NC * k2] = INV ? cconj(X[k2]) : X[k2];
  }
}

// ---------------------------------------------------------------------------
// residual of the far field
// ---------------------------------------------------------------------------
// Amplitude-flow residual of a far-field value: the factor f of R = f Psi, f = 1 - sqrt(I) / |Psi| (1 where
// Psi counts as zero), and the loss term added to `lsum`.
__device__ __forceinline__ float residual_exact(float a2, float I, float zthr2, float& lsum) {
  const float a = sqrtf(a2), rt = sqrtf(I);
  const float d = rt - a;
  lsum = fmaf(d, d, lsum);
  return (a2 > zthr2) ? (1.f - rt / a) : 1.f;   // a2 > zthr2 >= 0 implies a > 0
}
// The same for a2 and I in range (residual_in_range) without a branch: zero counts are the usual case in a pattern, and
// the library's square root and quotient leave their short path for zero operands (measured: of 165
// thousand cycles per position, W = 128, L = 4, 19 went into this pass; W = 64, L = 5, 2115 positions,
// loss and gradients: 398 -> 383 us).  sqrt(x) = s + (x - s s) y / 2 and n / a = q + (n - q a) y from the
// reciprocal square root y, with one fused residual each (Markstein 1990): the residuals are exact, so each result is
// within half an ulp but for ties (tests/test_gpu_device_functions.py).
__device__ __forceinline__ float residual_fast(float a2, float I, float zthr2, float& lsum) {
  const float y = rsqrtf(a2), z = rsqrtf(I);
  float a = a2 * y, rt = I * z;
  a = fmaf(fmaf(-a, a, a2), 0.5f * y, a);
  rt = fmaf(fmaf(-rt, rt, I), 0.5f * z, rt);
  a = a2 > 0.f ? a : 0.f;
  rt = I > 0.f ? rt : 0.f;
  const float d = rt - a;
  lsum = fmaf(d, d, lsum);
  float q = rt * y;
  q = fmaf(fmaf(-q, a, rt), y, q);
  return a2 > zthr2 ? 1.f - q : 1.f;
}
// a2 = 0 or 2^-100 <= a2 < infinity (between, the residuals' last bits and the quotient leave FP32's range), 0 <= I < infinity.
// Zeros are usual: outside the aperture of empty slices the far field cancels exactly here and there, and the general form
// for a warp that holds one cost 5 % of the W = 128 gradient pass in that state.
__device__ __forceinline__ bool residual_in_range(float a2, float I) {
  constexpr uint32_t least = 27u << 23;   // 2^-100
  return __float_as_uint(a2) - 1u >= least - 1u && a2 <= 3.402823466e+38f && I >= 0.f && I <= 3.402823466e+38f;
}

// v <- f v for N far-field values of a thread and their measured intensities.
template <int N>
__device__ __forceinline__ void residual(float2 (&v)[N], const float (&I)[N], float zthr2, float& lsum) {
  bool in_range = true;
#pragma unroll
  for (int m = 0; m < N; ++m) in_range = in_range && residual_in_range(fmaf(v[m].x, v[m].x, v[m].y * v[m].y), I[m]);
#pragma unroll
  for (int m = 0; m < N; ++m) {
    const float a2 = fmaf(v[m].x, v[m].x, v[m].y * v[m].y);
    const float f = in_range ? residual_fast(a2, I[m], zthr2, lsum) : residual_exact(a2, I[m], zthr2, lsum);
    v[m] = make_float2(v[m].x * f, v[m].y * f);
  }
}

// ---------------------------------------------------------------------------
// small DFTs in registers, both directions
// ---------------------------------------------------------------------------
// cos(2 pi k / 32) for k = 0..8 (the regular 32-gon), sin by symmetry
__host__ __device__ constexpr double cos32(int k) {
  constexpr double c[9] = {1.0, 0.98078528040323044913, 0.92387953251128675613, 0.83146961230254523708,
                           0.70710678118654752440, 0.55557023301960222474, 0.38268343236508977173,
                           0.19509032201612826785, 0.0};
  return k <= 8 ? c[k] : -c[16 - k];
}
__host__ __device__ constexpr double sin32(int k) { return k <= 8 ? cos32(8 - k) : cos32(k - 8); }

// Packed FP32 pairs (sm_100 and later): one instruction works on both components.  The FP32 pipe runs
// them at half the rate of the scalar instructions (measured: 1.87 against 3.72 warp instructions per
// clock and SM), so they halve the issue slots and leave the arithmetic rate as it is.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {   // a b + c
  float2 d;
  asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%6, %7};\n\t"
      "fma.rn.f32x2 x, x, y, z;\n\tmov.b64 {%0, %1}, x;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
#define MSP_PACKED_OP(name, op)                                                                            \
  __device__ __forceinline__ float2 name(float2 a, float2 b) {                                             \
    float2 d;                                                                                              \
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t" op " x, x, y;\n\t"      \
        "mov.b64 {%0, %1}, x;\n\t}"                                                                        \
        : "=f"(d.x), "=f"(d.y)                                                                             \
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));                                                         \
    return d;                                                                                              \
  }
MSP_PACKED_OP(add2, "add.rn.f32x2")
MSP_PACKED_OP(sub2, "sub.rn.f32x2")
MSP_PACKED_OP(mul2, "mul.rn.f32x2")
#undef MSP_PACKED_OP

__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// Two complex values side by side, (re0, re1) and (im0, im1).
struct C2 {
  float2 re, im;
};
__device__ __forceinline__ C2 add(C2 a, C2 b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ C2 sub(C2 a, C2 b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
__device__ __forceinline__ float2 add(float2 a, float2 b) { return cadd(a, b); }
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return csub(a, b); }
// e + i o, e - i o
__device__ __forceinline__ void quarter(C2 e, C2 o, C2& p, C2& m) {
  p = {sub2(e.re, o.im), add2(e.im, o.re)};
  m = {add2(e.re, o.im), sub2(e.im, o.re)};
}
__device__ __forceinline__ void quarter(float2 e, float2 o, float2& p, float2& m) {
  p = make_float2(e.x - o.y, e.y + o.x);
  m = make_float2(e.x + o.y, e.y - o.x);
}
// u = (re + q im, im - q re)
__device__ __forceinline__ C2 rot_tan(C2 o, float q) {
  const float2 p = make_float2(q, q), n = make_float2(-q, -q);
  return {fma2(p, o.im, o.re), fma2(n, o.re, o.im)};
}
__device__ __forceinline__ float2 rot_tan(float2 o, float q) {
  return make_float2(fmaf(q, o.y, o.x), fmaf(-q, o.x, o.y));
}
// u = (q re + im, q im - re)
__device__ __forceinline__ C2 rot_cot(C2 o, float q) {
  const float2 p = make_float2(q, q), one = make_float2(-1.f, -1.f);
  return {fma2(p, o.re, o.im), fma2(p, o.im, mul2(one, o.re))};
}
__device__ __forceinline__ float2 rot_cot(float2 o, float q) {
  return make_float2(fmaf(q, o.x, o.y), fmaf(q, o.y, -o.x));
}
__device__ __forceinline__ C2 axpy(float m, C2 u, C2 e) {   // m u + e
  const float2 p = make_float2(m, m);
  return {fma2(p, u.re, e.re), fma2(p, u.im, e.im)};
}
__device__ __forceinline__ float2 axpy(float m, float2 u, float2 e) {
  return make_float2(fmaf(m, u.x, e.x), fmaf(m, u.y, e.y));
}

// The butterfly e + w o, e - w o with w = exp(-2 pi i K / N) (INV: conjugated), 0 <= K < N / 2, on one
// complex value (float2) or two (C2).  w is applied as its larger component times (1, tan) or (cot, 1),
// |tan|, |cot| <= 1 (Linzer and Feig, IEEE Trans. Signal Process. 1993): two fused multiply-adds for the rotation and
// four that scale and add, six operations where a complex product and two sums take eight, with no more roundings on the way.
template <int N, int K, bool INV, typename T>
__device__ __forceinline__ void butterfly(T e, T o, T& x0, T& x1) {
  if constexpr (K == 0) {
    x0 = add(e, o);
    x1 = sub(e, o);
  } else if constexpr (4 * K == N) {   // w = -i (INV: +i)
    if constexpr (INV) quarter(e, o, x0, x1);
    else quarter(e, o, x1, x0);
  } else {
    constexpr int k = K * (32 / N);
    constexpr double c = cos32(k), s = INV ? -sin32(k) : sin32(k);   // w o = (c re + s im, c im - s re)
    if constexpr (c * c >= s * s) {
      const T u = rot_tan(o, (float)(s / c));
      x0 = axpy((float)c, u, e);
      x1 = axpy((float)-c, u, e);
    } else {
      const T u = rot_cot(o, (float)(c / s));
      x0 = axpy((float)s, u, e);
      x1 = axpy((float)-s, u, e);
    }
  }
}
template <int N, int K, bool INV, typename T>
__device__ __forceinline__ void butterflies(const T* E, const T* O, T* X) {
  if constexpr (K < N / 2) {
    butterfly<N, K, INV>(E[K], O[K], X[K], X[K + N / 2]);
    butterflies<N, K + 1, INV>(E, O, X);
  }
}
// X[k] = sum_n x[n S] exp(-+2 pi i n k / N), N <= 32 (radix-2 decimation in time, unrolled)
template <int N, int S, bool INV, typename T>
__device__ __forceinline__ void fft(const T* x, T* X) {
  if constexpr (N == 1) {
    X[0] = x[0];
  } else {
    T E[N / 2], O[N / 2];
    fft<N / 2, 2 * S, INV>(x, E);
    fft<N / 2, 2 * S, INV>(x + S, O);
    butterflies<N, 0, INV>(E, O, X);
  }
}

// A 32-point transform as two 16-point ones side by side in pairs and one stage of scalars.
// fft32_dif: scalars in, spectrum out in pairs (X[2i], X[2i+1]); ifft32_dit: pairs in, scalars out.
template <int K>
__device__ __forceinline__ void dif32_stage(const float2* x, C2* ab) {
  if constexpr (K < 16) {
    const float2 a = cadd(x[K], x[K + 16]), d = csub(x[K], x[K + 16]);
    constexpr float c = (float)cos32(K), s = (float)sin32(K);
    float2 b;
    if constexpr (K == 0) b = d;
    else if constexpr (K == 8) b = make_float2(d.y, -d.x);
    else b = make_float2(fmaf(c, d.x, s * d.y), fmaf(c, d.y, -s * d.x));
    ab[K] = {make_float2(a.x, b.x), make_float2(a.y, b.y)};
    dif32_stage<K + 1>(x, ab);
  }
}
__device__ __forceinline__ void fft32_dif(const float2 (&x)[32], C2 (&X)[16]) {
  C2 ab[16];
  dif32_stage<0>(x, ab);
  fft<16, 1, false>(ab, X);
}
template <int K>
__device__ __forceinline__ void dit32_stage(const C2* eo, float2* x) {
  if constexpr (K < 16) {
    butterfly<32, K, true>(make_float2(eo[K].re.x, eo[K].im.x), make_float2(eo[K].re.y, eo[K].im.y), x[K], x[K + 16]);
    dit32_stage<K + 1>(eo, x);
  }
}
__device__ __forceinline__ void ifft32_dit(const C2 (&X)[16], float2 (&x)[32]) {
  C2 eo[16];
  fft<16, 1, true>(X, eo);
  dit32_stage<0>(eo, x);
}

}  // namespace msp
