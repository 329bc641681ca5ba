// Conversions and tests on the bit patterns of floats and doubles, and the two
// FP64 recipes that start from an FP32 quotient.  GB300 issues FP64 compares,
// conversions and divisions at the FP64 rate, 1/64 of the FP32 rate; integer
// instructions do the same exactly.  Plain C++ outside a CUDA compiler (there
// the quotient is the host's), so that these very functions can be run on the
// host.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#include <cuda_runtime.h>
#define FEMPIC_HD __host__ __device__ __forceinline__
#else
#define FEMPIC_HD static inline
#endif
#ifndef FEMPIC_HOST_FAST_DIV
#define FEMPIC_HOST_FAST_DIV(a, b) ((a) / (b))
#endif

namespace fempic {

FEMPIC_HD int hi_word(double r) {
#ifdef __CUDA_ARCH__
  return __double2hiint(r);
#else
  uint64_t u;
  memcpy(&u, &r, 8);
  return (int)(uint32_t)(u >> 32);
#endif
}

FEMPIC_HD int lo_word(double r) {
#ifdef __CUDA_ARCH__
  return __double2loint(r);
#else
  uint64_t u;
  memcpy(&u, &r, 8);
  return (int)(uint32_t)u;
#endif
}

FEMPIC_HD double from_words(int hi, int lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(hi, lo);
#else
  const uint64_t u = (uint64_t)(uint32_t)hi << 32 | (uint32_t)lo;
  double r;
  memcpy(&r, &u, 8);
  return r;
#endif
}

FEMPIC_HD unsigned float_word(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  uint32_t u;
  memcpy(&u, &f, 4);
  return u;
#endif
}

FEMPIC_HD float from_word(unsigned u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float f;
  memcpy(&f, &u, 4);
  return f;
#endif
}

FEMPIC_HD float mul_rn(float a, float b) {   // never contracted
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}

FEMPIC_HD float fast_div(float a, float b) {   // within 2 ulp for 2^-126 <= |b| <= 2^126
#ifdef __CUDA_ARCH__
  return __fdividef(a, b);
#else
  return FEMPIC_HOST_FAST_DIV(a, b);
#endif
}

// Sign and finiteness tests of doubles on their bit patterns: integer
// instructions instead of FP64 compares, which GB300 issues at the FP64 rate.
FEMPIC_HD bool finite_bits(double r) {
  return (((unsigned)hi_word(r) >> 20) & 0x7ffu) != 0x7ffu;
}

FEMPIC_HD bool negative_bits(double r) {   // r < 0 for finite r (-0 is not negative)
  const int hi = hi_word(r);
  return hi < 0 && (((unsigned)hi & 0x7fffffffu) | (unsigned)lo_word(r)) != 0u;
}

struct FF {
  float hi, lo;
};

// Exact widening of a float to double with integer operations (rebias the
// exponent, shift the significand): GB300 runs the hardware conversion at
// the FP64 rate, 1/64 of the FP32 rate.  Zero keeps its sign; subnormal,
// infinite and NaN inputs take the hardware conversion, so the result is the
// double the conversion gives for every float.
FEMPIC_HD double f32_to_f64(float f) {
  const unsigned u = float_word(f);
  const unsigned e = (u >> 23) & 0xffu, m = u & 0x7fffffu, sign = u & 0x80000000u;
  if (e - 1u >= 0xfeu) {
    if ((u << 1) == 0u) return from_words((int)sign, 0);
    return (double)f;
  }
  return from_words((int)(sign | ((e + 896u) << 20) | (m >> 3)), (int)(m << 29));
}

// r = hi + lo: hi keeps the leading 24 bits of the FP64 significand
// (truncated, so exactly a float), lo the remaining 29 bits rounded to FP32.
// |r| outside [2^-126, 2^128) maps to 0 (non-finite values are rejected
// before this is called).
FEMPIC_HD FF split_f64(double r) {
  const unsigned hi = (unsigned)hi_word(r), lo = (unsigned)lo_word(r);
  const unsigned e = (hi >> 20) & 0x7ffu;
  if (e < 897u || e > 1150u) return FF{0.f, 0.f};
  const unsigned sign = hi & 0x80000000u;
  const float fhi = from_word(sign | ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
  const float scale = e > 948u ? from_word((e - 948u) << 23) : 0.f;   // 2^(e - 1075)
  const float flo = mul_rn((float)(lo & 0x1fffffffu), scale);
  return FF{fhi, sign ? -flo : flo};
}

// FP64 -> FP32, nearest even, with integer operations (the hardware
// conversion runs at the FP64 rate); values outside the normal FP32 range
// take it.
FEMPIC_HD float f64_to_f32(double r) {
  const unsigned hi = (unsigned)hi_word(r), lo = (unsigned)lo_word(r);
  const unsigned e = (hi >> 20) & 0x7ffu;
  if (e - 897u >= 253u) return (float)r;
  const unsigned m = ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
  const unsigned rest = lo & 0x1fffffffu;
  const unsigned up = rest > 0x10000000u || (rest == 0x10000000u && (m & 1u)) ? 1u : 0u;
  return from_word((hi & 0x80000000u) | (m + up));   // a carry moves into the exponent
}

// The same with zero left to the hardware conversion: in the per-tet pass of the
// mixed downshifted step, where a DoF is rarely zero, the test for it costs more
// than it saves (10537 against 10328 us for eight steps of that pass's case).
FEMPIC_HD double widen32(float f) {
  const unsigned u = float_word(f), e = (u >> 23) & 0xffu;
  if (e - 1u >= 0xfeu) return (double)f;
  return from_words((int)((u & 0x80000000u) | ((e + 896u) << 20) | ((u & 0x7fffffu) >> 3)), (int)(u << 29));
}

// Leading 24 bits of an FP64 value as a float (truncated, so at most 2^-23
// relative below it in magnitude): 0 below 2^-126, infinite from 2^128 on.
FEMPIC_HD float trunc32(double r) {
  const unsigned hi = (unsigned)hi_word(r), lo = (unsigned)lo_word(r);
  const unsigned e = (hi >> 20) & 0x7ffu, sign = hi & 0x80000000u;
  if (e < 897u) return 0.f;
  if (e > 1150u) return from_word(sign | 0x7f800000u);
  return from_word(sign | ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
}

// 1 / w for w >= 1 within 0.502 ulp: an FP32 reciprocal (relative error e
// below 2^-21) and one step r (1 + e + e^2) of the residual series, whose
// remainder e^3 lies below an FP64 ulp.  Past the FP32 range (and for a
// non-finite w) the division.
FEMPIC_HD double recip_ge1(double w) {
  if ((unsigned)hi_word(w) >= (1143u << 20)) return 1.0 / w;
  const double r = f32_to_f64(fast_div(1.0f, trunc32(w)));
  const double e = fma(-w, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// Exit face of the piece with end barycentrics la -> lb (entry face
// excluded): the smallest s_k = la_k / (la_k - lb_k) clamped at 0, the lowest
// face on ties, -1 when the piece stays inside.  FP32 quotients order the
// faces (relative error below 2^-20: la >= 0 > lb, so la - lb does not
// cancel) and one FP64 division serves the winner; where two faces come
// within 2^-17, a start lies outside (la < 0) or so near a face that FP32
// loses bits of it (0 < la < 2^-104), or a quotient is not finite or below
// 2^-100 without being 0, every face is divided in FP64.
FEMPIC_HD int exit_face64(const double la[4], const double lb[4], int entry, double& smin) {
  float q1 = INFINITY, q2 = INFINITY;
  bool close = false;
  int kx = -1;
  double a = 0.0, b = 0.0;
#pragma unroll
  for (int k = 0; k < 4; k++) {
    if (k == entry || !negative_bits(lb[k])) continue;
    const float x = trunc32(la[k]), y = trunc32(lb[k]);
    const float q = fast_div(x, x - y);
    const unsigned h = (unsigned)hi_word(la[k]);
    close = close || !(q >= 0.f && q < INFINITY) || !(h - (919u << 20) < (1128u << 20) || (h | (unsigned)lo_word(la[k])) == 0u);
    if (q < q1) {
      q2 = q1;
      q1 = q;
      kx = k;
      a = la[k];
      b = lb[k];
    } else {
      q2 = fminf(q2, q);
    }
  }
  smin = INFINITY;
  if (close || (kx >= 0 && (q2 <= q1 + q1 * 0x1p-17f || (q1 < 0x1p-100f && (hi_word(a) | lo_word(a)) != 0)))) {
    kx = -1;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      if (k == entry || !negative_bits(lb[k])) continue;
      double sk = la[k] / (la[k] - lb[k]);
      if (sk < 0.0) sk = 0.0;
      if (sk < smin) {
        smin = sk;
        kx = k;
      }
    }
  } else if (kx >= 0) {
    smin = a / (a - b);
  }
  return kx;
}

}  // namespace fempic
