// Velocity rule and Adams-Bashforth velocity of the downshifted integrator
// (Sec. III-D; include/fempic_downshift.h), per particle.  The step kernels
// that run it (fempic_env.cu) go on to track and deposit the AB4 segment in
// the same pass, so a particle's state is read and written once.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "fempic_downshift.h"
#include "fempic_internal.h"

namespace fempic {

// Per-tet envelope coefficients: Re (E0, W, B0, beta), Im (E0, W, B0, beta),
// a flag word (0, or 1 when a DoF of the tet is not finite), padding.
constexpr int kDsCoef64 = 22;   // doubles per tet
constexpr int kDsCoef32 = 24;   // floats per tet

struct DsRule {
  int64_t n;
  void* h;                      // history planes [FEMPIC_DS_PLANES][n], the velocity type
  const double* coef;           // FP64 form: [nt][kDsCoef64]
  const float* coef32;          // mixed forms: [nt][kDsCoef32]
  int32_t start;
  double qm[kMaxSpecies];
  double w[24];                 // M^r[3], M^i[3], L^r[3][3], L^i[3][3]
  float qm32[kMaxSpecies];      // mixed forms: the same rounded to FP32
  float w32[24];
};

template <typename R>
__device__ __forceinline__ void ds_cross3(const R a[3], const R b[3], R o[3]) {
  o[0] = a[1] * b[2] - a[2] * b[1];
  o[1] = a[2] * b[0] - a[0] * b[2];
  o[2] = a[0] * b[1] - a[1] * b[0];
}

// History of a particle: v^{n-1..n-3} and the samples of the last two levels.
template <typename R>
struct DsHistory {
  R vh[3][3], f1[12], f2[12];
};

template <typename R>
__device__ __forceinline__ void ds_load(const DsRule& A, int64_t p, DsHistory<R>& h) {
  if (A.start) return;   // filled from this step's own values (ds_fill)
  const R* H = static_cast<const R*>(A.h);
  const int64_t n = A.n;
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int a = 0; a < 3; a++) h.vh[i][a] = H[(FEMPIC_DS_VH + 3 * i + a) * n + p];
#pragma unroll
  for (int c = 0; c < 12; c++) {
    h.f1[c] = H[(FEMPIC_DS_F + c) * n + p];
    h.f2[c] = H[(FEMPIC_DS_F + 12 + c) * n + p];
  }
}

template <typename R>
__device__ __forceinline__ void ds_fill(const DsRule& A, const R v0[3], const R cur[12], DsHistory<R>& h) {
  if (!A.start) return;   // constant extrapolation backwards
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int a = 0; a < 3; a++) h.vh[i][a] = v0[a];
#pragma unroll
  for (int c = 0; c < 12; c++) h.f1[c] = h.f2[c] = cur[c];
}

// The history one step on: this step's velocity and sample in front.
template <typename R>
__device__ __forceinline__ void ds_store(const DsRule& A, int64_t p, const R v0[3], const R cur[12],
                                         const DsHistory<R>& h) {
  R* H = static_cast<R*>(A.h);
  const int64_t n = A.n;
#pragma unroll
  for (int a = 0; a < 3; a++) {
    H[(FEMPIC_DS_VH + 6 + a) * n + p] = h.vh[1][a];
    H[(FEMPIC_DS_VH + 3 + a) * n + p] = h.vh[0][a];
    H[(FEMPIC_DS_VH + a) * n + p] = v0[a];
  }
#pragma unroll
  for (int c = 0; c < 12; c++) {
    H[(FEMPIC_DS_F + 12 + c) * n + p] = h.f1[c];
    H[(FEMPIC_DS_F + c) * n + p] = cur[c];
  }
}

// A particle's wall mirrors also mirror its velocity history.
template <typename R>
__device__ __forceinline__ void ds_mirror(const DsRule& A, int64_t p, unsigned flips) {
  R* H = static_cast<R*>(A.h);
#pragma unroll
  for (int a = 0; a < 3; a++)
    if (flips & (1u << a)) {
#pragma unroll
      for (int i = 0; i < 3; i++) {
        R& h = H[(FEMPIC_DS_VH + 3 * i + a) * A.n + p];
        h = -h;
      }
    }
}

// FP32 (mixed forms): sample at d = r - x0, rule, AB4 velocity; `hist(k)` is
// the particle's value of history plane k.  One level at a time, so that few
// history values are held in registers.  Returns the tet's flag.
template <typename Hist>
__device__ __forceinline__ bool ds_rule32(const DsRule& A, int64_t p, int32_t T, int s, const float d[3],
                                          const float v0[3], float vn[3], float u[3], Hist hist) {
  const float4* C = reinterpret_cast<const float4*>(A.coef32 + kDsCoef32 * (int64_t)T);
  float c[kDsCoef32];
#pragma unroll
  for (int i = 0; i < kDsCoef32 / 4; i++) {
    const float4 v = C[i];
    c[4 * i] = v.x;
    c[4 * i + 1] = v.y;
    c[4 * i + 2] = v.z;
    c[4 * i + 3] = v.w;
  }
  float cur[12];
#pragma unroll
  for (int part = 0; part < 2; part++) {
    const float* q = c + 10 * part;
    float dw[3];
    ds_cross3<float>(d, q + 3, dw);
#pragma unroll
    for (int a = 0; a < 3; a++) {
      cur[3 * part + a] = q[a] + dw[a];
      cur[6 + 3 * part + a] = q[6 + a] + q[9] * d[a];
    }
  }
  float* H = static_cast<float*>(A.h);
  const int64_t n = A.n;
  const bool start = A.start != 0;   // constant extrapolation backwards
  // weights from the kernel parameters: M^r at 0, M^i at 3, L^r at 6, L^i at 15
  const float* w = A.w32;
  float dv[3] = {0.f, 0.f, 0.f}, B[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
  float S[12];
#pragma unroll
  for (int c2 = 0; c2 < 12; c2++) S[c2] = cur[c2];
#pragma unroll
  for (int k = 0; k < 3; k++) {   // the level's sample into the sums, then one plane back
#pragma unroll
    for (int a = 0; a < 3; a++) {
      dv[a] += S[a] * w[k] + S[3 + a] * w[3 + k];
#pragma unroll
      for (int j = 0; j < 3; j++) B[j][a] += S[6 + a] * w[6 + 3 * j + k] + S[9 + a] * w[15 + 3 * j + k];
    }
    if (k == 2) break;
#pragma unroll
    for (int c2 = 0; c2 < 12; c2++) {
      const float older = start ? cur[c2] : hist(FEMPIC_DS_F + 12 * k + c2);
      H[(FEMPIC_DS_F + 12 * k + c2) * n + p] = S[c2];
      S[c2] = older;
    }
  }
  float vh[3][3];
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int a = 0; a < 3; a++) vh[i][a] = start ? v0[a] : hist(FEMPIC_DS_VH + 3 * i + a);
  const float* V[3] = {v0, vh[0], vh[1]};
#pragma unroll
  for (int j = 0; j < 3; j++) {
    float vc[3];
    ds_cross3<float>(V[j], B[j], vc);
#pragma unroll
    for (int a = 0; a < 3; a++) dv[a] += vc[a];
  }
  const float qm = A.qm32[s];
  constexpr float ab[4] = {(float)(55.0 / 24.0), (float)(-59.0 / 24.0), (float)(37.0 / 24.0), (float)(-9.0 / 24.0)};
#pragma unroll
  for (int a = 0; a < 3; a++) {
    u[a] = ab[0] * v0[a] + ab[1] * vh[0][a] + ab[2] * vh[1][a] + ab[3] * vh[2][a];
    vn[a] = v0[a] + qm * dv[a];
    H[(FEMPIC_DS_VH + 6 + a) * n + p] = vh[1][a];
    H[(FEMPIC_DS_VH + 3 + a) * n + p] = vh[0][a];
    H[(FEMPIC_DS_VH + a) * n + p] = v0[a];
  }
  return c[20] != 0.f;
}

// FP64 form: the same as chained multiply-adds (126 FP64-pipe operations, the
// bound of the FP64 step; 181 with separate products and sums).
__device__ __forceinline__ bool ds_rule(const DsRule& A, int64_t p, int32_t T, int s, const double d[3],
                                        const double v0[3], double vn[3], double u[3]) {
  DsHistory<double> h;
  ds_load(A, p, h);
  const double2* C = reinterpret_cast<const double2*>(A.coef + kDsCoef64 * (int64_t)T);
  double cur[12];
#pragma unroll
  for (int part = 0; part < 2; part++) {
    double q[10];
#pragma unroll
    for (int i = 0; i < 5; i++) {
      const double2 v = C[5 * part + i];
      q[2 * i] = v.x;
      q[2 * i + 1] = v.y;
    }
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const int i = (a + 1) % 3, j = (a + 2) % 3;   // (d x W)_a = d_i W_j - d_j W_i
      cur[3 * part + a] = fma(d[i], q[3 + j], fma(-d[j], q[3 + i], q[a]));
      cur[6 + 3 * part + a] = fma(q[9], d[a], q[6 + a]);
    }
  }
  const bool bad = reinterpret_cast<const double*>(C)[20] != 0.0;
  ds_fill(A, v0, cur, h);
  const double* S[3] = {cur, h.f1, h.f2};
  const double* V[3] = {v0, h.vh[0], h.vh[1]};
  const double* w = A.w;
  double dv[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int k = 0; k < 3; k++)
#pragma unroll
    for (int a = 0; a < 3; a++) dv[a] = fma(S[k][a], w[k], fma(S[k][3 + a], w[3 + k], dv[a]));
#pragma unroll
  for (int j = 0; j < 3; j++) {
    double B[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < 3; k++)
#pragma unroll
      for (int a = 0; a < 3; a++) B[a] = fma(S[k][6 + a], w[6 + 3 * j + k], fma(S[k][9 + a], w[15 + 3 * j + k], B[a]));
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const int i = (a + 1) % 3, l = (a + 2) % 3;
      dv[a] = fma(V[j][i], B[l], fma(-V[j][l], B[i], dv[a]));
    }
  }
  const double qm = A.qm[s];
#pragma unroll
  for (int a = 0; a < 3; a++) {
    u[a] = fma(-9.0 / 24.0, h.vh[2][a], fma(37.0 / 24.0, h.vh[1][a], fma(-59.0 / 24.0, h.vh[0][a], (55.0 / 24.0) * v0[a])));
    vn[a] = fma(qm, dv[a], v0[a]);
  }
  ds_store(A, p, v0, cur, h);
  return bad;
}

// The step of the particles under the rule (fempic_env.cu): every argument
// already checked on the host.
int push_downshift(fempic_env* env, const fempic_particles* p, const DsRule& rule, double dt, cudaStream_t st);

}  // namespace fempic
