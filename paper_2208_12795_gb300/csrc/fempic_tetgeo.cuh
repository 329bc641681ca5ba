// Per-tet geometry of the FP64 field passes (device code shared by the CUDA
// translation units).  With G_k = grad lambda_k, G_0 = -(G_1 + G_2 + G_3),
// every cross product and determinant of the Whitney sums is a sum of
//   c12 = G_1 x G_2,  c13 = G_1 x G_3,  c23 = G_2 x G_3,  det = G_1 . c23,
// so the affine field of a tet (E = E0 + d x W, B = B0 + beta d, d = r - x0)
// comes from its 6 edge and 4 face values as
//   E0   = e01 G_1 + e02 G_2 + e03 G_3
//   W    = (e02 - e01 - e12) c12 + (e03 - e01 - e13) c13 + (e03 - e02 - e23) c23
//   B0   = 2 (b1 c23 + b2 c13 + b3 c12),  beta = 2 det (b0 - b1 + b2 - b3)
// (the brackets of W are the circulations around the faces at node 0).  The
// FP64 pipe bounds these passes: 37 operations here against about 130 with
// each cross product formed where it is used.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace fempic {

constexpr int kTetGeo = 10;   // doubles per tet: c12 (3), c13 (3), c23 (3), det

struct TetGeo {
  double g[9];    // G_1, G_2, G_3
  double c[10];   // c12, c13, c23, det
};

__device__ __forceinline__ void tet_cross(const double* a, const double* b, double* o) {
  o[0] = a[1] * b[2] - a[2] * b[1];
  o[1] = a[2] * b[0] - a[0] * b[2];
  o[2] = a[0] * b[1] - a[1] * b[0];
}

__device__ __forceinline__ double tet_dot(const double* a, const double* b) {
  return fma(a[2], b[2], fma(a[1], b[1], a[0] * b[0]));
}

// geom [nt][12] (x0, G_1, G_2, G_3) -> tgeo [nt][kTetGeo]; once per mesh.
static __global__ void k_tet_geo(int64_t nt, const double* __restrict__ geom, double* __restrict__ tgeo) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nt) return;
  const double* G = geom + 12 * t + 3;
  double* o = tgeo + kTetGeo * t;
  tet_cross(G, G + 3, o);
  tet_cross(G, G + 6, o + 3);
  tet_cross(G + 3, G + 6, o + 6);
  o[9] = tet_dot(G, o + 6);
}

__device__ __forceinline__ void ld_tet_geo(const double* __restrict__ geom, const double* __restrict__ tgeo, int64_t t,
                                           TetGeo& T) {
  const double2* a = reinterpret_cast<const double2*>(geom + 12 * t);
  const double2* b = reinterpret_cast<const double2*>(tgeo + kTetGeo * t);
  double v[10];
#pragma unroll
  for (int k = 0; k < 5; k++) {
    const double2 p = __ldg(a + 1 + k), q = __ldg(b + k);
    v[2 * k] = p.x;
    v[2 * k + 1] = p.y;
    T.c[2 * k] = q.x;
    T.c[2 * k + 1] = q.y;
  }
#pragma unroll
  for (int k = 0; k < 9; k++) T.g[k] = v[k + 1];
}

// out = (E0, W, B0, beta) from the edge values e and twice the face values b2.
__device__ __forceinline__ void whitney_affine(const TetGeo& T, const double e[6], const double b2[4], double out[10]) {
  const double k12 = (e[1] - e[0]) - e[3], k13 = (e[2] - e[0]) - e[4], k23 = (e[2] - e[1]) - e[5];
#pragma unroll
  for (int a = 0; a < 3; a++) {
    out[a] = fma(e[2], T.g[6 + a], fma(e[1], T.g[3 + a], e[0] * T.g[a]));
    out[3 + a] = fma(k23, T.c[6 + a], fma(k13, T.c[3 + a], k12 * T.c[a]));
    out[6 + a] = fma(b2[3], T.c[a], fma(b2[2], T.c[3 + a], b2[1] * T.c[6 + a]));
  }
  out[9] = T.c[9] * ((b2[0] - b2[1]) + (b2[2] - b2[3]));
}

// Transpose of whitney_affine: adjoint a of (E0, W, B0, beta) -> adjoints of
// the edge values and of the face values themselves (not doubled).
__device__ __forceinline__ void whitney_affine_adjoint(const TetGeo& T, const double a[10], double e[6], double b[4]) {
  const double w12 = tet_dot(a + 3, T.c), w13 = tet_dot(a + 3, T.c + 3), w23 = tet_dot(a + 3, T.c + 6);
  e[0] = tet_dot(a, T.g) - (w12 + w13);
  e[1] = tet_dot(a, T.g + 3) + (w12 - w23);
  e[2] = tet_dot(a, T.g + 6) + (w13 + w23);
  e[3] = -w12;
  e[4] = -w13;
  e[5] = -w23;
  const double d = T.c[9] * a[9];
  b[0] = 2.0 * d;
  b[1] = 2.0 * (tet_dot(a + 6, T.c + 6) - d);
  b[2] = 2.0 * (tet_dot(a + 6, T.c + 3) + d);
  b[3] = 2.0 * (tet_dot(a + 6, T.c) - d);
}

}  // namespace fempic
