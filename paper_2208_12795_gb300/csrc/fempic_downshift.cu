// Downshifted particle integrator of Sec. III-D on the FP64 form and the
// FP32-mixed forms: the velocity rule with the carrier integrated
// analytically (M and L weights) and AB4 positions.  Per step: the per-tet
// envelope coefficients (k_ds_field64, k_ds_field32), then the env's step
// kernels with the rule in place of gather and Boris (fempic_ds_rule.cuh):
// sample, velocity rule, AB4 velocity, history shift, tracking, walls and
// deposit of the AB4 segment.
#include <cuda_runtime.h>

#include <cmath>
#include <complex>
#include <string>

#include "fempic_downshift.h"
#include "fempic_bits.cuh"
#include "fempic_ds_rule.cuh"
#include "fempic_internal.h"
#include "fempic_launch.cuh"
#include "fempic_tetgeo.cuh"

namespace {

using fempic::HostMesh;
using fempic::kMaxSpecies;
using fempic::grid_wait;
using fempic::launch;

thread_local std::string g_ds_error;

int fail(int code, const std::string& msg) {
  g_ds_error = msg;
  return code;
}

#define DS_CUDA(call)                                                                       \
  do {                                                                                      \
    cudaError_t e_ = (call);                                                                \
    if (e_ != cudaSuccess) return fail(FEMPIC_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

constexpr int kThreads = 256;

// Local edge e joins sorted local nodes (le0, le1) in the order 01,02,03,12,
// 13,23; local face f is opposite node f and its i-th node is lf(f, i).
__host__ __device__ constexpr int le0(int e) { return e < 3 ? 0 : (e < 5 ? 1 : 2); }
__host__ __device__ constexpr int le1(int e) { return e < 3 ? e + 1 : (e == 3 ? 2 : 3); }
__host__ __device__ constexpr int lf(int f, int i) { return i < f ? i : i + 1; }

// Debug build (FEMPIC_BOUNDS_CHECK): an edge or face id read from this unit's
// tables is checked against its range before it addresses a DoF array; an
// out-of-range id is counted in the env's bounds counter (reported by
// fempic_error_count) and its DoF reads as zero.
#ifdef FEMPIC_BOUNDS_CHECK
constexpr bool kBoundsCheck = true;
#else
constexpr bool kBoundsCheck = false;
#endif
__device__ __forceinline__ bool ds_idx_in(int64_t i, int64_t n, unsigned long long* stats) {
  if (!kBoundsCheck) return true;
  if (i >= 0 && i < n) return true;
  if (stats) atomicAdd(stats + 3, 1ull);
  return false;
}

template <typename R>
__device__ __forceinline__ void cross3(const R a[3], const R b[3], R o[3]) {
  o[0] = a[1] * b[2] - a[2] * b[1];
  o[1] = a[2] * b[0] - a[0] * b[2];
  o[2] = a[0] * b[1] - a[1] * b[0];
}

// Per-tet complex envelope coefficients of one step (Sec. III-A).  Inside a
// tet both Whitney sums are affine in d = r - x0 (x0 = the tet's node 0,
// lambda_k = delta_k0 + g_k . d with g_k = grad lambda_k):
//   W1_ij = const + d x (g_j x g_i), so E~ = E0 + d x W with
//     E0 = sum_j e~_0j g_j,  W = sum_{i<j} e~_ij (g_j x g_i);
//   W2_ijk = const + 2 det[g_i, g_j, g_k] d, so B~ = B0 + beta d with
//     B0 = 2 sum over the faces (0, j, k) of b~_f g_j x g_k,
//     beta = 2 sum_f b~_f det[g_i, g_j, g_k].
// The coefficients of a step are Re (E0, W, B0, beta), then Im (E0, W, B0,
// beta), times a(t).  Both passes are bound by the FP64 pipe, so the
// geometry's products come from tables built once.

// A tet with a DoF that is not finite is flagged: its particles freeze with
// status NONFINITE (as under a field that is not finite), also where a later
// sum would hide it.
__device__ __forceinline__ bool not_finite(double x) {
  return (((unsigned)__double2hiint(x) >> 20) & 0x7ffu) == 0x7ffu;
}
__device__ __forceinline__ bool not_finite(float x) { return ((__float_as_uint(x) >> 23) & 0xffu) == 0xffu; }

// FP64 form: the shared table of fempic_tetgeo.cuh, about 94 operations per
// tet (196k tets: 77 -> 39 us).
__global__ void __launch_bounds__(kThreads) k_ds_field64(int64_t nt, const double* __restrict__ geom,
                                                         const double* __restrict__ tgeo,
                                                         const int32_t* __restrict__ te,
                                                         const int32_t* __restrict__ tf,
                                                         const double2* e, const double2* b, int64_t ne, int64_t nf,
                                                         unsigned long long* stats, double amp,
                                                         double* __restrict__ coef) {
  grid_wait();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nt) return;
  double2 ev[6], bv[4];
#pragma unroll
  for (int k = 0; k < 6; k++) {
    const int32_t id = te[6 * t + k];
    ev[k] = ds_idx_in(id, ne, stats) ? e[id] : make_double2(0.0, 0.0);
  }
#pragma unroll
  for (int f = 0; f < 4; f++) {
    const int32_t id = tf[4 * t + f];
    bv[f] = ds_idx_in(id, nf, stats) ? b[id] : make_double2(0.0, 0.0);
  }
  fempic::TetGeo G;
  fempic::ld_tet_geo(geom, tgeo, t, G);
  const double amp2 = 2.0 * amp;
#pragma unroll
  for (int part = 0; part < 2; part++) {
    double es[6], b2[4], o[10];
#pragma unroll
    for (int k = 0; k < 6; k++) es[k] = amp * (part ? ev[k].y : ev[k].x);
#pragma unroll
    for (int f = 0; f < 4; f++) b2[f] = amp2 * (part ? bv[f].y : bv[f].x);
    fempic::whitney_affine(G, es, b2, o);
    double2* out = reinterpret_cast<double2*>(coef + fempic::kDsCoef64 * t + 10 * part);
#pragma unroll
    for (int c = 0; c < 5; c++) out[c] = make_double2(o[2 * c], o[2 * c + 1]);
  }
  bool bad = false;
#pragma unroll
  for (int k = 0; k < 6; k++) bad = bad || not_finite(ev[k].x) || not_finite(ev[k].y);
#pragma unroll
  for (int f = 0; f < 4; f++) bad = bad || not_finite(bv[f].x) || not_finite(bv[f].y);
  coef[fempic::kDsCoef64 * t + 20] = bad ? 1.0 : 0.0;
}

// Mixed forms: the FP64 sums rounded once to FP32.  A coefficient that rounds
// the other way moves a particle's FP32 velocity by an ulp, so the sums keep
// one order of operations; their geometry factors (g_j x g_i per edge, g_j x
// g_k per face at node 0, det per face) are formed once per mesh, and the
// conversions of DoFs and results run in integer operations off the FP64 pipe
// (663k tets: 280 -> 155 us with a(t) = 1, past the envelope's rise, 182 during
// it, when the 20 sums are scaled).
constexpr int kDsGeo = 32;   // doubles per tet: 6 x 3, 3 x 3, 4, unused

__global__ void __launch_bounds__(kThreads) k_ds_geo32(int64_t nt, const double* __restrict__ geom,
                                                       double* __restrict__ dgeo) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nt) return;
  const double* G = geom + 12 * t;
  double g[4][3];
#pragma unroll
  for (int k = 1; k < 4; k++)
#pragma unroll
    for (int a = 0; a < 3; a++) g[k][a] = G[3 * k + a];
#pragma unroll
  for (int a = 0; a < 3; a++) g[0][a] = -(g[1][a] + g[2][a] + g[3][a]);
  double* o = dgeo + kDsGeo * t;
#pragma unroll
  for (int k = 0; k < 6; k++) {
    double gji[3];
    cross3(g[le1(k)], g[le0(k)], gji);
#pragma unroll
    for (int a = 0; a < 3; a++) o[3 * k + a] = gji[a];
  }
#pragma unroll
  for (int f = 0; f < 4; f++) {
    const int i = lf(f, 0), j = lf(f, 1), k = lf(f, 2);
    double gjk[3];
    cross3(g[j], g[k], gjk);
    o[27 + f] = g[i][0] * gjk[0] + g[i][1] * gjk[1] + g[i][2] * gjk[2];
    if (i == 0) {
#pragma unroll
      for (int a = 0; a < 3; a++) o[18 + 3 * (f - 1) + a] = gjk[a];
    }
  }
  o[31] = 0.0;
}

__global__ void __launch_bounds__(kThreads) k_ds_field32(int64_t nt, const double* __restrict__ geom,
                                                         const double* __restrict__ dgeo,
                                                         const int32_t* __restrict__ te,
                                                         const int32_t* __restrict__ tf,
                                                         const float2* e, const float2* b,
                                                         int64_t ne, int64_t nf, unsigned long long* stats,
                                                         double amp, float* __restrict__ coef32) {
  grid_wait();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nt) return;
  const double2* D = reinterpret_cast<const double2*>(dgeo + kDsGeo * t);
  double w[kDsGeo];
#pragma unroll
  for (int c = 0; c < kDsGeo / 2; c++) {
    const double2 v = __ldg(D + c);
    w[2 * c] = v.x;
    w[2 * c + 1] = v.y;
  }
  const double* g1 = geom + 12 * t + 3;
  bool bad = false;
  double o[20];
#pragma unroll
  for (int c = 0; c < 20; c++) o[c] = 0.0;
#pragma unroll
  for (int k = 0; k < 6; k++) {
    const int32_t id = te[6 * t + k];
    double2 c = make_double2(0.0, 0.0);
    if (ds_idx_in(id, ne, stats)) {
      const float2 cc = e[id];
      bad = bad || not_finite(cc.x) || not_finite(cc.y);
      c = make_double2(fempic::widen32(cc.x), fempic::widen32(cc.y));
    }
#pragma unroll
    for (int a = 0; a < 3; a++) {
      if (le0(k) == 0) {
        const double g = __ldg(g1 + 3 * k + a);   // le1(k) = k + 1: g_{k+1}
        o[a] += c.x * g;
        o[10 + a] += c.y * g;
      }
      o[3 + a] += c.x * w[3 * k + a];
      o[13 + a] += c.y * w[3 * k + a];
    }
  }
#pragma unroll
  for (int f = 0; f < 4; f++) {
    const int32_t id = tf[4 * t + f];
    double2 c = make_double2(0.0, 0.0);
    if (ds_idx_in(id, nf, stats)) {
      const float2 cc = b[id];
      bad = bad || not_finite(cc.x) || not_finite(cc.y);
      c = make_double2(fempic::widen32(cc.x), fempic::widen32(cc.y));
    }
    const double bx = 2.0 * c.x, by = 2.0 * c.y;
    if (f > 0) {
#pragma unroll
      for (int a = 0; a < 3; a++) {
        o[6 + a] += bx * w[18 + 3 * (f - 1) + a];
        o[16 + a] += by * w[18 + 3 * (f - 1) + a];
      }
    }
    o[9] += bx * w[27 + f];
    o[19] += by * w[27 + f];
  }
  if (amp != 1.0) {   // a(t) = 1 (past the envelope's rise) leaves the sums as they are
#pragma unroll
    for (int c = 0; c < 20; c++) o[c] = amp * o[c];
  }
  float4* o32 = reinterpret_cast<float4*>(coef32 + fempic::kDsCoef32 * t);
#pragma unroll
  for (int c = 0; c < 5; c++)
    o32[c] = make_float4(fempic::f64_to_f32(o[4 * c]), fempic::f64_to_f32(o[4 * c + 1]), fempic::f64_to_f32(o[4 * c + 2]), fempic::f64_to_f32(o[4 * c + 3]));
  o32[5] = make_float4(bad ? 1.f : 0.f, 0.f, 0.f, 0.f);
}

// int_0^1 x^m e^{j theta x} dx, m = 0..4: the power series of the exponential
// integrated term by term for |theta| <= 1, else the integration-by-parts
// recurrence J_m = (e^{j theta} - m J_{m-1}) / (j theta).
void moments(double theta, std::complex<double> J[5]) {
  using cd = std::complex<double>;
  if (std::fabs(theta) <= 1.0) {
    for (int m = 0; m < 5; m++) {
      cd term(1.0, 0.0), sum(0.0, 0.0);   // term = (j theta)^l / l!
      for (int l = 0; l < 40; l++) {
        sum += term / double(m + l + 1);
        term *= cd(0.0, theta) / double(l + 1);
      }
      J[m] = sum;
    }
  } else {
    const cd e = std::polar(1.0, theta), jt(0.0, theta);
    J[0] = (e - 1.0) / jt;
    for (int m = 1; m < 5; m++) J[m] = (e - double(m) * J[m - 1]) / jt;
  }
}

void compute_weights(double t, double dt, double omega0, double* w) {
  using cd = std::complex<double>;
  // basis on the nodes x_k = -k (x = (t' - t) / dt) as coefficient vectors
  double c[3][3];
  for (int k = 0; k < 3; k++) {
    double poly[3] = {1.0, 0.0, 0.0};
    for (int j = 0; j < 3; j++) {
      if (j == k) continue;
      const double xk = -double(k), xj = -double(j), den = xk - xj;
      double nxt[3] = {0.0, 0.0, 0.0};   // poly * (x - xj) / den
      for (int m = 0; m < 3; m++) {
        if (m + 1 < 3) nxt[m + 1] += poly[m] / den;
        nxt[m] -= poly[m] * xj / den;
      }
      for (int m = 0; m < 3; m++) poly[m] = nxt[m];
    }
    for (int m = 0; m < 3; m++) c[k][m] = poly[m];
  }
  cd J[5];
  moments(omega0 * dt, J);
  const cd f = dt * std::polar(1.0, omega0 * t);
  for (int k = 0; k < 3; k++) {
    cd I(0.0, 0.0);
    for (int m = 0; m < 3; m++) I += c[k][m] * J[m];
    I *= f;
    w[k] = I.real();
    w[3 + k] = -I.imag();
  }
  for (int j = 0; j < 3; j++)
    for (int k = 0; k < 3; k++) {
      double prod[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
      for (int a = 0; a < 3; a++)
        for (int b = 0; b < 3; b++) prod[a + b] += c[j][a] * c[k][b];
      cd I(0.0, 0.0);
      for (int m = 0; m < 5; m++) I += prod[m] * J[m];
      I *= f;
      w[6 + 3 * j + k] = I.real();
      w[15 + 3 * j + k] = -I.imag();
    }
}

unsigned blocks_for(int64_t n) { return (unsigned)((n + kThreads - 1) / kThreads); }

}  // namespace

struct fempic_downshift {
  int64_t nn = 0, ne = 0, nf = 0, nt = 0;
  double* geom = nullptr;
  double* tgeo = nullptr;       // FP64 form: [nt][kTetGeo] products of the gradients (fempic_tetgeo.cuh)
  int32_t* te = nullptr;
  int32_t* tf = nullptr;
  double* coef = nullptr;       // FP64 form: [nt][kDsCoef64]
  double* dgeo = nullptr;       // mixed forms: [nt][kDsGeo] geometry factors
  float* coef32 = nullptr;      // mixed forms: [nt][kDsCoef32]
};

static void free_ds(fempic_downshift* d) {
  if (!d) return;
  cudaFree(d->geom);
  cudaFree(d->tgeo);
  cudaFree(d->te);
  cudaFree(d->tf);
  cudaFree(d->coef);
  cudaFree(d->dgeo);
  cudaFree(d->coef32);
  delete d;
}

// History planes follow a particle sort: out[k][q] = in[k][perm[q]] for the
// planes that outlive a step (velocities and envelope samples; the two
// scratch vectors are rewritten by every step).
template <typename R>
__global__ void __launch_bounds__(kThreads) k_ds_permute(int64_t n, const int32_t* __restrict__ perm,
                                                          const R* __restrict__ in, R* __restrict__ out) {
  const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (q >= n) return;
  const int64_t src = perm[q];
#pragma unroll 3
  for (int k = 0; k < FEMPIC_DS_VN; k++) out[k * n + q] = __ldg(in + k * n + src);
}

extern "C" const char* fempic_downshift_last_error(void) { return g_ds_error.c_str(); }

extern "C" int fempic_downshift_permute(const fempic_downshift_history* in, const fempic_downshift_history* out,
                                        const int32_t* perm, void* stream) {
  if (!in || !out || !perm) return fail(FEMPIC_EINVAL, "downshift_permute: NULL argument");
  if (in->n != out->n || in->n < 0) return fail(FEMPIC_EINVAL, "downshift_permute: sizes differ");
  if (in->n == 0) return FEMPIC_OK;
  if (!in->planes || !out->planes || in->planes == out->planes)
    return fail(FEMPIC_EINVAL, "downshift_permute: NULL or overlapping planes");
  if (in->f32 != out->f32 || (in->f32 != 0 && in->f32 != 1))
    return fail(FEMPIC_EINVAL, "downshift_permute: plane types differ");
  if (in->n >= (int64_t(1) << 31)) return fail(FEMPIC_EINVAL, "downshift_permute: more than 2^31 particles");
  const unsigned blocks = (unsigned)((in->n + kThreads - 1) / kThreads);
  if (in->f32)
    k_ds_permute<float><<<blocks, kThreads, 0, (cudaStream_t)stream>>>(
        in->n, perm, static_cast<const float*>(in->planes), static_cast<float*>(out->planes));
  else
    k_ds_permute<double><<<blocks, kThreads, 0, (cudaStream_t)stream>>>(
        in->n, perm, static_cast<const double*>(in->planes), static_cast<double*>(out->planes));
  DS_CUDA(cudaGetLastError());
  return FEMPIC_OK;
}

extern "C" void fempic_downshift_destroy(fempic_downshift* ds) { free_ds(ds); }

extern "C" int fempic_downshift_debug_set_table(fempic_downshift* ds, int32_t table, int64_t index,
                                                int32_t value) {
  if (!ds) return fail(FEMPIC_EINVAL, "downshift_debug_set_table: NULL handle");
  if (!kBoundsCheck)
    return fail(FEMPIC_EINVAL, "downshift_debug_set_table: only the debug build (FEMPIC_BOUNDS_CHECK) accepts it");
  int32_t* dst = nullptr;
  if (table == FEMPIC_TABLE_EDGE) {
    if (index < 0 || index >= 6 * ds->nt) return fail(FEMPIC_EINVAL, "downshift_debug_set_table: edge index out of range");
    dst = ds->te + index;
  } else if (table == FEMPIC_TABLE_FACE) {
    if (index < 0 || index >= 4 * ds->nt) return fail(FEMPIC_EINVAL, "downshift_debug_set_table: face index out of range");
    dst = ds->tf + index;
  } else {
    return fail(FEMPIC_EINVAL, "downshift_debug_set_table: unknown table");
  }
  DS_CUDA(cudaMemcpy(dst, &value, sizeof(int32_t), cudaMemcpyHostToDevice));
  return FEMPIC_OK;
}

extern "C" int fempic_downshift_weights(double t, double dt, double omega0, double* w_out) {
  if (!w_out) return fail(FEMPIC_EINVAL, "downshift_weights: NULL output");
  if (!std::isfinite(t) || !std::isfinite(dt) || !std::isfinite(omega0) || !(dt > 0.0))
    return fail(FEMPIC_EINVAL, "downshift_weights: non-finite scalar or dt <= 0");
  compute_weights(t, dt, omega0, w_out);
  return FEMPIC_OK;
}

// A table of the mesh's geometry, filled by `fill` on a stream of its own that
// is waited for: later steps may be on any stream, and a first step that is
// being captured must not defer the table to its replay.
template <typename F>
static cudaError_t fill_table(F fill) {
  cudaStream_t own = nullptr;
  cudaError_t rc = cudaStreamCreateWithFlags(&own, cudaStreamNonBlocking);
  if (rc != cudaSuccess) return rc;
  fill(own);
  rc = cudaGetLastError();
  if (rc == cudaSuccess) rc = cudaStreamSynchronize(own);
  cudaStreamDestroy(own);
  return rc;
}

// A form's coefficients and geometry products, when the handle is made for that
// form (FP64) or on first use: nothing is held for a form that never steps.
// The handle is left unchanged by an error.
template <typename C>
static int make_tables(fempic_downshift* ds, int per_tet, int coef_per_tet, double** geo, C** coef,
                       void (*kernel)(int64_t, const double*, double*)) {
  double* g = nullptr;
  C* c = nullptr;
  if (cudaMalloc(&g, sizeof(double) * per_tet * (size_t)ds->nt) != cudaSuccess ||
      cudaMalloc(&c, sizeof(C) * coef_per_tet * (size_t)ds->nt) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(g);
    return fail(FEMPIC_ENOMEM, "downshift: device allocation");
  }
  const cudaError_t rc =
      fill_table([&](cudaStream_t st) { kernel<<<blocks_for(ds->nt), kThreads, 0, st>>>(ds->nt, ds->geom, g); });
  if (rc != cudaSuccess) {
    cudaFree(g);
    cudaFree(c);
  }
  DS_CUDA(rc);
  *geo = g;
  *coef = c;
  return FEMPIC_OK;
}

static int make_form_tables(fempic_downshift* ds, bool mixed) {
  if (mixed)
    return ds->coef32 ? FEMPIC_OK
                      : make_tables(ds, kDsGeo, fempic::kDsCoef32, &ds->dgeo, &ds->coef32, k_ds_geo32);
  return ds->coef ? FEMPIC_OK
                  : make_tables(ds, fempic::kTetGeo, fempic::kDsCoef64, &ds->tgeo, &ds->coef, fempic::k_tet_geo);
}

static int create_impl(const fempic_mesh_desc* mesh, bool fp64_tables, fempic_downshift** out) {
  *out = nullptr;
  HostMesh m;
  std::string err;
  int rc = fempic::build_host_mesh(*mesh, &m, &err);
  if (rc != FEMPIC_OK) return fail(rc, "downshift_create: " + err);
  fempic_downshift* d = new (std::nothrow) fempic_downshift();
  if (!d) return fail(FEMPIC_ENOMEM, "downshift_create: host allocation");
  d->nn = m.nn;
  d->ne = m.ne;
  d->nf = m.nf;
  d->nt = m.nt;
  const size_t sg = sizeof(double) * 12 * (size_t)m.nt, se = sizeof(int32_t) * 6 * (size_t)m.nt,
               sf = sizeof(int32_t) * 4 * (size_t)m.nt;
  if (cudaMalloc(&d->geom, sg) != cudaSuccess || cudaMalloc(&d->te, se) != cudaSuccess ||
      cudaMalloc(&d->tf, sf) != cudaSuccess) {
    free_ds(d);
    cudaGetLastError();
    return fail(FEMPIC_ENOMEM, "downshift_create: device allocation");
  }
  if (cudaMemcpy(d->geom, m.geom.data(), sg, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(d->te, m.te.data(), se, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(d->tf, m.tf.data(), sf, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaDeviceSynchronize() != cudaSuccess) {
    free_ds(d);
    return fail(FEMPIC_ECUDA, "downshift_create: upload");
  }
  rc = fp64_tables ? make_form_tables(d, false) : FEMPIC_OK;
  if (rc != FEMPIC_OK) {
    free_ds(d);
    return rc;
  }
  *out = d;
  return FEMPIC_OK;
}

extern "C" int fempic_downshift_create(const fempic_mesh_desc* mesh, fempic_downshift** out) {
  if (!mesh || !out) return fail(FEMPIC_EINVAL, "downshift_create: NULL argument");
  return create_impl(mesh, true, out);
}

extern "C" int fempic_downshift_create_form(const fempic_mesh_desc* mesh, int32_t precision,
                                            fempic_downshift** out) {
  if (!mesh || !out) return fail(FEMPIC_EINVAL, "downshift_create: NULL argument");
  if (precision != FEMPIC_FP64 && precision != FEMPIC_MIXED && precision != FEMPIC_MIXED_Q24)
    return fail(FEMPIC_EINVAL, "downshift_create: unknown precision form");
  return create_impl(mesh, precision == FEMPIC_FP64, out);
}

extern "C" int fempic_push_step_downshift(fempic_env* env, fempic_downshift* ds, const fempic_particles* p,
                                          const fempic_downshift_history* hist, const fempic_envelope* envl,
                                          double omega0, double t, double dt, int32_t start, void* stream) {
  if (!env || !ds || !p || !hist || !envl) return fail(FEMPIC_EINVAL, "push_step_downshift: NULL argument");
  if (p->n < 0 || hist->n != p->n) return fail(FEMPIC_EINVAL, "push_step_downshift: history size != particles");
  if (!envl->e_tilde || !envl->b_tilde) return fail(FEMPIC_EINVAL, "push_step_downshift: NULL DoF arrays");
  if (!std::isfinite(t) || !std::isfinite(dt) || !(dt > 0.0) || !std::isfinite(omega0) ||
      !std::isfinite(envl->amp))
    return fail(FEMPIC_EINVAL, "push_step_downshift: non-finite scalar or dt <= 0");
  if (start != 0 && start != 1) return fail(FEMPIC_EINVAL, "push_step_downshift: start must be 0 or 1");
  const bool mixed = fempic::env_precision(env) != FEMPIC_FP64;
  if (hist->f32 != (mixed ? 1 : 0))
    return fail(FEMPIC_EINVAL, "push_step_downshift: history planes must be f64 for an FP64-form env and f32 "
                               "for a mixed-form env (fempic_downshift_history.f32)");
  // the env step it runs checks its arguments only after this step has
  // launched its own kernels: run those checks first, so that an error
  // leaves the particles and the history untouched
  if (fempic::validate_push_step(p, envl, omega0, t, dt) != FEMPIC_OK)
    return fail(FEMPIC_EINVAL, std::string("push_step_downshift: ") + fempic_last_error());
  int64_t counts[4];
  if (fempic_env_query(env, counts, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr) != FEMPIC_OK ||
      counts[3] != ds->nt || counts[1] != ds->ne || counts[2] != ds->nf)
    return fail(FEMPIC_EINVAL, "push_step_downshift: env and downshift tables are of different meshes");
  if (p->n == 0) return FEMPIC_OK;
  if (!hist->planes || !p->x || !p->y || !p->z || !p->vx || !p->vy || !p->vz || !p->tet || !p->status)
    return fail(FEMPIC_EINVAL, "push_step_downshift: NULL particle or history array");
  if (p->n_species < 1 || p->n_species > kMaxSpecies || !p->species_begin || !p->q || !p->m)
    return fail(FEMPIC_EINVAL, "push_step_downshift: species table (1..8 ranges, q, m)");
  if (p->species_begin[0] != 0 || p->species_begin[p->n_species] != p->n)
    return fail(FEMPIC_EINVAL, "push_step_downshift: species ranges must cover [0, n)");
  fempic::DsRule A{};
  for (int s = 0; s < p->n_species; s++) {
    if (p->species_begin[s + 1] < p->species_begin[s])
      return fail(FEMPIC_EINVAL, "push_step_downshift: species ranges decrease");
    if (!(p->m[s] > 0.0) || !std::isfinite(p->q[s])) return fail(FEMPIC_EINVAL, "push_step_downshift: q, m");
    A.qm[s] = p->q[s] / p->m[s];
    A.qm32[s] = (float)A.qm[s];
  }
  A.n = p->n;
  A.h = hist->planes;
  A.start = start;
  compute_weights(t, dt, omega0, A.w);
  for (int i = 0; i < 24; i++) A.w32[i] = (float)A.w[i];
  int rc = make_form_tables(ds, mixed);
  if (rc != FEMPIC_OK) return rc;
  A.coef = ds->coef;
  A.coef32 = ds->coef32;
  cudaStream_t st = (cudaStream_t)stream;
  if (mixed) {   // complex64 DoFs; FP32 velocities, samples and history
    launch(k_ds_field32, blocks_for(ds->nt), kThreads, 0, st, 
        ds->nt, ds->geom, ds->dgeo, ds->te, ds->tf, static_cast<const float2*>(envl->e_tilde),
        static_cast<const float2*>(envl->b_tilde), ds->ne, ds->nf, fempic::env_stats(env), envl->amp, ds->coef32);
  } else {
    launch(k_ds_field64, blocks_for(ds->nt), kThreads, 0, st, 
        ds->nt, ds->geom, ds->tgeo, ds->te, ds->tf, static_cast<const double2*>(envl->e_tilde),
        static_cast<const double2*>(envl->b_tilde), ds->ne, ds->nf, fempic::env_stats(env), envl->amp, ds->coef);
  }
  DS_CUDA(cudaGetLastError());
  rc = fempic::push_downshift(env, p, A, dt, st);
  if (rc != FEMPIC_OK) return fail(rc, std::string("push_step_downshift: ") + fempic_last_error());
  return FEMPIC_OK;
}
