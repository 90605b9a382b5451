// Element kernels: recovery (K5), pressure, lattice conversion and diagnostics (the FP64 stage kernel
// is in k_stage64.cu, the mixed form's in k_stage_df.cu). One thread per triangle; the reference
// tables sit in shared memory and are read as warp broadcasts.
#include "device.cuh"
#include "dfloat.cuh"
#include "kcommon.cuh"
#include "ktables.cuh"

namespace dgdf {

// Recovery (eq. (12) eliminated locally): u_T = P_T f_T - G_T^T lam_T, with
// lam_T the multipliers of T's three facets mapped to T's own orientation.
template <int K>
__global__ void __launch_bounds__(128) k_recover(DevMesh m, double* out) {
  using D = Dims<K>;
  constexpr int ND = D::ND, NL = D::NL, L3 = 3 * NL;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= m.n_tri) return;
  double lam[L3];
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const int f = m.tri_facet[size_t(t) * 3 + e];
    const bool flip = m.tri_orient[size_t(t) * 3 + e] < 0;
#pragma unroll
    for (int mm = 0; mm < NL; ++mm) {
      const double v = m.lam[size_t(f) * NL + mm];
      lam[e * NL + mm] = (flip && (mm & 1)) ? -v : v;
    }
  }
  const double* G = m.G + size_t(m.tri_class[t]) * L3 * ND;
#pragma unroll 4
  for (int i = 0; i < ND; ++i) {
    double v = m.h[size_t(t) * ND + i];
#pragma unroll
    for (int l = 0; l < L3; ++l) v -= G[l * ND + i] * lam[l];
    out[size_t(t) * ND + i] = v;
  }
}

// The same with a thread per coefficient, for meshes of fewer than kRecoverSmall triangles (a warp for
// each of the four quarters of this chip's 152 SMs): below that a thread per triangle leaves quarters
// without a warp (FP64 instructions take one 64 cycles), above it the shared multipliers win. 8^2,
// BDM_2: 10.4 us a thread per triangle, 6.0 per coefficient; 64^2, BDM_2: 11.1, 8.3; 128^2, BDM_3:
// 22.9, 28.7.
constexpr int kRecoverSmall = 608 * 32;
template <int K>
__global__ void __launch_bounds__(128) k_recover_coef(DevMesh m, double* out) {
  using D = Dims<K>;
  constexpr int ND = D::ND, NL = D::NL, L3 = 3 * NL;
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= m.n_tri * ND) return;
  const int t = o / ND, i = o - t * ND;
  const double* G = m.G + size_t(__ldg(&m.tri_class[t])) * L3 * ND + i;
  double v = m.h[o], w = 0.0;
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const double* lam = m.lam + size_t(__ldg(&m.tri_facet[size_t(t) * 3 + e])) * NL;
    const bool flip = __ldg(&m.tri_orient[size_t(t) * 3 + e]) < 0;
#pragma unroll
    for (int mm = 0; mm < NL; ++mm) {
      const double g = __ldg(&G[(e * NL + mm) * ND]);
      if (mm & 1) w -= (flip ? -g : g) * lam[mm];
      else v -= g * lam[mm];
    }
  }
  out[o] = v + w;
}

// Element pressure w_T = W_T f_T - (W C^T)_T lam_T; block partial sums of the
// integral of w for the L^2_0 shift go to red[0][block].
template <int K>
__global__ void __launch_bounds__(128) k_pressure(DevMesh m, double* w) {
  using D = Dims<K>;
  constexpr int ND = D::ND, NL = D::NL, L3 = 3 * NL, NW = D::NW;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  double integral = 0.0;
  if (t < m.n_tri) {
    double lam[L3];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      const int f = m.tri_facet[size_t(t) * 3 + e];
      const bool flip = m.tri_orient[size_t(t) * 3 + e] < 0;
#pragma unroll
      for (int mm = 0; mm < NL; ++mm) {
        const double v = m.lam[size_t(f) * NL + mm];
        lam[e * NL + mm] = (flip && (mm & 1)) ? -v : v;
      }
    }
    const int c = m.tri_class[t];
    const double* W = m.W + size_t(c) * NW * ND;
    const double* WC = m.WCt + size_t(c) * NW * L3;
    for (int i = 0; i < NW; ++i) {
      double v = 0.0;
      for (int j = 0; j < ND; ++j) v += W[i * ND + j] * m.h[size_t(t) * ND + j];
      for (int l = 0; l < L3; ++l) v -= WC[i * L3 + l] * lam[l];
      w[size_t(t) * NW + i] = v;
    }
    integral = w[size_t(t) * NW] * m.geo[size_t(c) * kGeo + G_ZINT0];
  }
  integral = block_sum(integral);
  if (threadIdx.x == 0) m.red[blockIdx.x] = integral;
}

// Lattice output of the shifted pressure: c = (integral of w) / |Omega| from the
// block partials, w <- w - c, lam <- lam - c (the constant is mode 0 on facets).
template <int K>
__global__ void __launch_bounds__(128) k_pressure_lattice(DevMesh m, const double* w, double* pe, double* pf,
                                                          int nparts) {
  using D = Dims<K>;
  constexpr int NW = D::NW, NL = D::NL;
  __shared__ double cshift;
  if (threadIdx.x < 32) {
    double v = 0.0;
    for (int i = threadIdx.x; i < nparts; i += 32) v += m.red[i];
    v = warp_sum(v);
    // with outflow facets p = 0 there fixes the constant (eq. (be)): no shift
    if (threadIdx.x == 0) cshift = m.has_kernel ? v / m.area_total : 0.0;
  }
  __syncthreads();
  const double c = cshift;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m.n_tri) {
    const double* geo = m.geo + size_t(m.tri_class[i]) * kGeo;
    double wl[NW];
#pragma unroll
    for (int j = 0; j < NW; ++j) wl[j] = w[size_t(i) * NW + j];
    wl[0] -= c * geo[G_CINV0];
    const double s = geo[G_S];
#pragma unroll
    for (int p = 0; p < NW; ++p) {
      double v = 0.0;
#pragma unroll
      for (int j = 0; j < NW; ++j) v += m.plat_phi[p * NW + j] * wl[j];
      pe[size_t(i) * NW + p] = s * v;
    }
  }
  if (pf && i < m.n_facet) {
    const int fo = m.facet_ext ? m.facet_ext[i] : i;
    double lam[NL];
#pragma unroll
    for (int j = 0; j < NL; ++j) lam[j] = m.lam[size_t(i) * NL + j];
    lam[0] -= c;
#pragma unroll
    for (int p = 0; p < NL; ++p) {
      double v = 0.0;
#pragma unroll
      for (int j = 0; j < NL; ++j) v += m.mu_lat[p * NL + j] * lam[j];
      pf[size_t(fo) * NL + p] = v;
    }
  }
}

// Lattice values -> orthonormal coefficients: coef = sqrt(det) Vhat^-1 vals per component; a thread
// per value, as the recovery.
template <int K>
__global__ void __launch_bounds__(128) k_lattice_to_coef(DevMesh m, const double* __restrict__ vals,
                                                         double* __restrict__ coef) {
  constexpr int NS = Dims<K>::NS, ND = 2 * NS;
  const long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (o >= (long long)m.n_tri * ND) return;
  const int t = int(o / ND), r = int(o - (long long)t * ND), c = r / NS, j = r - c * NS;
  const double* v = vals + size_t(t) * ND + c;
  double x = 0.0;
#pragma unroll
  for (int p = 0; p < NS; ++p) x += __ldg(&m.lat_inv[j * NS + p]) * v[2 * p];
  const double* geo = m.geo + size_t(__ldg(&m.tri_class[t])) * kGeo;
  coef[o] = __ldg(&geo[G_DET]) * __ldg(&geo[G_S]) * x;   // sqrt(det) = det / sqrt(det): no FP64 division
}

template <int K>
__global__ void __launch_bounds__(128) k_coef_to_lattice(DevMesh m, const double* __restrict__ coef,
                                                         double* __restrict__ vals) {
  constexpr int NS = Dims<K>::NS, ND = 2 * NS;
  const long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (o >= (long long)m.n_tri * ND) return;
  const int t = int(o / ND), r = int(o - (long long)t * ND), p = r >> 1, c = r & 1;
  const double* u = coef + size_t(t) * ND + c * NS;
  double x = 0.0;
#pragma unroll
  for (int j = 0; j < NS; ++j) x += __ldg(&m.lat_phi[p * NS + j]) * u[j];
  vals[o] = __ldg(&m.geo[size_t(__ldg(&m.tri_class[t])) * kGeo + G_S]) * x;
}

// The same conversions for the mixed form, in double-float arithmetic on the FP32 pipes (the
// FP64 pipe, 1/64 of the FP32 rate here, only splits the inputs and rounds the outputs). The
// tables are split into double-float pairs once per block; a block's 128 triangles pass through
// shared memory, so that global reads and writes are coalesced.
constexpr int kConvTris = 128;

template <int K>
__global__ void __launch_bounds__(kConvTris) k_lattice_to_coef_df(DevMesh m, const double* vals, double* coef) {
  using D = Dims<K>;
  constexpr int NS = D::NS, NV = 2 * NS, RS = NV + 1;
  __shared__ float2 tab[NS * NS];
  __shared__ double tile[kConvTris * RS];
  for (int i = threadIdx.x; i < NS * NS; i += kConvTris) tab[i] = to_float2(dfl(m.lat_inv[i]));
  const int t0 = blockIdx.x * kConvTris;
  const int nt = min(kConvTris, m.n_tri - t0);
  const double* vb = vals + size_t(t0) * NV;
  for (int e = threadIdx.x; e < nt * NV; e += kConvTris) tile[(e / NV) * RS + e % NV] = vb[e];
  __syncthreads();
  if (int(threadIdx.x) < nt) {
    const int t = t0 + threadIdx.x;
    const dfl sq(1.0 / m.geo[size_t(m.tri_class[t]) * kGeo + G_S]);
    double* row = tile + threadIdx.x * RS;
    dfl v[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = dfl(row[i]);   // [p][c]
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      dacc c0 = dacc_zero(), c1 = dacc_zero();
#pragma unroll
      for (int p = 0; p < NS; ++p) {
        const dfl a = to_dfl(tab[j * NS + p]);
        mad(c0, a, v[2 * p]);
        mad(c1, a, v[2 * p + 1]);
      }
      row[j] = to_double(sq * val(c0));
      row[NS + j] = to_double(sq * val(c1));
    }
  }
  __syncthreads();
  double* cb = coef + size_t(t0) * NV;
  for (int e = threadIdx.x; e < nt * NV; e += kConvTris) cb[e] = tile[(e / NV) * RS + e % NV];
}

template <int K>
__global__ void __launch_bounds__(kConvTris) k_coef_to_lattice_df(DevMesh m, const double* coef, double* vals) {
  using D = Dims<K>;
  constexpr int NS = D::NS, NV = 2 * NS, RS = NV + 1;
  __shared__ float2 tab[NS * NS];
  __shared__ double tile[kConvTris * RS];
  for (int i = threadIdx.x; i < NS * NS; i += kConvTris) tab[i] = to_float2(dfl(m.lat_phi[i]));
  const int t0 = blockIdx.x * kConvTris;
  const int nt = min(kConvTris, m.n_tri - t0);
  const double* cb = coef + size_t(t0) * NV;
  for (int e = threadIdx.x; e < nt * NV; e += kConvTris) tile[(e / NV) * RS + e % NV] = cb[e];
  __syncthreads();
  if (int(threadIdx.x) < nt) {
    const int t = t0 + threadIdx.x;
    const dfl sc(m.geo[size_t(m.tri_class[t]) * kGeo + G_S]);
    double* row = tile + threadIdx.x * RS;
    dfl c[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) c[i] = dfl(row[i]);   // [c][j]
#pragma unroll
    for (int p = 0; p < NS; ++p) {
      dacc v0 = dacc_zero(), v1 = dacc_zero();
#pragma unroll
      for (int j = 0; j < NS; ++j) {
        const dfl a = to_dfl(tab[p * NS + j]);
        mad(v0, a, c[j]);
        mad(v1, a, c[NS + j]);
      }
      row[2 * p] = to_double(sc * val(v0));
      row[2 * p + 1] = to_double(sc * val(v1));
    }
  }
  __syncthreads();
  double* vb = vals + size_t(t0) * NV;
  for (int e = threadIdx.x; e < nt * NV; e += kConvTris) vb[e] = tile[(e / NV) * RS + e % NV];
}

// Diagnostics partials per block: red[0] energy, red[1] enstrophy, red[2] max |div|,
// red[3] max |[u.n]| (each facet is seen from both sides).
template <int K>
__global__ void __launch_bounds__(128) k_diagnostics(DevMesh m, const double* coef) {
  using D = Dims<K>;
  constexpr int NS = D::NS, ND = D::ND;
  __shared__ SmemTables<K, double> T;
  load_tables<K, double>(m, T);
  __syncthreads();
  double en = 0.0, ens = 0.0, dmax = 0.0, jmax = 0.0;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < m.n_tri; t += gridDim.x * blockDim.x) {
    double c[ND];
    load_coef<ND>(coef + size_t(t) * ND, c);
#pragma unroll
    for (int i = 0; i < ND; ++i) en += c[i] * c[i];
    const double* geo = m.geo + size_t(m.tri_class[t]) * kGeo;
    const double Ji[4] = {geo[0], geo[1], geo[2], geo[3]};
    const double det = geo[G_DET], s = geo[G_S];
    for (int q = 0; q < D::NQ; ++q) {
      double a00 = 0, a01 = 0, a10 = 0, a11 = 0;
#pragma unroll
      for (int j = 0; j < NS; ++j) {
        a00 += T.vdphi[q][j][0] * c[j];
        a01 += T.vdphi[q][j][1] * c[j];
        a10 += T.vdphi[q][j][0] * c[NS + j];
        a11 += T.vdphi[q][j][1] * c[NS + j];
      }
      const double g00 = s * (a00 * Ji[0] + a01 * Ji[2]), g01 = s * (a00 * Ji[1] + a01 * Ji[3]);
      const double g10 = s * (a10 * Ji[0] + a11 * Ji[2]), g11 = s * (a10 * Ji[1] + a11 * Ji[3]);
      const double om = g10 - g01;
      ens += T.vw[q] * det * om * om;
      dmax = fmax(dmax, fabs(g00 + g11));
    }
    for (int e = 0; e < 3; ++e) {
      // on a wall the jump is u.n itself: the missing side counts as zero; on an inflow facet
      // it is (u - u_in).n; on an outflow facet u.n is free (Sec. 2.5)
      const int tnr = m.tri_nbr[size_t(t) * 3 + e];
      const int fid = m.tri_facet[size_t(t) * 3 + e];
      const int kd = (tnr < 0 && m.facet_kind) ? int(m.facet_kind[fid]) : int(kFacetWall);
      if (kd == kFacetOutflow) continue;
      const bool canon = m.tri_orient[size_t(t) * 3 + e] > 0;
      const int tn = tnr < 0 ? t : tnr;
      const int el = tnr < 0 ? e : m.tri_nbr_loc[size_t(t) * 3 + e];
      const double sn = tnr < 0 ? 0.0 : m.geo[size_t(m.tri_class[tn]) * kGeo + G_S];
      const double n0 = geo[G_NRM + 2 * e], n1 = geo[G_NRM + 2 * e + 1];
      double cn[ND];
      load_coef<ND>(coef + size_t(tn) * ND, cn);
      for (int q = 0; q < D::NQF; ++q) {
        const int qn = D::NQF - 1 - q;
        double a0 = 0, a1 = 0, b0 = 0, b1 = 0;
#pragma unroll
        for (int j = 0; j < NS; ++j) {
          a0 += T.fphi[e][q][j] * c[j];
          a1 += T.fphi[e][q][j] * c[NS + j];
          b0 += T.fphi[el][qn][j] * cn[j];
          b1 += T.fphi[el][qn][j] * cn[NS + j];
        }
        double x0 = sn * b0, x1 = sn * b1;
        if (kd == kFacetInflow) {
          const double* uq = m.inflow_q + (size_t(fid) * D::NQF + (canon ? q : qn)) * 2;
          x0 = uq[0];
          x1 = uq[1];
        }
        jmax = fmax(jmax, fabs((s * a0 - x0) * n0 + (s * a1 - x1) * n1));
      }
    }
  }
  en = block_sum(en);
  ens = block_sum(ens);
  dmax = block_max(dmax);
  jmax = block_max(jmax);
  if (threadIdx.x == 0) {
    m.red[0 * kMaxSolverBlocks + blockIdx.x] = en;
    m.red[1 * kMaxSolverBlocks + blockIdx.x] = ens;
    m.red[2 * kMaxSolverBlocks + blockIdx.x] = dmax;
    m.red[3 * kMaxSolverBlocks + blockIdx.x] = jmax;
  }
}

__global__ void k_diag_finish(DevMesh m, int nparts) {
  if (threadIdx.x >= 32) return;
  double a = 0, b = 0, c = 0, d = 0;
  for (int i = threadIdx.x; i < nparts; i += 32) {
    a += m.red[0 * kMaxSolverBlocks + i];
    b += m.red[1 * kMaxSolverBlocks + i];
    c = fmax(c, m.red[2 * kMaxSolverBlocks + i]);
    d = fmax(d, m.red[3 * kMaxSolverBlocks + i]);
  }
  a = warp_sum(a);
  b = warp_sum(b);
  c = warp_max(c);
  d = warp_max(d);
  if (threadIdx.x == 0) {
    m.diag[0] = a;
    m.diag[1] = b;
    m.diag[2] = c;
    m.diag[3] = d;
  }
}

__global__ void k_check_finite(const double* v, long long n, int* flag) {
  bool bad = false;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    bad |= !isfinite(v[i]);
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, kFlagNonFinite);
}

__global__ void __launch_bounds__(256) k_energy_part(const double* u, long long n, double* part) {
  double a = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double v = __ldcg(&u[i]);
    a = fma(v, v, a);
  }
  a = block_sum(a);
  if (threadIdx.x == 0) part[blockIdx.x] = a;
}

__global__ void k_energy_watch(double* watch, int nparts, double tol, DevStats* st) {
  if (threadIdx.x >= 32) return;
  double e = 0.0;
  for (int i = threadIdx.x; i < nparts; i += 32) e += watch[2 + i];
  e = warp_sum(e);
  if (threadIdx.x == 0) {
    const double prev = watch[0];
    if (prev >= 0.0) {
      watch[1] = prev > 0.0 ? e / prev : (e > 0.0 ? INFINITY : 1.0);
      if (!(e <= prev * (1.0 + tol))) atomicOr(&st->flags, kFlagEnergyGrowth);
    }
    watch[0] = e;
  }
}

// ------------------------------------------------------------------- launchers
namespace {
inline int blocks_for(long long n, int bs) { return int((n + bs - 1) / bs); }
}

#define DGDF_DISPATCH_K(kv, CALL) \
  switch (kv) {                   \
    case 1: { constexpr int K = 1; CALL; break; } \
    case 2: { constexpr int K = 2; CALL; break; } \
    case 3: { constexpr int K = 3; CALL; break; } \
    default: return cudaErrorInvalidValue;        \
  }

// Lattice conversions: FP64 arithmetic in the FP64 form, double-float in the mixed form.
cudaError_t launch_lattice_to_coef(const DevMesh& m, const double* vals, double* coef, cudaStream_t s) {
  if (m.elem_df)
    DGDF_DISPATCH_K(m.k, (k_lattice_to_coef_df<K><<<blocks_for(m.n_tri, kConvTris), kConvTris, 0, s>>>(m, vals, coef)))
  else
    DGDF_DISPATCH_K(m.k, (k_lattice_to_coef<K><<<blocks_for((long long)m.n_tri * m.nd, 128), 128, 0, s>>>(m, vals, coef)))
  return cudaGetLastError();
}

cudaError_t launch_coef_to_lattice(const DevMesh& m, const double* coef, double* vals, cudaStream_t s) {
  if (m.elem_df)
    DGDF_DISPATCH_K(m.k, (k_coef_to_lattice_df<K><<<blocks_for(m.n_tri, kConvTris), kConvTris, 0, s>>>(m, coef, vals)))
  else
    DGDF_DISPATCH_K(m.k, (k_coef_to_lattice<K><<<blocks_for((long long)m.n_tri * m.nd, 128), 128, 0, s>>>(m, coef, vals)))
  return cudaGetLastError();
}

cudaError_t launch_recover(const DevMesh& m, double* out, float2* out_df, cudaStream_t s) {
  if (m.elem_df) return launch_recover_df(m, out, out_df, s);
  if (m.n_tri < kRecoverSmall) {
    DGDF_DISPATCH_K(m.k, (k_recover_coef<K><<<blocks_for((long long)m.n_tri * m.nd, 128), 128, 0, s>>>(m, out)));
  } else {
    DGDF_DISPATCH_K(m.k, (k_recover<K><<<blocks_for(m.n_tri, 128), 128, 0, s>>>(m, out)));
  }
  return cudaGetLastError();
}

cudaError_t launch_pressure(const DevMesh& m, double* w, cudaStream_t s) {
  DGDF_DISPATCH_K(m.k, (k_pressure<K><<<blocks_for(m.n_tri, 128), 128, 0, s>>>(m, w)));
  return cudaGetLastError();
}

cudaError_t launch_pressure_lattice(const DevMesh& m, const double* w, double* pe, double* pf, cudaStream_t s) {
  const int nparts = blocks_for(m.n_tri, 128);
  const long long n = m.n_tri > m.n_facet ? m.n_tri : m.n_facet;
  DGDF_DISPATCH_K(m.k, (k_pressure_lattice<K><<<blocks_for(n, 128), 128, 0, s>>>(m, w, pe, pf, nparts)));
  return cudaGetLastError();
}

cudaError_t launch_diagnostics(const DevMesh& m, const double* coef, cudaStream_t s) {
  int nb = blocks_for(m.n_tri, 128);
  if (nb > kMaxSolverBlocks) nb = kMaxSolverBlocks;
  DGDF_DISPATCH_K(m.k, (k_diagnostics<K><<<nb, 128, 0, s>>>(m, coef)));
  k_diag_finish<<<1, 32, 0, s>>>(m, nb);
  return cudaGetLastError();
}

cudaError_t launch_energy_watch(const double* u, long long n, double* watch, double tol, DevStats* st,
                                cudaStream_t s) {
  long long nb = (n + 255) / 256;
  if (nb > 1024) nb = 1024;
  if (nb < 1) nb = 1;
  k_energy_part<<<int(nb), 256, 0, s>>>(u, n, watch + 2);
  k_energy_watch<<<1, 32, 0, s>>>(watch, int(nb), tol, st);
  return cudaGetLastError();
}

cudaError_t launch_check_finite(const double* v, long long n, int* flag, cudaStream_t s) {
  long long nb = (n + 255) / 256;
  if (nb > 1024) nb = 1024;
  if (nb < 1) nb = 1;
  k_check_finite<<<int(nb), 256, 0, s>>>(v, n, flag);
  return cudaGetLastError();
}

}  // namespace dgdf
