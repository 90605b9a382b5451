// FP64 element kernels of the residual: the stage functional with its condensation (K1-K3) and the
// transposed residual Jacobian of the adjoint.
//
// Bound: the FP64 pipes. A quarter of an SM takes 64 cycles for an FP64 instruction of a warp,
// whatever number of its lanes is live, so the time is the instructions of the busiest quarter: a
// thread a triangle left 8192 triangles (64^2) on 256 of the chip's 608 quarters, each with one
// serial chain. Here a block takes a tile of E triangles through shared memory, and each phase
// deals out its tasks to all threads:
//   1  a quadrature point of a triangle (volume, or facet with both traces): traces, gradients, flux
//   2  a test function of a component: its sum over all points, then the stage combination
//   3  a row of the class operators P and G
// Operands come from shared memory, which the slow pipes leave idle. E is a power of two, at most
// 16 and small enough to give every SM two tiles. Time per launch, a thread a triangle -> tasks:
// 8^2 BDM_2 107 -> 18 us, 48^2 perturbed BDM_2 113 -> 39, 64^2 BDM_2 107 -> 44, 128^2 BDM_3 438 -> 282
// (320 of that before the own viscous terms became a matrix); the adjoint's at 64^2 BDM_2 130 -> 52.
#include <algorithm>

#include "device.cuh"
#include "kcommon.cuh"
#include "ktables.cuh"

namespace dgdf {
namespace {

constexpr int kTileThreads = 128;

// How a kernel takes the viscous terms: none (nu = 0), with the normal derivatives of the basis at
// the facet points from a per-class table (m.dn64, at most kDnClasses classes), or from reference
// gradients. The stage kernel with tables takes the terms of a triangle's own gradient (volume, own
// consistency) as one matrix per class (m.vown64): its volume points then need no gradients, its facet
// points no own normal derivative. The symmetry term stays at the facet points, where both traces,
// nearly equal in a smooth field, meet before a derivative multiplies them.
enum Visc { VISC_NONE, VISC_TABLE, VISC_GENERAL };

template <int K>
struct Tile {
  using D = Dims<K>;
  static constexpr int NQ = D::NQ, ND = D::ND, NF = 3 * D::NQF;
  static constexpr int PTS = NQ + NF;             // points of a triangle
  static constexpr int LU = ND + 1, LN = 3 * ND + 1, LF = ND + 1;   // odd row lengths: no bank conflicts
};

// Trace of the neighbour's and own basis at facet point q of facet e: value and derivative along the
// own outward normal, both components. u: coefficient rows (own at U, the neighbour's at N).
template <int K, int V>
struct FacetGeo {
  int e, en, cls, ncls;
  double s, sn, n0, n1, len, sig, mo0, mo1, mn0, mn1;
};

template <int K, int V>
__device__ __forceinline__ void facet_geo(const DevMesh& m, int t, int e, int tn, FacetGeo<K, V>& g) {
  g.e = e;
  g.cls = __ldg(&m.tri_class[t]);
  const double* geo = m.geo + size_t(g.cls) * kGeo;
  g.s = __ldg(&geo[G_S]);
  g.n0 = __ldg(&geo[G_NRM + 2 * e]);
  g.n1 = __ldg(&geo[G_NRM + 2 * e + 1]);
  g.len = __ldg(&geo[G_FLEN + e]);
  if (tn < 0) return;
  g.en = __ldg(&m.tri_nbr_loc[size_t(t) * 3 + e]);
  g.ncls = __ldg(&m.tri_class[tn]);
  const double* geon = m.geo + size_t(g.ncls) * kGeo;
  g.sn = __ldg(&geon[G_S]);
  if constexpr (V != VISC_NONE) g.sig = __ldg(&m.facet_sigma[__ldg(&m.tri_facet[size_t(t) * 3 + e])]);
  if constexpr (V == VISC_GENERAL) {
    // normal derivative in reference gradients: d_n psi = s sum_r d_r psihat (Jinv n)_r
    g.mo0 = __ldg(&geo[G_JINV]) * g.n0 + __ldg(&geo[G_JINV + 1]) * g.n1;
    g.mo1 = __ldg(&geo[G_JINV + 2]) * g.n0 + __ldg(&geo[G_JINV + 3]) * g.n1;
    g.mn0 = __ldg(&geon[G_JINV]) * g.n0 + __ldg(&geon[G_JINV + 1]) * g.n1;
    g.mn1 = __ldg(&geon[G_JINV + 2]) * g.n0 + __ldg(&geon[G_JINV + 3]) * g.n1;
  }
}

// v[c] = values, d[c] = derivatives along n of the field with coefficients U (component-major) at
// point q of facet e of a triangle of class cls (scale s; n = sgn times its outward normal)
template <int K, int V, bool DERIV>
__device__ __forceinline__ void facet_trace(const SmemTables<K, double>& T, const double* dn, const double* U, int e,
                                            int q, int cls, double s, double sgn, double m0, double m1, double (&v)[2],
                                            double (&d)[2]) {
  using D = Dims<K>;
  constexpr int NS = D::NS;
  const double *ph = T.fphi[e][q], *tab = dn + ((cls * 3 + e) * D::NQF + q) * NS;
  double a0 = 0, a1 = 0, b0 = 0, b1 = 0, c0 = 0, c1 = 0;
#pragma unroll
  for (int j = 0; j < NS; ++j) {
    a0 += ph[j] * U[j];
    a1 += ph[j] * U[NS + j];
    if constexpr (DERIV && V == VISC_TABLE) {
      b0 += tab[j] * U[j];
      b1 += tab[j] * U[NS + j];
    } else if constexpr (DERIV && V == VISC_GENERAL) {
      const double g0 = T.fdphi[e][q][j][0], g1 = T.fdphi[e][q][j][1];
      b0 += g0 * U[j];
      b1 += g0 * U[NS + j];
      c0 += g1 * U[j];
      c1 += g1 * U[NS + j];
    }
  }
  v[0] = s * a0;
  v[1] = s * a1;
  if constexpr (DERIV && V == VISC_TABLE) {
    d[0] = sgn * s * b0;
    d[1] = sgn * s * b1;
  } else if constexpr (DERIV && V == VISC_GENERAL) {
    d[0] = s * (m0 * b0 + m1 * c0);
    d[1] = s * (m0 * b1 + m1 * c1);
  }
}

// Fills the own rows X[el][ND] of the tile's triangles and, with X3, the neighbours' [el][3][ND]
// (left as they are where there is no neighbour).
template <int K>
__device__ __forceinline__ void load_tile(const DevMesh& m, const double* __restrict__ src, int t0, int E, double* X,
                                          double* X3) {
  using L = Tile<K>;
  for (int i = threadIdx.x; i < E * L::ND; i += blockDim.x) {
    const int el = i / L::ND, j = i - el * L::ND, t = min(t0 + el, m.n_tri - 1);
    X[el * L::LU + j] = src[size_t(t) * L::ND + j];
  }
  if (!X3) return;
  for (int i = threadIdx.x; i < E * 3 * L::ND; i += blockDim.x) {
    const int el = i / (3 * L::ND), r = i - el * 3 * L::ND, e = r / L::ND, j = r - e * L::ND;
    const int t = min(t0 + el, m.n_tri - 1), tn = __ldg(&m.tri_nbr[size_t(t) * 3 + e]);
    if (tn >= 0) X3[el * L::LN + r] = src[size_t(tn) * L::ND + j];
  }
}

// The terms of L(u)(phi) at the tile's points (eq. (7), eq. (18)): -C_h(u;u,phi) - B_h(u,phi).
// Volume point q: H[c][r], the flux (u x u - nu grad u) in reference directions, times the weight;
// facet point: A[c] against phi_c and B[c] (VISC_GENERAL: B mo0, B mo1) against its normal
// derivative, with u.n the average of both traces and the upwind value, the SIPG consistency,
// symmetry and penalty terms (the neighbour's point q is our point NQF-1-q). A wall adds nothing;
// inflow and outflow facets add the convective flux against the exterior state (Sec. 2.5), which is
// u_in on an inflow facet (stored in the canonical direction) and the own trace on an outflow facet.
template <int K, int V>
struct StageTile : Tile<K> {
  using L = Tile<K>;
  static constexpr int NH = 4, NA = V == VISC_NONE ? 2 : (V == VISC_TABLE ? 4 : 6);
  static constexpr int LH = L::NQ * NH + 1, LA = (L::NF * NA) | 1;
  static constexpr int words = L::LU + L::LN + LH + LA + L::LF;   // doubles a triangle
};

template <int K, int V>
__global__ void __launch_bounds__(kTileThreads) k_stage64(DevMesh m, StageArgs a, int log_e) {
  using D = Dims<K>;
  using L = StageTile<K, V>;
  constexpr int NS = D::NS, ND = D::ND, NQ = D::NQ, NQF = D::NQF, NF = 3 * NQF, L3 = 3 * D::NL;
  __shared__ SmemTables<K, double> T;
  __shared__ int info[16];   // 8 x class + a bit per boundary facet
  extern __shared__ double tile_smem[];
  const int E = 1 << log_e;
  double* U = tile_smem;
  double* N = U + E * L::LU;
  double* H = N + E * L::LN;
  double* A = H + E * L::LH;
  double* F = A + E * L::LA;
  double* dn = F + E * L::LF;
  load_tables<K, double>(m, T);
  if constexpr (V == VISC_TABLE) {
    for (int i = threadIdx.x; i < m.n_class * NF * NS; i += blockDim.x) dn[i] = __ldg(&m.dn64[i]);
    for (int i = threadIdx.x; i < m.n_class * NS * NS; i += blockDim.x) dn[m.n_class * NF * NS + i] = __ldg(&m.vown64[i]);
  }
  const double nu = m.nu;
  const int ntiles = (m.n_tri + E - 1) >> log_e;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int t0 = tile << log_e;
    __syncthreads();
    const bool res = a.mode != MODE_PROJECT;
    load_tile<K>(m, a.up, t0, E, U, res ? N : nullptr);
    if (int(threadIdx.x) < E) {
      const int t = min(t0 + int(threadIdx.x), m.n_tri - 1);
      int v = __ldg(&m.tri_class[t]) * 8;
#pragma unroll
      for (int e = 0; e < 3; ++e) v |= __ldg(&m.tri_nbr[size_t(t) * 3 + e]) < 0 ? 1 << e : 0;
      info[threadIdx.x] = v;
    }
    __syncthreads();
    if (res) {
      // 1: points
      for (int i = threadIdx.x; i < (L::PTS << log_e); i += blockDim.x) {
        const int el = i & (E - 1), pt = i >> log_e, t = min(t0 + el, m.n_tri - 1);
        const double* u = U + el * L::LU;
        if (pt < NQ) {
          const double* geo = m.geo + size_t(__ldg(&m.tri_class[t])) * kGeo;
          const double J0 = __ldg(&geo[G_JINV]), J1 = __ldg(&geo[G_JINV + 1]), J2 = __ldg(&geo[G_JINV + 2]),
                       J3 = __ldg(&geo[G_JINV + 3]), s = __ldg(&geo[G_S]);
          double u0 = 0, u1 = 0, a00 = 0, a01 = 0, a10 = 0, a11 = 0;
#pragma unroll
          for (int j = 0; j < NS; ++j) {
            const double ph = T.vphi[pt][j], x = u[j], y = u[NS + j];
            u0 += ph * x;
            u1 += ph * y;
            if constexpr (V == VISC_GENERAL) {
              const double d0 = T.vdphi[pt][j][0], d1 = T.vdphi[pt][j][1];
              a00 += d0 * x;
              a01 += d1 * x;
              a10 += d0 * y;
              a11 += d1 * y;
            }
          }
          u0 *= s;
          u1 *= s;
          double F00 = u0 * u0, F01 = u0 * u1, F11 = u1 * u1, F10 = F01;
          if constexpr (V == VISC_GENERAL) {
            // physical gradient du_c/dx_d = s sum_r a_cr Jinv[r][d]
            const double ns = nu * s;
            F00 -= ns * (a00 * J0 + a01 * J2);
            F01 -= ns * (a00 * J1 + a01 * J3);
            F10 -= ns * (a10 * J0 + a11 * J2);
            F11 -= ns * (a10 * J1 + a11 * J3);
          }
          const double w = T.vw[pt] * __ldg(&geo[G_DET]) * s;
          double* h = H + el * L::LH + pt * L::NH;
          h[0] = w * (F00 * J0 + F01 * J1);
          h[1] = w * (F00 * J2 + F01 * J3);
          h[2] = w * (F10 * J0 + F11 * J1);
          h[3] = w * (F10 * J2 + F11 * J3);
        } else {
          const int e = (pt - NQ) / NQF, q = pt - NQ - e * NQF;
          const int tn = __ldg(&m.tri_nbr[size_t(t) * 3 + e]);
          double* out = A + el * L::LA + (pt - NQ) * L::NA;
          int kd = kFacetWall;
          if (tn < 0 && m.facet_kind) kd = __ldg(&m.facet_kind[__ldg(&m.tri_facet[size_t(t) * 3 + e])]);
          if (tn < 0 && kd == kFacetWall) {
#pragma unroll
            for (int x = 0; x < L::NA; ++x) out[x] = 0.0;
            continue;
          }
          FacetGeo<K, V> g;
          facet_geo<K, V>(m, t, e, tn, g);
          double ui[2], di[2], uo[2], dd[2];
          if (tn >= 0) {
            facet_trace<K, V, V == VISC_GENERAL>(T, dn, u, e, q, g.cls, g.s, 1.0, g.mo0, g.mo1, ui, di);
            facet_trace<K, V, true>(T, dn, N + el * L::LN + e * ND, g.en, NQF - 1 - q, g.ncls, g.sn, -1.0, g.mn0, g.mn1,
                                    uo, dd);
          } else {
            facet_trace<K, V, false>(T, dn, u, e, q, g.cls, g.s, 1.0, 0.0, 0.0, ui, di);
            uo[0] = ui[0];
            uo[1] = ui[1];
            if (kd == kFacetInflow) {
              const int f = __ldg(&m.tri_facet[size_t(t) * 3 + e]);
              const bool canon = __ldg(&m.tri_orient[size_t(t) * 3 + e]) > 0;
              const double* uq = m.inflow_q + (size_t(f) * NQF + (canon ? q : NQF - 1 - q)) * 2;
              uo[0] = __ldg(&uq[0]);
              uo[1] = __ldg(&uq[1]);
            }
          }
          const double vn = 0.5 * ((ui[0] + uo[0]) * g.n0 + (ui[1] + uo[1]) * g.n1);
          const double w = T.fw[q] * g.len * g.s, wv = w * vn;
          const bool own = vn >= 0.0;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            double x = -wv * (own ? ui[c] : uo[c]);
            if constexpr (V == VISC_NONE) {
              out[c] = x;
            } else {
              double B = 0.0;
              if (tn >= 0) {
                const double jc = ui[c] - uo[c], wn = w * nu;
                if constexpr (V == VISC_TABLE) {
                  x += wn * (0.5 * dd[c] - g.sig * jc);
                  B = 0.5 * wn * jc;
                } else {
                  x += wn * (0.5 * (di[c] + dd[c]) - g.sig * jc);
                  B = 0.5 * wn * jc;
                }
              }
              out[c] = x;
              if constexpr (V == VISC_TABLE) {
                out[2 + c] = B;
              } else {
                out[2 + 2 * c] = tn >= 0 ? B * g.mo0 : 0.0;
                out[3 + 2 * c] = tn >= 0 ? B * g.mo1 : 0.0;
              }
            }
          }
        }
      }
      __syncthreads();
    }
    // 2: test functions
    for (int i = threadIdx.x; i < (ND << log_e); i += blockDim.x) {
      const int el = i & (E - 1), r = i >> log_e, c = r / NS, j = r - c * NS, t = min(t0 + el, m.n_tri - 1);
      double f = U[el * L::LU + r];
      if (res) {
        const double *h = H + el * L::LH + 2 * c, *A_ = A + el * L::LA;
        double x = 0.0, y = 0.0;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          x += h[q * L::NH] * T.vdphi[q][j][0];
          y += h[q * L::NH + 1] * T.vdphi[q][j][1];
        }
#pragma unroll
        for (int p = 0; p < NF; ++p) {
          x += A_[p * L::NA + c] * T.fphi[p / NQF][p % NQF][j];
          if constexpr (V == VISC_GENERAL) {
            y += A_[p * L::NA + 2 + 2 * c] * T.fdphi[p / NQF][p % NQF][j][0];
            y += A_[p * L::NA + 3 + 2 * c] * T.fdphi[p / NQF][p % NQF][j][1];
          }
        }
        if constexpr (V == VISC_TABLE) {
          const int cls = info[el] >> 3, walls = info[el] & 7;
          const double *tab = dn + cls * NF * NS + j, *vo = dn + m.n_class * NF * NS + cls * NS * NS + j;
          const double* u = U + el * L::LU + c * NS;
#pragma unroll
          for (int p = 0; p < NF; ++p) y += A_[p * L::NA + 2 + c] * tab[p * NS];
          double z = 0.0;
#pragma unroll
          for (int k = 1; k < NS; ++k) z += vo[k * NS] * u[k];   // (mode 0 has no gradient)
          for (int e = 0; walls >> e; ++e)
            if (walls >> e & 1) {   // a boundary facet has no viscous terms
              const double* vf = m.vfac64 + (size_t(cls) * 3 + e) * NS * NS + j;
#pragma unroll
              for (int k = 1; k < NS; ++k) z -= __ldg(&vf[k * NS]) * u[k];
            }
          x += nu * z;
        }
        x += y;
        f = a.mode == MODE_STAGE ? a.a * a.un[size_t(t) * ND + r] + a.b * f + a.c * x : x;
      }
      F[el * L::LF + r] = f;
    }
    __syncthreads();
    // 3: outputs
    if (a.mode == MODE_RESIDUAL || a.mode == MODE_PRESSURE)
      for (int i = threadIdx.x; i < E * ND; i += blockDim.x) {
        const int el = i / ND, r = i - el * ND;
        if (t0 + el < m.n_tri) m.h[size_t(t0 + el) * ND + r] = F[el * L::LF + r];
      }
    if (a.mode == MODE_RESIDUAL) continue;
    const int r0 = a.mode == MODE_PRESSURE ? ND : 0;
    for (int i = threadIdx.x + (r0 << log_e); i < ((ND + L3) << log_e); i += blockDim.x) {
      const int el = i & (E - 1), r = i >> log_e, t = min(t0 + el, m.n_tri - 1);
      const size_t cls = info[el] >> 3;
      const double* row = r < ND ? m.P + (cls * ND + r) * ND : m.G + (cls * L3 + r - ND) * ND;
      const double* f = F + el * L::LF;
      double x = 0.0, y = 0.0;
#pragma unroll
      for (int j = 0; j < ND; j += 2) {
        x += __ldg(&row[j]) * f[j];
        y += __ldg(&row[j + 1]) * f[j + 1];
      }
      if (t0 + el < m.n_tri) {
        if (r < ND) m.h[size_t(t) * ND + r] = x + y;
        else m.gl[size_t(t) * L3 + r - ND] = x + y;
      }
    }
  }
}

// Transposed Jacobian of the residual (adjoint of the stage functional): for the
// state u and a functional w (coefficients), out = c_w w + c_J J_L(u)^T w with
//   (J_L(u)^T w)_j = d/du_j L(u)(w)
//     volume : int psi_j [(u.grad) w + (grad w)^T u]_c - nu int grad psi_j . grad w_c
//     facets : -int psi_j [n_c (u^up . [w]) / 2 + max(u.n, 0) [w]_c]        (upwind flux in its
//              1/2 (u.n)(u+ + u-) + 1/2 |u.n| (u+ - u-) form, sign(0) = 0)
//              + nu int [psi_j ({d_n w}_c - sigma [w]_c) + 1/2 d_n psi_j [w]_c]  (SIPG, symmetric)
// with [w] = w_T - w_neighbour and n the outward normal of T. The viscous part is the
// SIPG residual of w itself (eq. (18) is symmetric). Block partials of
// <u, dL/dnu(u)> = B_h(u, w)/nu with the sign of L, i.e. the nu-derivative of
// L(u)(w), go to red[blockIdx]. Tasks as in k_stage64.
template <int K, int V>
struct AdjointTile : Tile<K> {
  using L = Tile<K>;
  static constexpr int NH = 6, NA = V == VISC_TABLE ? 4 : 6;
  static constexpr int LH = L::NQ * NH + 1, LA = (L::NF * NA) | 1;
  static constexpr int words = 2 * (L::LU + L::LN) + LH + LA;
};

template <int K, int V>
__global__ void __launch_bounds__(kTileThreads) k_adjoint64(DevMesh m, const double* ug, const double* wg, double* out,
                                                            double cw, double cj, int accumulate, int log_e) {
  using D = Dims<K>;
  using L = AdjointTile<K, V>;
  constexpr int NS = D::NS, ND = D::ND, NQ = D::NQ, NQF = D::NQF, NF = 3 * NQF;
  __shared__ SmemTables<K, double> T;
  extern __shared__ double tile_smem[];
  const int E = 1 << log_e;
  double* U = tile_smem;
  double* W = U + E * L::LU;
  double* UN = W + E * L::LU;
  double* WN = UN + E * L::LN;
  double* H = WN + E * L::LN;
  double* A = H + E * L::LH;
  double* dn = A + E * L::LA;
  load_tables<K, double>(m, T);
  if constexpr (V == VISC_TABLE)
    for (int i = threadIdx.x; i < m.n_class * NF * NS; i += blockDim.x) dn[i] = __ldg(&m.dn64[i]);
  const double nu = m.nu;
  double nupart = 0.0;
  const int ntiles = (m.n_tri + E - 1) >> log_e;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int t0 = tile << log_e;
    __syncthreads();
    load_tile<K>(m, ug, t0, E, U, UN);
    load_tile<K>(m, wg, t0, E, W, WN);
    __syncthreads();
    for (int i = threadIdx.x; i < (L::PTS << log_e); i += blockDim.x) {
      const int el = i & (E - 1), pt = i >> log_e, t = min(t0 + el, m.n_tri - 1);
      const bool live = t0 + el < m.n_tri;
      const double *u = U + el * L::LU, *x = W + el * L::LU;
      if (pt < NQ) {
        const double* geo = m.geo + size_t(__ldg(&m.tri_class[t])) * kGeo;
        const double J0 = __ldg(&geo[G_JINV]), J1 = __ldg(&geo[G_JINV + 1]), J2 = __ldg(&geo[G_JINV + 2]),
                     J3 = __ldg(&geo[G_JINV + 3]), s = __ldg(&geo[G_S]);
        double u0 = 0, u1 = 0, p[2][2] = {{0, 0}, {0, 0}}, b[2][2] = {{0, 0}, {0, 0}};
#pragma unroll
        for (int j = 0; j < NS; ++j) {
          const double ph = T.vphi[pt][j], d0 = T.vdphi[pt][j][0], d1 = T.vdphi[pt][j][1];
          u0 += ph * u[j];
          u1 += ph * u[NS + j];
          p[0][0] += d0 * x[j];
          p[0][1] += d1 * x[j];
          p[1][0] += d0 * x[NS + j];
          p[1][1] += d1 * x[NS + j];
          b[0][0] += d0 * u[j];
          b[0][1] += d1 * u[j];
          b[1][0] += d0 * u[NS + j];
          b[1][1] += d1 * u[NS + j];
        }
        u0 *= s;
        u1 *= s;
        double gw[2][2], gu[2][2];   // physical gradients d w_c / d x_d, d u_c / d x_d
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          gw[c][0] = s * (p[c][0] * J0 + p[c][1] * J2);
          gw[c][1] = s * (p[c][0] * J1 + p[c][1] * J3);
          gu[c][0] = s * (b[c][0] * J0 + b[c][1] * J2);
          gu[c][1] = s * (b[c][0] * J1 + b[c][1] * J3);
        }
        const double w = T.vw[pt] * __ldg(&geo[G_DET]), ws = w * s, wn = -ws * nu;
        double* h = H + el * L::LH + pt * L::NH;
        // value-type test terms A_c = (u.grad) w_c + sum_d u_d d_c w_d
        h[0] = ws * (u0 * gw[0][0] + u1 * gw[0][1] + u0 * gw[0][0] + u1 * gw[1][0]);
        h[1] = ws * (u0 * gw[1][0] + u1 * gw[1][1] + u0 * gw[0][1] + u1 * gw[1][1]);
        // gradient-type test terms: -nu grad w_c . grad psi_j, written through reference gradients
        h[2] = wn * (gw[0][0] * J0 + gw[0][1] * J1);
        h[3] = wn * (gw[0][0] * J2 + gw[0][1] * J3);
        h[4] = wn * (gw[1][0] * J0 + gw[1][1] * J1);
        h[5] = wn * (gw[1][0] * J2 + gw[1][1] * J3);
        if (live) nupart -= w * (gu[0][0] * gw[0][0] + gu[0][1] * gw[0][1] + gu[1][0] * gw[1][0] + gu[1][1] * gw[1][1]);
      } else {
        const int e = (pt - NQ) / NQF, q = pt - NQ - e * NQF;
        const int tn = __ldg(&m.tri_nbr[size_t(t) * 3 + e]);
        double* o = A + el * L::LA + (pt - NQ) * L::NA;
        if (tn < 0) {   // walls: no term in the forward residual, none in its transpose
#pragma unroll
          for (int z = 0; z < L::NA; ++z) o[z] = 0.0;
          continue;
        }
        FacetGeo<K, V> g;
        facet_geo<K, V>(m, t, e, tn, g);
        double ui[2], uo[2], wi[2], wo[2], dui[2], dwi[2], dwo[2], none[2];
        facet_trace<K, V, true>(T, dn, u, e, q, g.cls, g.s, 1.0, g.mo0, g.mo1, ui, dui);
        facet_trace<K, V, true>(T, dn, x, e, q, g.cls, g.s, 1.0, g.mo0, g.mo1, wi, dwi);
        facet_trace<K, V, false>(T, dn, UN + el * L::LN + e * ND, g.en, NQF - 1 - q, g.ncls, g.sn, -1.0, 0.0, 0.0, uo,
                                 none);
        facet_trace<K, V, true>(T, dn, WN + el * L::LN + e * ND, g.en, NQF - 1 - q, g.ncls, g.sn, -1.0, g.mn0, g.mn1, wo,
                                dwo);
        const double vn = 0.5 * ((ui[0] + uo[0]) * g.n0 + (ui[1] + uo[1]) * g.n1);
        const double sg = vn > 0.0 ? 1.0 : (vn < 0.0 ? -1.0 : 0.0);
        const double jw[2] = {wi[0] - wo[0], wi[1] - wo[1]};
        const double upj = 0.5 * (((ui[0] + uo[0]) + sg * (ui[0] - uo[0])) * jw[0] +
                                  ((ui[1] + uo[1]) + sg * (ui[1] - uo[1])) * jw[1]);
        const double vp = vn > 0.0 ? vn : 0.0;
        const double w = T.fw[q] * g.len, ws = w * g.s;
        // value-type: convective adjoint + SIPG consistency and penalty of w (nu)
        // u.n is the average of both traces: d(u.n)/du_T = n/2
        const double nrm[2] = {g.n0, g.n1};
        double np = 0.0;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const double sip = 0.5 * (dwi[c] + dwo[c]) - g.sig * jw[c];
          o[c] = ws * (nu * sip - (0.5 * nrm[c] * upj + vp * jw[c]));
          // normal-derivative test: SIPG symmetry term
          const double B = ws * 0.5 * nu * jw[c];
          if constexpr (V == VISC_TABLE) {
            o[2 + c] = B;
          } else {
            o[2 + 2 * c] = B * g.mo0;
            o[3 + 2 * c] = B * g.mo1;
          }
          np += ui[c] * sip + 0.5 * dui[c] * jw[c];
        }
        if (live) nupart += w * np;
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < (ND << log_e); i += blockDim.x) {
      const int el = i & (E - 1), r = i >> log_e, c = r / NS, j = r - c * NS;
      if (t0 + el >= m.n_tri) continue;
      const double *h = H + el * L::LH, *A_ = A + el * L::LA;
      double x = 0.0, y = 0.0;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        x += h[q * L::NH + c] * T.vphi[q][j];
        y += h[q * L::NH + 2 + 2 * c] * T.vdphi[q][j][0];
        x += h[q * L::NH + 3 + 2 * c] * T.vdphi[q][j][1];
      }
#pragma unroll
      for (int p = 0; p < NF; ++p) {
        x += A_[p * L::NA + c] * T.fphi[p / NQF][p % NQF][j];
        if constexpr (V == VISC_GENERAL) {
          y += A_[p * L::NA + 2 + 2 * c] * T.fdphi[p / NQF][p % NQF][j][0];
          y += A_[p * L::NA + 3 + 2 * c] * T.fdphi[p / NQF][p % NQF][j][1];
        }
      }
      if constexpr (V == VISC_TABLE) {
        const double* tab = dn + __ldg(&m.tri_class[t0 + el]) * NF * NS + j;
#pragma unroll
        for (int p = 0; p < NF; ++p) y += A_[p * L::NA + 2 + c] * tab[p * NS];
      }
      const size_t o = size_t(t0 + el) * ND + r;
      const double v = cw * W[el * L::LU + r] + cj * (x + y);
      out[o] = accumulate ? out[o] + v : v;
    }
  }
  nupart = block_sum(nupart);
  if (threadIdx.x == 0) m.red[blockIdx.x] = nupart;
}

// acc_dev += coef * (sum of the k_adjoint64 block partials), in fixed order.
__global__ void k_nu_accumulate(DevMesh m, int nparts, double coef, double* acc_dev) {
  if (threadIdx.x >= 32) return;
  double v = 0.0;
  for (int i = threadIdx.x; i < nparts; i += 32) v += m.red[i];
  v = warp_sum(v);
  if (threadIdx.x == 0) *acc_dev += coef * v;
}

// Triangles a tile (log2), threads, blocks and dynamic shared memory: a tile's points fill the
// threads, a block's tables and tile stay within the 48 KB that need no opt-in, and blocks (eight an
// SM at most) take several tiles each, so that the tables are read once.
struct TileShape {
  int log_e, threads, blocks;
  size_t smem;
};
template <int K, int V, typename T>
cudaError_t tile_shape(const DevMesh& m, TileShape& s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const size_t table =
      V == VISC_TABLE ? size_t(m.n_class) * (3 * Dims<K>::NQF + Dims<K>::NS) * Dims<K>::NS : 0;
  const size_t room = 48 * 1024 - sizeof(SmemTables<K, double>) - 512;
  s.log_e = 4;
  while (s.log_e > 0 && ((m.n_tri >> s.log_e) < 2 * sms || ((size_t(T::words) << s.log_e) + table) * 8 > room)) --s.log_e;
  s.threads = s.log_e >= 2 ? kTileThreads : 32 << s.log_e;
  s.smem = ((size_t(T::words) << s.log_e) + table) * 8;
  s.blocks = std::min((m.n_tri + (1 << s.log_e) - 1) >> s.log_e, 8 * sms);
  return cudaSuccess;
}

template <int K, int V>
cudaError_t stage64(const DevMesh& m, const StageArgs& a, cudaStream_t st) {
  TileShape s;
  const cudaError_t e = tile_shape<K, V, StageTile<K, V>>(m, s);
  if (e != cudaSuccess) return e;
  k_stage64<K, V><<<s.blocks, s.threads, s.smem, st>>>(m, a, s.log_e);
  return cudaGetLastError();
}

template <int K, int V>
cudaError_t adjoint64(const DevMesh& m, const double* u, const double* w, double* out, double cw, double cj,
                      int accumulate, double nu_coef, double* nu_acc, cudaStream_t st) {
  TileShape s;
  const cudaError_t e = tile_shape<K, V, AdjointTile<K, V>>(m, s);
  if (e != cudaSuccess) return e;
  k_adjoint64<K, V><<<s.blocks, s.threads, s.smem, st>>>(m, u, w, out, cw, cj, accumulate, s.log_e);
  k_nu_accumulate<<<1, 32, 0, st>>>(m, s.blocks, nu_coef, nu_acc);
  return cudaGetLastError();
}

}  // namespace

#define DGDF_DISPATCH_K(kv, ...) \
  switch (kv) {                   \
    case 1: { constexpr int K = 1; __VA_ARGS__; break; } \
    case 2: { constexpr int K = 2; __VA_ARGS__; break; } \
    case 3: { constexpr int K = 3; __VA_ARGS__; break; } \
    default: return cudaErrorInvalidValue;        \
  }

cudaError_t launch_stage(const DevMesh& m, const StageArgs& a, cudaStream_t s) {
  if (m.elem_df) return launch_stage_df(m, a, s);
  // nu = 0 leaves out every gradient and normal derivative: they would be multiplied by zero
  if (m.nu == 0.0) {
    DGDF_DISPATCH_K(m.k, return stage64<K, VISC_NONE>(m, a, s));
  } else if (m.dn64) {
    DGDF_DISPATCH_K(m.k, return stage64<K, VISC_TABLE>(m, a, s));
  } else {
    DGDF_DISPATCH_K(m.k, return stage64<K, VISC_GENERAL>(m, a, s));
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_adjoint(const DevMesh& m, const double* u, const double* w, double* out, double cw, double cj,
                           int accumulate, double nu_coef, double* nu_acc, cudaStream_t s) {
  if (cj == 0.0 && nu_coef == 0.0)   // no Jacobian: out (+)= cw w
    return launch_axpby64(accumulate ? out : w, w, out, accumulate ? 1.0 : cw, accumulate ? cw : 0.0,
                          (long long)m.n_tri * m.nd, s);
  if (m.dn64) {
    DGDF_DISPATCH_K(m.k, return adjoint64<K, VISC_TABLE>(m, u, w, out, cw, cj, accumulate, nu_coef, nu_acc, s));
  } else {
    DGDF_DISPATCH_K(m.k, return adjoint64<K, VISC_GENERAL>(m, u, w, out, cw, cj, accumulate, nu_coef, nu_acc, s));
  }
  return cudaErrorInvalidValue;
}

}  // namespace dgdf
