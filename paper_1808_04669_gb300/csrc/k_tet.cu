// Kernels of the three-dimensional path (closed tetrahedral meshes, FP64): the stage residual +
// condensation, the recovery, the face-system PCG and the lattice / diagnostics helpers.
// The volume tables sit in shared memory, the face tables (four local faces x six vertex orderings) are read through the L1 cache.
// Conventions (canonical face coordinates, perm index, face rule): setup3.hpp.
#include <algorithm>

#include "device3.cuh"
#include "kcommon.cuh"
#include "solver_common.cuh"

namespace dgdf {

template <int K>
struct Dims3 {
  static constexpr int NS = (K + 1) * (K + 2) * (K + 3) / 6;
  static constexpr int ND = 3 * NS;
  static constexpr int NL = (K + 1) * (K + 2) / 2;
  static constexpr int NQ1 = (3 * K + 1) / 2;
  static constexpr int NQ = NQ1 * NQ1 * NQ1;
  static constexpr int NQF1 = (3 * K + 2) / 2;
  static constexpr int NQF = NQF1 * NQF1;
};

namespace {

constexpr int kTetThreads = 128;

template <int K>
struct VolTables3 {
  double vw[Dims3<K>::NQ];
  double vphi[Dims3<K>::NQ][Dims3<K>::NS];
  double vdphi[Dims3<K>::NQ][Dims3<K>::NS][3];
};

template <int K>
__device__ void load_vol3(const DevMesh3& m, VolTables3<K>& T) {
  using D = Dims3<K>;
  for (int i = threadIdx.x; i < D::NQ; i += blockDim.x) T.vw[i] = m.vw[i];
  for (int i = threadIdx.x; i < D::NQ * D::NS; i += blockDim.x) (&T.vphi[0][0])[i] = m.vphi[i];
  for (int i = threadIdx.x; i < D::NQ * D::NS * 3; i += blockDim.x) (&T.vdphi[0][0][0])[i] = m.vdphi[i];
}

// How the stage kernel takes the viscous terms: none (nu = 0), with the normal derivatives of the
// basis at the face points from a per-class table (m.dn, at most kDnClasses3 classes), or from
// reference gradients.
enum Visc3 { VISC3_NONE, VISC3_TABLE, VISC3_GENERAL };

// Values v and derivatives d along our normal of the field with coefficients U at face point q: ph,
// fd the basis values and reference gradients of its (local face, vertex order), tab its row of the
// table of derivatives along its own outward normal (sgn times ours), mm = Jinv n.
template <int K, int V>
__device__ __forceinline__ void face_trace3(const double* __restrict__ ph, const double* __restrict__ fd,
                                            const double* __restrict__ tab, const double* U, double s, double sgn,
                                            const double (&mm)[3], double (&v)[3], double (&d)[3]) {
  constexpr int NS = Dims3<K>::NS;
#pragma unroll
  for (int c = 0; c < 3; ++c) v[c] = d[c] = 0.0;
#pragma unroll
  for (int j = 0; j < NS; ++j) {
    const double p = __ldg(&ph[j]);
    double g = 0.0;
    if constexpr (V == VISC3_TABLE) g = __ldg(&tab[j]);
    if constexpr (V == VISC3_GENERAL) g = __ldg(&fd[3 * j]) * mm[0] + __ldg(&fd[3 * j + 1]) * mm[1] + __ldg(&fd[3 * j + 2]) * mm[2];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double x = U[c * NS + j];
      v[c] += p * x;
      if constexpr (V != VISC3_NONE) d[c] += g * x;
    }
  }
  const double sd = V == VISC3_TABLE ? sgn * s : s;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    v[c] *= s;
    d[c] *= sd;
  }
}

// Words of a tetrahedron in a tile: own and neighbours' coefficients, the point terms (volume, then
// faces) and the functional; odd row lengths against bank conflicts.
template <int K, int V>
struct Tile3 {
  using D = Dims3<K>;
  static constexpr int NF = 4 * D::NQF, NA = V == VISC3_NONE ? 3 : (V == VISC3_TABLE ? 6 : 12);
  static constexpr int LU = D::ND + 1, LN = 4 * D::ND + 1, LF = D::ND + 1;
  static constexpr int LH = (D::NQ * 9 > NF * NA ? D::NQ * 9 : NF * NA) | 1;
  static constexpr int words = LU + LN + LH + LF;
};

// Stage kernel (modes as StageMode): f = a u^n + b u' + c L(u') (MODE_STAGE), L(u') alone
// (MODE_RESIDUAL: h = f, the Riesz representer since M = I; MODE_PRESSURE: h = f and gl = G f),
// or f = u' (MODE_PROJECT); then h = P f and gl = G f per class.
// L(u)(phi) = -C_h(u; u, phi) - B_h(u, phi) (eq. (7), eq. (18)). Volume: int (u x u - nu grad u) :
// grad phi. Faces: the upwind flux with u.n the average of both traces, and the SIPG consistency,
// symmetry and penalty terms, at the shared face points (both sides evaluate at the same canonical
// points, so point q is point q on either side).
// Bound: the FP64 pipes (an instruction of a warp takes a quarter of an SM 64 cycles). A thread a
// tetrahedron held 255 registers and spilled, and 24576 tetrahedra left the last wave a quarter
// full; here a block takes a tile of E = 2^log_e through shared memory and deals out volume points,
// face points, test functions and operator rows to all its threads, in phases. 16^3 cubes, BDM_2:
// 2.09 -> 1.05 ms a launch.
template <int K, int V>
__global__ void __launch_bounds__(kTetThreads) k_stage3(DevMesh3 m, StageArgs a, int log_e) {
  using D = Dims3<K>;
  using L = Tile3<K, V>;
  constexpr int NS = D::NS, ND = D::ND, NQ = D::NQ, NQF = D::NQF, L4 = 4 * D::NL;
  __shared__ VolTables3<K> T;
  extern __shared__ double tile3_smem[];
  const int E = 1 << log_e;
  double* U = tile3_smem;
  double* N = U + E * L::LU;
  double* H = N + E * L::LN;   // volume terms, then face terms
  double* F = H + E * L::LH;
  load_vol3<K>(m, T);
  const double nu = m.nu;
  const int ntiles = (m.n_tet + E - 1) >> log_e;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int t0 = tile << log_e;
    auto tet = [&](int el) { return min(t0 + el, m.n_tet - 1); };
    __syncthreads();
    for (int i = threadIdx.x; i < E * ND; i += blockDim.x) {
      const int el = i / ND, j = i - el * ND;
      U[el * L::LU + j] = a.up[size_t(tet(el)) * ND + j];
    }
    const bool res = a.mode != MODE_PROJECT;
    if (res)
      for (int i = threadIdx.x; i < E * 4 * ND; i += blockDim.x) {
        const int el = i / (4 * ND), r = i - el * 4 * ND, e = r / ND, j = r - e * ND;
        N[el * L::LN + r] = a.up[size_t(__ldg(&m.tet_nbr[size_t(tet(el)) * 4 + e])) * ND + j];
      }
    __syncthreads();
    if (res) {
      // volume points: H[c][r], the flux in reference directions times the weight
      for (int i = threadIdx.x; i < (NQ << log_e); i += blockDim.x) {
        const int el = i & (E - 1), q = i >> log_e;
        const double* up = U + el * L::LU;
        const double* geo = m.geo + size_t(__ldg(&m.tet_class[tet(el)])) * kGeo3;
        double Ji[9];
#pragma unroll
        for (int x = 0; x < 9; ++x) Ji[x] = __ldg(&geo[G3_JINV + x]);
        const double s = __ldg(&geo[G3_S]);
        double u[3], g[3][3];
#pragma unroll
        for (int c = 0; c < 3; ++c) u[c] = g[c][0] = g[c][1] = g[c][2] = 0.0;
#pragma unroll
        for (int j = 0; j < NS; ++j) {
          const double ph = T.vphi[q][j];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const double x = up[c * NS + j];
            u[c] += ph * x;
            if constexpr (V != VISC3_NONE)
#pragma unroll
              for (int r = 0; r < 3; ++r) g[c][r] += T.vdphi[q][j][r] * x;
          }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) u[c] *= s;
        const double w = T.vw[q] * __ldg(&geo[G3_DET]) * s, ns = nu * s;
        double* h = H + el * L::LH + q * 9;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          double f[3];
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            f[d] = u[c] * u[d];
            // physical gradient du_c/dx_d = s sum_r g_cr Jinv[r][d]
            if constexpr (V != VISC3_NONE)
              f[d] -= ns * (g[c][0] * Ji[d] + g[c][1] * Ji[3 + d] + g[c][2] * Ji[6 + d]);
          }
#pragma unroll
          for (int r = 0; r < 3; ++r) h[3 * c + r] = w * (f[0] * Ji[3 * r] + f[1] * Ji[3 * r + 1] + f[2] * Ji[3 * r + 2]);
        }
      }
      __syncthreads();
      for (int i = threadIdx.x; i < (ND << log_e); i += blockDim.x) {
        const int el = i & (E - 1), r = i >> log_e, c = r / NS, j = r - c * NS;
        const double* h = H + el * L::LH + 3 * c;
        double x = 0.0, y = 0.0, z = 0.0;
#pragma unroll 9
        for (int q = 0; q < NQ; ++q) {
          x += h[9 * q] * T.vdphi[q][j][0];
          y += h[9 * q + 1] * T.vdphi[q][j][1];
          z += h[9 * q + 2] * T.vdphi[q][j][2];
        }
        F[el * L::LF + r] = x + y + z;
      }
      __syncthreads();
      // face points: A[c] against phi_c, B[c] against its normal derivative (general: B (Jinv n)_r
      // against its reference gradient)
      for (int i = threadIdx.x; i < (L::NF << log_e); i += blockDim.x) {
        const int el = i & (E - 1), p = i >> log_e, e = p / NQF, q = p - e * NQF, t = tet(el);
        const int tn = __ldg(&m.tet_nbr[size_t(t) * 4 + e]), en = __ldg(&m.tet_nbr_loc[size_t(t) * 4 + e]);
        const int co = __ldg(&m.tet_class[t]), cn = __ldg(&m.tet_class[tn]);
        const double *geo = m.geo + size_t(co) * kGeo3, *geon = m.geo + size_t(cn) * kGeo3;
        const int ro = (e * 6 + int(__ldg(&geo[G3_PERM + e]))) * NQF + q;
        const int rn = (en * 6 + int(__ldg(&geon[G3_PERM + en]))) * NQF + q;
        const double n[3] = {__ldg(&geo[G3_NRM + 3 * e]), __ldg(&geo[G3_NRM + 3 * e + 1]), __ldg(&geo[G3_NRM + 3 * e + 2])};
        const double s = __ldg(&geo[G3_S]), sn = __ldg(&geon[G3_S]);
        double mo[3] = {0, 0, 0}, mn[3] = {0, 0, 0};
        if constexpr (V == VISC3_GENERAL)
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            mo[r] = __ldg(&geo[G3_JINV + 3 * r]) * n[0] + __ldg(&geo[G3_JINV + 3 * r + 1]) * n[1] + __ldg(&geo[G3_JINV + 3 * r + 2]) * n[2];
            mn[r] = __ldg(&geon[G3_JINV + 3 * r]) * n[0] + __ldg(&geon[G3_JINV + 3 * r + 1]) * n[1] +
                    __ldg(&geon[G3_JINV + 3 * r + 2]) * n[2];
          }
        const double *to = nullptr, *tb = nullptr;
        if constexpr (V == VISC3_TABLE) {
          to = m.dn + (size_t(co * 4 + e) * NQF + q) * NS;
          tb = m.dn + (size_t(cn * 4 + en) * NQF + q) * NS;
        }
        double ui[3], di[3], uo[3], dn[3];
        face_trace3<K, V>(m.fphi + size_t(ro) * NS, m.fdphi + size_t(ro) * NS * 3, to, U + el * L::LU, s, 1.0, mo, ui, di);
        face_trace3<K, V>(m.fphi + size_t(rn) * NS, m.fdphi + size_t(rn) * NS * 3, tb, N + el * L::LN + e * ND, sn, -1.0,
                          mn, uo, dn);
        const double vn = 0.5 * ((ui[0] + uo[0]) * n[0] + (ui[1] + uo[1]) * n[1] + (ui[2] + uo[2]) * n[2]);
        const double w = __ldg(&m.fw[q]) * 2.0 * __ldg(&geo[G3_AREA + e]) * s, wv = w * vn, wn = w * nu;
        const bool own = vn >= 0.0;
        double* out = H + el * L::LH + p * L::NA;
        double sig = 0.0;
        if constexpr (V != VISC3_NONE) sig = __ldg(&m.face_sigma[__ldg(&m.tet_face[size_t(t) * 4 + e])]);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          double x = -wv * (own ? ui[c] : uo[c]);
          if constexpr (V != VISC3_NONE) {
            const double jc = ui[c] - uo[c], B = 0.5 * wn * jc;
            x += wn * (0.5 * (di[c] + dn[c]) - sig * jc);
            if constexpr (V == VISC3_TABLE) {
              out[3 + c] = B;
            } else {
#pragma unroll
              for (int r = 0; r < 3; ++r) out[3 + 3 * c + r] = B * mo[r];
            }
          }
          out[c] = x;
        }
      }
      __syncthreads();
    }
    for (int i = threadIdx.x; i < (ND << log_e); i += blockDim.x) {
      const int el = i & (E - 1), r = i >> log_e, c = r / NS, j = r - c * NS, t = tet(el);
      double f = U[el * L::LU + r];
      if (res) {
        const int co = __ldg(&m.tet_class[t]);
        const double* geo = m.geo + size_t(co) * kGeo3;
        const double* h = H + el * L::LH;
        double x = F[el * L::LF + r], y = 0.0;
#pragma unroll 1
        for (int e = 0; e < 4; ++e) {
          const int ro = (e * 6 + int(__ldg(&geo[G3_PERM + e]))) * NQF;
          const double* ph = m.fphi + size_t(ro) * NS + j;
          const double* fd = m.fdphi + (size_t(ro) * NS + j) * 3;
          const double* tab = V == VISC3_TABLE ? m.dn + size_t(co * 4 + e) * NQF * NS + j : nullptr;
          const double* A = h + e * NQF * L::NA;
#pragma unroll 8
          for (int q = 0; q < NQF; ++q) {
            x += A[q * L::NA + c] * __ldg(&ph[q * NS]);
            if constexpr (V == VISC3_TABLE) y += A[q * L::NA + 3 + c] * __ldg(&tab[q * NS]);
            if constexpr (V == VISC3_GENERAL) {
              y += A[q * L::NA + 3 + 3 * c] * __ldg(&fd[q * NS * 3]);
              y += A[q * L::NA + 4 + 3 * c] * __ldg(&fd[q * NS * 3 + 1]);
              y += A[q * L::NA + 5 + 3 * c] * __ldg(&fd[q * NS * 3 + 2]);
            }
          }
        }
        x += y;
        f = a.mode == MODE_STAGE ? a.a * a.un[size_t(t) * ND + r] + a.b * f + a.c * x : x;
      }
      F[el * L::LF + r] = f;
    }
    __syncthreads();
    if (a.mode == MODE_RESIDUAL || a.mode == MODE_PRESSURE)
      for (int i = threadIdx.x; i < E * ND; i += blockDim.x) {
        const int el = i / ND, r = i - el * ND;
        if (t0 + el < m.n_tet) m.h[size_t(t0 + el) * ND + r] = F[el * L::LF + r];
      }
    if (a.mode == MODE_RESIDUAL) continue;
    const int r0 = a.mode == MODE_PRESSURE ? ND : 0;
    for (int i = threadIdx.x + (r0 << log_e); i < ((ND + L4) << log_e); i += blockDim.x) {
      const int el = i & (E - 1), r = i >> log_e, t = tet(el);
      const size_t cls = __ldg(&m.tet_class[t]);
      const double* row = r < ND ? m.P + (cls * ND + r) * ND : m.G + (cls * L4 + r - ND) * ND;
      const double* f = F + el * L::LF;
      double x = 0.0, y = 0.0;
#pragma unroll
      for (int j = 0; j < ND; j += 2) {
        x += __ldg(&row[j]) * f[j];
        y += __ldg(&row[j + 1]) * f[j + 1];
      }
      if (t0 + el < m.n_tet) {
        if (r < ND) m.h[size_t(t) * ND + r] = x + y;
        else m.gl[size_t(t) * L4 + r - ND] = x + y;
      }
    }
  }
}

// Recovery u = P f - G^T lam_T (eq. (12) condensed): h holds P f. A thread per coefficient.
template <int K>
__global__ void __launch_bounds__(kTetThreads) k_recover3(DevMesh3 m, double* out) {
  using D = Dims3<K>;
  constexpr int ND = D::ND, NL = D::NL, L4 = 4 * NL;
  const long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (o >= (long long)m.n_tet * ND) return;
  const int t = int(o / ND), i = int(o - (long long)t * ND);
  const double* G = m.G + size_t(__ldg(&m.tet_class[t])) * L4 * ND + i;
  double v = m.h[o], w = 0.0;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const double* lam = m.lam + size_t(__ldg(&m.tet_face[size_t(t) * 4 + e])) * NL;
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      if (j & 1) w -= __ldg(&G[(e * NL + j) * ND]) * lam[j];
      else v -= __ldg(&G[(e * NL + j) * ND]) * lam[j];
    }
  }
  out[o] = v + w;
}

// Element pressure of eq. (12) (h = f of MODE_PRESSURE, lam the solve's multipliers):
// w = W (f - C^T lam) = W f - WC lam, in the basis s phi_m (m < nw) of P^(k-1); its values at the
// (k-1)-lattice points go to pe, and each block's sum of the integrals of w to part.
template <int K>
__global__ void __launch_bounds__(kTetThreads) k_pressure3(DevMesh3 m, double* pe, double* part) {
  using D = Dims3<K>;
  constexpr int ND = D::ND, NS = D::NS, NL = D::NL, L4 = 4 * NL, NW = K * (K + 1) * (K + 2) / 6;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  double integral = 0.0;
  if (t < m.n_tet) {
    double f[ND], lam[L4], w[NW];
#pragma unroll
    for (int i = 0; i < ND; ++i) f[i] = m.h[size_t(t) * ND + i];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int fc = m.tet_face[size_t(t) * 4 + e];
#pragma unroll
      for (int j = 0; j < NL; ++j) lam[e * NL + j] = m.lam[size_t(fc) * NL + j];
    }
    const int cls = m.tet_class[t];
    const double* W = m.W + size_t(cls) * NW * ND;
    const double* WC = m.WC + size_t(cls) * NW * L4;
#pragma unroll
    for (int a = 0; a < NW; ++a) {
      double v = 0.0;
#pragma unroll
      for (int j = 0; j < ND; ++j) v += __ldg(&W[a * ND + j]) * f[j];
#pragma unroll
      for (int l = 0; l < L4; ++l) v -= __ldg(&WC[a * L4 + l]) * lam[l];
      w[a] = v;
    }
    const double sc = m.geo[size_t(cls) * kGeo3 + G3_S], det = m.geo[size_t(cls) * kGeo3 + G3_DET];
#pragma unroll
    for (int p = 0; p < NW; ++p) {
      double v = 0.0;
#pragma unroll
      for (int a = 0; a < NW; ++a) v += __ldg(&m.plat_phi[p * NW + a]) * w[a];
      pe[size_t(t) * NW + p] = sc * v;
    }
    for (int q = 0; q < D::NQ; ++q) {
      double v = 0.0;
#pragma unroll
      for (int a = 0; a < NW; ++a) v += __ldg(&m.vphi[q * NS + a]) * w[a];
      integral += __ldg(&m.vw[q]) * v;
    }
    integral *= det * sc;
  }
  integral = block_sum(integral);
  if (threadIdx.x == 0) part[blockIdx.x] = integral;
}

// The mean c = (sum of the block integrals) / vol, the same in every block (fixed order); pe -= c,
// and the face pressure pf = (the multiplier basis at the face's k-lattice) lam - c.
__global__ void k_pressure3_finish(DevMesh3 m, double* pe, double* pf, const double* part, int nparts, double vol) {
  double a = 0.0;
  for (int b = threadIdx.x; b < nparts; b += blockDim.x) a += part[b];
  const double c = block_sum(a) / vol;
  const size_t gtid = size_t(blockIdx.x) * blockDim.x + threadIdx.x, gsz = size_t(gridDim.x) * blockDim.x;
  const size_t npe = size_t(m.n_tet) * m.nw;
  for (size_t i = gtid; i < npe; i += gsz) pe[i] -= c;
  if (!pf) return;
  const int nl = m.nl;
  const size_t npf = size_t(m.n_face) * nl;
  for (size_t i = gtid; i < npf; i += gsz) {
    const size_t fc = i / nl;
    const int p = int(i - fc * nl);
    double v = 0.0;
    for (int j = 0; j < nl; ++j) v += __ldg(&m.mu_lat[p * nl + j]) * m.lam[fc * nl + j];
    pf[i] = v - c;
  }
}

// Grid sum of N per-thread partials (fixed order; the result in every thread).
template <int N>
__device__ bool reduce3(const DevMesh3& m, Barrier& bar, int slot0, double (&v)[N]) {
  double s[N];
#pragma unroll
  for (int i = 0; i < N; ++i) s[i] = block_sum(v[i]);
  if (threadIdx.x == 0)
#pragma unroll
    for (int i = 0; i < N; ++i) m.red[size_t(slot0 + i) * kMaxSolverBlocks + blockIdx.x] = s[i];
  if (!grid_sync(bar, m.stats)) return false;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    double a = 0.0;
    for (int b = threadIdx.x; b < gridDim.x; b += blockDim.x) a += __ldcg(&m.red[size_t(slot0 + i) * kMaxSolverBlocks + b]);
    v[i] = block_sum(a);
  }
  return true;
}

// y = (S x)_f: the face's own block and the blocks of the three other faces of each side
template <int NL>
__device__ __forceinline__ void spmv3(const DevMesh3& m, int f, const double* x, double (&y)[NL]) {
  const double* blk = m.st_blk + size_t(__ldg(&m.face_stencil[f])) * 7 * NL * NL;
#pragma unroll
  for (int i = 0; i < NL; ++i) y[i] = 0.0;
#pragma unroll
  for (int b = 0; b < 7; ++b) {
    const int g = b == 0 ? f : __ldg(&m.face_nbr[size_t(f) * 6 + b - 1]);
    double xs[NL];
#pragma unroll
    for (int j = 0; j < NL; ++j) xs[j] = __ldcg(&x[size_t(g) * NL + j]);
#pragma unroll
    for (int i = 0; i < NL; ++i)
#pragma unroll
      for (int j = 0; j < NL; ++j) y[i] += __ldg(&blk[(b * NL + i) * NL + j]) * xs[j];
  }
}

template <int NL>
__device__ __forceinline__ void binv3(const DevMesh3& m, int f, const double (&r)[NL], double (&z)[NL]) {
  const double* B = m.st_binv + size_t(__ldg(&m.face_stencil[f])) * NL * NL;
#pragma unroll
  for (int i = 0; i < NL; ++i) {
    double v = 0.0;
#pragma unroll
    for (int j = 0; j < NL; ++j) v += __ldg(&B[i * NL + j]) * r[j];
    z[i] = v;
  }
}

// Face-system solve, one persistent cooperative kernel: g = both sides' G f (no orientation
// signs: both sides use the canonical face basis), lam0 from the history or warm_scale lam
// (warm_start_row), the constant multiplier (mode 0 on every face, the kernel of S on a closed
// mesh) removed from g, then FP64 PCG with the block-Jacobi preconditioner. Residual norms
// leave out the mode-0 mean.
template <int K>
__global__ void __launch_bounds__(kSolverThreads) k_solve3(DevMesh3 m, SolveArgs a) {
  constexpr int NL = Dims3<K>::NL, L4 = 4 * NL;
  const int nF = m.n_face;
  const int gtid = blockIdx.x * blockDim.x + threadIdx.x, gsz = gridDim.x * blockDim.x;
  const double inv_nf = 1.0 / double(nF);
  Barrier bar(m.bar);
  double gg[2] = {0.0, 0.0};
  for (int f = gtid; f < nF; f += gsz) {
    const int t0 = m.face_tet[size_t(f) * 2], t1 = m.face_tet[size_t(f) * 2 + 1];
    const int e0 = m.face_loc[size_t(f) * 2], e1 = m.face_loc[size_t(f) * 2 + 1];
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      const double v = m.gl[size_t(t0) * L4 + e0 * NL + j] + m.gl[size_t(t1) * L4 + e1 * NL + j];
      const size_t o = size_t(f) * NL + j;
      m.g[o] = v;
      gg[0] += v * v;
      if (j == 0) gg[1] += v;
    }
    warm_start_row<NL>(m.lam, a, size_t(f) * NL);
  }
  if (!reduce3<2>(m, bar, 4, gg)) return;
  const double c0 = gg[1] * inv_nf;
  const double gnorm = sqrt(nonneg(gg[0] - gg[1] * gg[1] * inv_nf));
  const double stop = a.rtol * gnorm;
  int it = 0;
  bool conv = false;
  double rr = 0.0;
  if (!(gnorm > 0.0)) {   // no data, or a NaN (a state that holds one): zero
    for (int f = gtid; f < nF; f += gsz)
#pragma unroll
      for (int j = 0; j < NL; ++j) m.lam[size_t(f) * NL + j] = 0.0;
    conv = true;
  } else {
    // r = g - c0 1 - S lam, z = B r
    double red[3] = {0.0, 0.0, 0.0};
    for (int f = gtid; f < nF; f += gsz) {
      double y[NL], r[NL], z[NL];
      spmv3<NL>(m, f, m.lam, y);
#pragma unroll
      for (int j = 0; j < NL; ++j) r[j] = m.g[size_t(f) * NL + j] - (j == 0 ? c0 : 0.0) - y[j];
      binv3<NL>(m, f, r, z);
#pragma unroll
      for (int j = 0; j < NL; ++j) {
        m.r[size_t(f) * NL + j] = r[j];
        m.z[size_t(f) * NL + j] = z[j];
        red[0] += r[j] * z[j];
        red[1] += r[j] * r[j];
      }
      red[2] += r[0];
    }
    if (!reduce3<3>(m, bar, 1, red)) return;
    if (drop_start(a, nonneg(red[1] - red[2] * red[2] * inv_nf), gnorm)) {
      red[0] = red[1] = red[2] = 0.0;
      for (int f = gtid; f < nF; f += gsz) {
        double r[NL], z[NL];
#pragma unroll
        for (int j = 0; j < NL; ++j) r[j] = m.g[size_t(f) * NL + j] - (j == 0 ? c0 : 0.0);
        binv3<NL>(m, f, r, z);
#pragma unroll
        for (int j = 0; j < NL; ++j) {
          m.lam[size_t(f) * NL + j] = 0.0;
          m.r[size_t(f) * NL + j] = r[j];
          m.z[size_t(f) * NL + j] = z[j];
          red[0] += r[j] * z[j];
          red[1] += r[j] * r[j];
        }
        red[2] += r[0];
      }
      // (other slots: blocks may still read the first sums)
      if (!reduce3<3>(m, bar, 4, red)) return;
    }
    double rho = red[0];
    rr = nonneg(red[1] - red[2] * red[2] * inv_nf);
    double beta = 0.0;
    double* pold = m.pa;
    double* pnew = m.pb;
    for (;; ++it) {
      if (!isfinite(rr) || !isfinite(rho)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&m.stats->flags, kFlagNonFinite);
        break;
      }
      if (sqrt(rr) <= stop) {
        conv = true;
        break;
      }
      if (it >= a.maxit) break;
      // p_new = z + beta p_old (own rows), q = S p_new (from the neighbours' z and p_old)
      double pq[1] = {0.0};
      for (int f = gtid; f < nF; f += gsz) {
        const double* blk = m.st_blk + size_t(__ldg(&m.face_stencil[f])) * 7 * NL * NL;
        double y[NL], p0[NL];
#pragma unroll
        for (int i = 0; i < NL; ++i) y[i] = 0.0;
#pragma unroll
        for (int b = 0; b < 7; ++b) {
          const int g = b == 0 ? f : __ldg(&m.face_nbr[size_t(f) * 6 + b - 1]);
          double xs[NL];
#pragma unroll
          for (int j = 0; j < NL; ++j) {
            const size_t o = size_t(g) * NL + j;
            xs[j] = it == 0 ? __ldcg(&m.z[o]) : __ldcg(&m.z[o]) + beta * __ldcg(&pold[o]);
            if (b == 0) p0[j] = xs[j];
          }
#pragma unroll
          for (int i = 0; i < NL; ++i)
#pragma unroll
            for (int j = 0; j < NL; ++j) y[i] += __ldg(&blk[(b * NL + i) * NL + j]) * xs[j];
        }
#pragma unroll
        for (int j = 0; j < NL; ++j) {
          pnew[size_t(f) * NL + j] = p0[j];
          m.q[size_t(f) * NL + j] = y[j];
          pq[0] += p0[j] * y[j];
        }
      }
      if (!reduce3<1>(m, bar, 0, pq)) return;
      if (!(pq[0] > 0.0)) {
        if (!isfinite(pq[0]) && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&m.stats->flags, kFlagNonFinite);
        break;
      }
      const double alpha = rho / pq[0];
      double red2[3] = {0.0, 0.0, 0.0};
      for (int f = gtid; f < nF; f += gsz) {
        double r[NL], z[NL];
#pragma unroll
        for (int j = 0; j < NL; ++j) {
          const size_t o = size_t(f) * NL + j;
          m.lam[o] += alpha * pnew[o];
          r[j] = m.r[o] - alpha * m.q[o];
          m.r[o] = r[j];
        }
        binv3<NL>(m, f, r, z);
#pragma unroll
        for (int j = 0; j < NL; ++j) {
          m.z[size_t(f) * NL + j] = z[j];
          red2[0] += r[j] * z[j];
          red2[1] += r[j] * r[j];
        }
        red2[2] += r[0];
      }
      if (!reduce3<3>(m, bar, 1, red2)) return;
      beta = red2[0] / rho;
      rho = red2[0];
      rr = nonneg(red2[1] - red2[2] * red2[2] * inv_nf);
      double* tmp = pold;
      pold = pnew;
      pnew = tmp;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    DevStats* st = m.stats;
    st->last_iters = it;
    st->total_iters += it;
    st->solves += 1;
    st->last_relres = gnorm > 0.0 ? sqrt(rr) / gnorm : 0.0;
    st->last_sweeps = 1;
    st->total_sweeps += 1;
    if (!conv) atomicOr(&st->flags, kFlagNotConverged);
  }
}

// Lattice values [n_tet][ns][3] -> coefficients [n_tet][3 ns]: coef = sqrt(det) Vhat^-1 vals.
template <int K>
__global__ void k_lattice_to_coef3(DevMesh3 m, const double* vals, double* coef) {
  constexpr int NS = Dims3<K>::NS;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= m.n_tet) return;
  const double sq = 1.0 / m.geo[size_t(m.tet_class[t]) * kGeo3 + G3_S];
  for (int c = 0; c < 3; ++c)
    for (int j = 0; j < NS; ++j) {
      double v = 0.0;
      for (int p = 0; p < NS; ++p) v += m.lat_inv[j * NS + p] * vals[(size_t(t) * NS + p) * 3 + c];
      coef[size_t(t) * 3 * NS + c * NS + j] = sq * v;
    }
}

template <int K>
__global__ void __launch_bounds__(kTetThreads) k_coef_to_lattice3(DevMesh3 m, const double* __restrict__ coef,
                                                                  double* __restrict__ vals) {
  constexpr int NS = Dims3<K>::NS, ND = 3 * NS;
  const long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (o >= (long long)m.n_tet * ND) return;
  const int t = int(o / ND), r = int(o - (long long)t * ND), p = r / 3, c = r - 3 * p;
  const double* u = coef + size_t(t) * ND + c * NS;
  double v = 0.0;
#pragma unroll
  for (int j = 0; j < NS; ++j) v += __ldg(&m.lat_phi[p * NS + j]) * u[j];
  vals[o] = __ldg(&m.geo[size_t(__ldg(&m.tet_class[t])) * kGeo3 + G3_S]) * v;
}

// Diagnostics partials per block: energy, enstrophy (|curl u|^2), max |div u| at the volume
// points, max |[u.n]| at the face points (each face seen from both sides).
template <int K>
__global__ void __launch_bounds__(kTetThreads) k_diagnostics3(DevMesh3 m, const double* coef) {
  using D = Dims3<K>;
  constexpr int NS = D::NS, ND = D::ND;
  __shared__ VolTables3<K> T;
  load_vol3<K>(m, T);
  __syncthreads();
  double en = 0.0, ens = 0.0, dmax = 0.0, jmax = 0.0;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < m.n_tet; t += gridDim.x * blockDim.x) {
    double c[ND];
#pragma unroll
    for (int i = 0; i < ND; ++i) {
      c[i] = coef[size_t(t) * ND + i];
      en += c[i] * c[i];
    }
    const double* geo = m.geo + size_t(m.tet_class[t]) * kGeo3;
    const double det = geo[G3_DET], s = geo[G3_S];
    for (int q = 0; q < D::NQ; ++q) {
      double g[3][3];
      for (int cc = 0; cc < 3; ++cc) {
        double a[3] = {0, 0, 0};
        for (int j = 0; j < NS; ++j)
          for (int r = 0; r < 3; ++r) a[r] += T.vdphi[q][j][r] * c[cc * NS + j];
        for (int d = 0; d < 3; ++d)
          g[cc][d] = s * (a[0] * geo[G3_JINV + d] + a[1] * geo[G3_JINV + 3 + d] + a[2] * geo[G3_JINV + 6 + d]);
      }
      const double w0 = g[2][1] - g[1][2], w1 = g[0][2] - g[2][0], w2 = g[1][0] - g[0][1];
      ens += T.vw[q] * det * (w0 * w0 + w1 * w1 + w2 * w2);
      dmax = fmax(dmax, fabs(g[0][0] + g[1][1] + g[2][2]));
    }
    for (int e = 0; e < 4; ++e) {
      const int tn = m.tet_nbr[size_t(t) * 4 + e], en2 = m.tet_nbr_loc[size_t(t) * 4 + e];
      const double* geon = m.geo + size_t(m.tet_class[tn]) * kGeo3;
      const int pe = int(geo[G3_PERM + e]), pn = int(geon[G3_PERM + en2]);
      const double* fo = m.fphi + size_t(e * 6 + pe) * D::NQF * NS;
      const double* fn = m.fphi + size_t(en2 * 6 + pn) * D::NQF * NS;
      for (int q = 0; q < D::NQF; ++q) {
        double jn = 0.0;
        for (int cc = 0; cc < 3; ++cc) {
          double a = 0.0, b = 0.0;
          for (int j = 0; j < NS; ++j) {
            a += fo[q * NS + j] * c[cc * NS + j];
            b += fn[q * NS + j] * coef[size_t(tn) * ND + cc * NS + j];
          }
          jn += (s * a - geon[G3_S] * b) * geo[G3_NRM + 3 * e + cc];
        }
        jmax = fmax(jmax, fabs(jn));
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

__global__ void k_diag_finish3(DevMesh3 m, int nparts) {
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

int blocks3(long long n) { return int((n + kTetThreads - 1) / kTetThreads); }

template <int K>
int solve3_blocks_for() {
  int per_sm = 0, dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_solve3<K>, kSolverThreads, 0);
  return per_sm * sms;
}

}  // namespace

#define DGDF_DISPATCH_K3(k, CALL)                \
  switch (k) {                                   \
    case 1: { constexpr int K = 1; CALL; break; } \
    case 2: { constexpr int K = 2; CALL; break; } \
    default: return cudaErrorInvalidValue;       \
  }

bool tet_tables_match(int k, int nq, int nqf) {
  switch (k) {
    case 1: return nq == Dims3<1>::NQ && nqf == Dims3<1>::NQF;
    case 2: return nq == Dims3<2>::NQ && nqf == Dims3<2>::NQF;
    default: return false;
  }
}

namespace {
// Tiles of up to eight tetrahedra that fit in the 48 KB of shared memory beside the volume tables and
// leave every SM two; a block takes several.
template <int K, int V>
cudaError_t stage3(const DevMesh3& m, const StageArgs& a, cudaStream_t st) {
  using L = Tile3<K, V>;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const size_t room = 48 * 1024 - sizeof(VolTables3<K>) - 64;
  int log_e = 3;
  while (log_e > 0 && ((m.n_tet >> log_e) < 2 * sms || (size_t(L::words) << log_e) * 8 > room)) --log_e;
  const int tiles = (m.n_tet + (1 << log_e) - 1) >> log_e;
  k_stage3<K, V><<<std::min(tiles, 8 * sms), kTetThreads, (size_t(L::words) << log_e) * 8, st>>>(m, a, log_e);
  return cudaGetLastError();
}
template <int K>
cudaError_t stage3_visc(const DevMesh3& m, const StageArgs& a, cudaStream_t s) {
  // nu = 0 leaves out every gradient and normal derivative: they would be multiplied by zero
  if (m.nu == 0.0) return stage3<K, VISC3_NONE>(m, a, s);
  return m.dn ? stage3<K, VISC3_TABLE>(m, a, s) : stage3<K, VISC3_GENERAL>(m, a, s);
}
}  // namespace

cudaError_t launch_stage3(const DevMesh3& m, const StageArgs& a, cudaStream_t s) {
  DGDF_DISPATCH_K3(m.k, return stage3_visc<K>(m, a, s));
  return cudaErrorInvalidValue;
}

cudaError_t launch_recover3(const DevMesh3& m, double* out, cudaStream_t s) {
  DGDF_DISPATCH_K3(m.k, (k_recover3<K><<<blocks3((long long)m.n_tet * m.nd), kTetThreads, 0, s>>>(m, out)));
  return cudaGetLastError();
}

cudaError_t launch_lattice_to_coef3(const DevMesh3& m, const double* vals, double* coef, cudaStream_t s) {
  DGDF_DISPATCH_K3(m.k, (k_lattice_to_coef3<K><<<blocks3(m.n_tet), kTetThreads, 0, s>>>(m, vals, coef)));
  return cudaGetLastError();
}

cudaError_t launch_coef_to_lattice3(const DevMesh3& m, const double* coef, double* vals, cudaStream_t s) {
  DGDF_DISPATCH_K3(m.k, (k_coef_to_lattice3<K><<<blocks3((long long)m.n_tet * m.nd), kTetThreads, 0, s>>>(m, coef, vals)));
  return cudaGetLastError();
}

cudaError_t launch_diagnostics3(const DevMesh3& m, const double* coef, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int nb = blocks3(m.n_tet);
  if (nb > 2 * sms) nb = 2 * sms;
  if (nb > kMaxSolverBlocks) nb = kMaxSolverBlocks;
  DGDF_DISPATCH_K3(m.k, (k_diagnostics3<K><<<nb, kTetThreads, 0, s>>>(m, coef)));
  k_diag_finish3<<<1, 32, 0, s>>>(m, nb);
  return cudaGetLastError();
}

int pressure3_parts(const DevMesh3& m) { return blocks3(m.n_tet); }

cudaError_t launch_pressure3(const DevMesh3& m, double* pe, double* pf, double* part, double vol, cudaStream_t s) {
  const int nb = blocks3(m.n_tet);
  DGDF_DISPATCH_K3(m.k, (k_pressure3<K><<<nb, kTetThreads, 0, s>>>(m, pe, part)));
  const size_t n = std::max(size_t(m.n_tet) * m.nw, size_t(m.n_face) * m.nl);
  const int fb = int(std::min<size_t>((n + 255) / 256, 1024));
  k_pressure3_finish<<<fb, 256, 0, s>>>(m, pe, pf, part, nb, vol);
  return cudaGetLastError();
}

int solver3_blocks(const DevMesh3& m) {
  int nb = 0;
  switch (m.k) {
    case 1: nb = solve3_blocks_for<1>(); break;
    case 2: nb = solve3_blocks_for<2>(); break;
    default: return 0;
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (nb > 2 * sms) nb = 2 * sms;
  const int need = (m.n_face + kSolverThreads - 1) / kSolverThreads;
  if (nb > need) nb = need;
  if (nb > kMaxSolverBlocks) nb = kMaxSolverBlocks;
  return nb < 1 ? 1 : nb;
}

cudaError_t launch_solve3(const DevMesh3& m, const SolveArgs& a, int nblocks, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(m.bar, 0, sizeof(GridBar), s);
  if (e != cudaSuccess) return e;
  DevMesh3 mm = m;
  SolveArgs aa = a;
  void* args[] = {&mm, &aa};
  const void* fn = nullptr;
  switch (m.k) {
    case 1: fn = (const void*)k_solve3<1>; break;
    case 2: fn = (const void*)k_solve3<2>; break;
    default: return cudaErrorInvalidValue;
  }
  return cudaLaunchCooperativeKernel(fn, dim3(nblocks), dim3(kSolverThreads), args, 0, s);
}

}  // namespace dgdf
