// Device records of a multilevel hierarchy (MLHost) for the solver kernel, shared by the two- and
// three-dimensional meshes.
#pragma once

#include <type_traits>
#include <vector>

#include "device.cuh"
#include "multilevel.hpp"

namespace dgdf {

// Uploads the hierarchy's operators in the precision R and allocates its vectors: up(&ptr, vector)
// copies a host vector to the device, al(&ptr, n) allocates n zeroed values; both return a status.
// In FP64 level 0 works on the PCG vectors r and z; in FP32 it has vectors of its own (rows of three
// padded to four). A fused level's right-hand side is followed in memory by the next level's
// solution. The pseudo-inverse's rows and its right-hand side are padded to ld, a multiple of four.
template <typename R, typename Up, typename Al>
int ml_fill(const MLHost& ml, std::vector<MLLevelT<R>>& lv, Up up, Al al, double* r, double* z, const R** cpinv, R** xc,
            R** bc, int* ld) {
  constexpr bool f64 = std::is_same<R, double>::value;
  auto conv = [](const std::vector<double>& v) { return std::vector<R>(v.begin(), v.end()); };
  lv.assign(ml.lv.size(), MLLevelT<R>{});
  int rc = 0;
  R* behind = nullptr;   // the solution slot behind the previous (fused) level's right-hand side
  for (size_t l = 0; l < ml.lv.size(); ++l) {
    const MLHostLevel& H = ml.lv[l];
    MLLevelT<R>& L = lv[l];
    L.stencil = H.stencil ? 1 : 0;
    L.bs = H.bs;
    L.n = H.n;
    L.inject = H.inject ? 1 : 0;
    L.n_next = H.n_next;
    L.bs_next = H.bs_next;
    L.c0 = R(H.cheb[0]);
    L.c1 = R(H.cheb[1]);
    L.c2 = R(H.cheb[2]);
    L.fused = H.fused ? 1 : 0;
    const size_t nv = size_t(H.n) * (!f64 && H.bs == 3 ? 4 : H.bs);
    if (f64 && l == 0) {
      L.b = reinterpret_cast<R*>(r);
      L.x = reinterpret_cast<R*>(z);
    }
    if (behind) L.x = behind;
    behind = nullptr;
    if (!L.x && (rc = al(&L.x, nv))) return rc;
    if (!L.b && (rc = al(&L.b, nv + (H.fused ? H.n_next : 0)))) return rc;
    if (H.fused) {
      L.dg = H.D.G;
      L.ug = H.U.G;
      if ((rc = up(&L.d_ptr, H.D.ptr)) || (rc = up(&L.d_ci, H.D.ci)) || (rc = up(&L.d_v, conv(H.D.v))) ||
          (rc = up(&L.u_ptr, H.U.ptr)) || (rc = up(&L.u_ci, H.U.ci)) || (rc = up(&L.u_v, conv(H.U.v))))
        return rc;
      behind = L.b + H.n;
      continue;
    }
    if ((rc = al(&L.r, nv)) || (rc = al(&L.d, nv))) return rc;
    if (!H.stencil && ((rc = up(&L.binv, conv(H.binv))) || (rc = up(&L.a_rp, H.A.rp)) || (rc = up(&L.a_ci, H.A.ci)) ||
                       (rc = up(&L.a_v, conv(H.A.v)))))
      return rc;
    if (!H.inject && ((rc = up(&L.p_rp, H.P.rp)) || (rc = up(&L.p_ci, H.P.ci)) || (rc = up(&L.p_v, conv(H.P.v))) ||
                      (rc = up(&L.r_rp, H.R.rp)) || (rc = up(&L.r_ci, H.R.ci)) || (rc = up(&L.r_v, conv(H.R.v)))))
      return rc;
  }
  *ld = (ml.nc + 3) / 4 * 4;
  std::vector<R> A(size_t(ml.nc) * *ld, R(0));
  for (int i = 0; i < ml.nc; ++i)
    for (int j = 0; j < ml.nc; ++j) A[size_t(i) * *ld + j] = R(ml.cpinv[size_t(i) * ml.nc + j]);
  if ((rc = up(cpinv, A)) || (rc = al(bc, size_t(*ld)))) return rc;
  *xc = behind;
  return behind ? 0 : al(xc, size_t(ml.nc));
}

}  // namespace dgdf
