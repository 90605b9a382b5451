// Facet-system solve with the multilevel preconditioner (multilevel.hpp): FP64
// PCG on S lam = g (the condensed system of eq. (12), Sec. 2.4), preconditioned
// by one V-cycle per iteration, in one persistent cooperative kernel (2-D facets
// and 3-D faces share it).
//
// Every phase is a loop over the rows of one level followed by a bounded grid
// barrier (solver_common.cuh). A V-cycle with L smoothing levels:
//   down, level l: [A] x = d + c1 d + c2 B (b - A d)  (d = c0 B b, set by the
//                  previous phase: the second Chebyshev step from x = 0)
//                  [B] r = b - A x; an injected transfer writes the next level's b
//                  (and its first Chebyshev step) in the same phase
//                  [C] a CSR transfer: b_next = R r (and its first step)
//   coarsest:      x_c = pinv b_c (added into the last level's mode 0 if it injects)
//   up, level l:   [U] a CSR transfer: x += P x_next
//                  [Q] r = b - A x, d = c0 B r
//                  [R] x += d + c1 d + c2 B (r - A d); an injected transfer adds x
//                  into the finer level's leading modes in the same phase
// A fused level (fuse_levels) takes one phase each way instead: b_next = D b and
// x = U [b; x_next].
//
// What bounds it: latency. At 128^2 (49408 facets) a phase moves one to ten MB, all from L2,
// and holds a few dependent loads; the barrier is another microsecond. So the design counts
// phases and dependent loads:
//   - one block of 1024 threads per SM: 152 barrier arrivals, 32 warps to hide the loads;
//   - a facet's modes go to 2 or 4 lanes, one output mode a lane (3-D: three): neighbours' values are
//     one vector load shared by the lanes, and a phase is a dozen instructions deep;
//   - each block owns a contiguous run of facets, whose neighbour lists stay in shared memory
//     for the whole solve, as do the operators of the stencil classes, of all (structured 2-D
//     meshes have a few) or of its own facets; otherwise the facets' own operators are read
//     transposed, coalesced;
//   - fused coarse levels: at 128^2, BDM_3, 13 phases a V-cycle instead of 27.
// Measured (walls, 128^2, BDM_3, mixed form, per solve of 14.3 iterations): 2.89 ms
// with a thread a row, 193 blocks of 256 threads and unfused levels; 1.16 ms in this form, of which
// the barriers take a third, the FP64 pass S p 13 of 74 us an iteration (7.3 of the FP64 pipes).
#include <algorithm>
#include <type_traits>
#include <vector>

#include "device.cuh"
#include "device3.cuh"
#include "kcommon.cuh"
#include "multilevel.hpp"
#include "solver_common.cuh"

namespace dgdf {

namespace {

constexpr int kMLThreads = 1024;         // most threads of a block
// Threads of a block: 1024 (64 registers) in FP32; 512 (128 registers) in FP64 and for the six modes
// of 3-D faces, whose rows of operands do not fit 64 (FP64, 48^2 BDM_2: 1.33 -> 1.26 ms a solve; FP32
// at 128^2 BDM_3: 1.26 ms with 512, 1.21 with 1024). At 64 registers the four modes of BDM_3 spill 250
// bytes, and the three of 3-D BDM_1, on seven blocks, 310: there the line could lie on either side (two
// steps with 1024 and 512: 5.38 and 4.85 ms at 8^3, 12.3 and 11.4 at 16^3, 27.3 and 27.6 at 24^3).
template <int NL, typename R>
constexpr int ml_threads() {
  return NL == 6 || std::is_same<R, double>::value ? 512 : 1024;
}
constexpr int kMLSmemMax = 200 * 1024;   // dynamic shared memory a block may ask for
constexpr int kMLIdxMax = 64 * 1024;     // of which neighbour lists
constexpr int kMLMapMax = 2 * (3 * kMLThreads + 192);   // classes a block can number (ints of the scratch)

// The system and the hierarchy as the kernel takes them.
template <typename R>
struct MLSys {
  int n;                      // facets
  int ncls;                   // operator tables: classes (0: per facet)
  int nslot;                  // of which a block holds in shared memory (ncls: all; fewer: ml_context)
  int idx_smem;               // 1: the block's neighbour lists fit in shared memory
  int nlev, nc, ld;
  int has_kernel;
  const int32_t *nbr, *cls;   // [n][NB - 1], [n]
  const double* tab64;
  const R* tab;
  const MLLevelT<R>* lv;
  const R* cpinv;
  R *xc, *bc;
  double *lam, *g, *r, *z, *pa, *q, *red;
  double* hist;
  GridBar* bar;
  DevStats* stats;
};

// ---- vector loads of one row of N values (row stride a multiple of the vector width). Vectors that
// other blocks wrote before the last barrier are read by plain loads: the barrier's acquire orders
// them, and neighbours' rows then come from L1 after their first use in a phase.
template <int N>
__device__ __forceinline__ void ld_row(const float* p, float (&v)[N]) {
  if constexpr (N == 1) {
    v[0] = p[0];
  } else if constexpr (N == 2) {
    const float2 w = *reinterpret_cast<const float2*>(p);
    v[0] = w.x, v[1] = w.y;
  } else if constexpr (N == 3 || N == 4) {
    const float4 w = *reinterpret_cast<const float4*>(p);
    v[0] = w.x, v[1] = w.y, v[2] = w.z;
    if constexpr (N == 4) v[3] = w.w;
  } else {
    static_assert(N == 6, "row of 6");
#pragma unroll
    for (int h = 0; h < 3; ++h) {
      const float2 w = reinterpret_cast<const float2*>(p)[h];
      v[2 * h] = w.x, v[2 * h + 1] = w.y;
    }
  }
}
template <int N>
__device__ __forceinline__ void ld_row(const double* p, double (&v)[N]) {
  if constexpr (N % 2 == 0) {
#pragma unroll
    for (int h = 0; h < N / 2; ++h) {
      const double2 w = reinterpret_cast<const double2*>(p)[h];
      v[2 * h] = w.x, v[2 * h + 1] = w.y;
    }
  } else {
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = p[j];
  }
}
// a row of N values of a shared-memory operator table (row stride ml_row_stride)
template <int N, typename R>
__device__ __forceinline__ void ld_tab(const R* p, R (&v)[N]) {
  if constexpr (std::is_same<R, float>::value && (N == 3 || N == 4)) {
    const float4 w = *reinterpret_cast<const float4*>(p);
    v[0] = w.x, v[1] = w.y, v[2] = w.z;
    if constexpr (N == 4) v[3] = w.w;
  } else if constexpr (std::is_same<R, float>::value && N % 2 == 0) {
#pragma unroll
    for (int h = 0; h < N / 2; ++h) {
      const float2 w = reinterpret_cast<const float2*>(p)[h];
      v[2 * h] = w.x, v[2 * h + 1] = w.y;
    }
  } else if constexpr (N % 2 == 0) {
#pragma unroll
    for (int h = 0; h < N / 2; ++h) {
      const double2 w = reinterpret_cast<const double2*>(p)[h];
      v[2 * h] = w.x, v[2 * h + 1] = w.y;
    }
  } else {
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = p[j];
  }
}

// Row stride of the vectors of a stencil level with BS values a row: FP32 rows of three are
// padded to four; FP64 level 0 shares the PCG vectors' layout.
template <typename R>
__device__ __host__ constexpr int ml_vs(int bs) {
  return std::is_same<R, float>::value && bs == 3 ? 4 : bs;
}

// Per-block context: the block's facets [f0, f1), its neighbour lists (shared or global memory,
// indexed from f0) and the operator tables (classes in shared memory, or per facet in global memory).
template <int NL, int NB, typename R>
struct MLCtx {
  static constexpr int LP = ml_lanes(NL) * ml_modes(NL), RS = ml_row_stride(NL);
  static constexpr int BLK = NB * NL * RS;                       // words of a class's blocks
  int n, f0, f1;
  bool classes;
  const int32_t *nbr, *cls;
  const double* tab64;
  const R* tab;
  const double* gtab64;        // tables of all classes in global memory
  const R* gtab;
};

// operators of the class of the block's facet fl (class tables). On faces of tetrahedra c.cls is a
// slot of the shared tables, or ~class of a class that found no slot
template <int NL, int NB, typename R, typename T>
__device__ __forceinline__ const T* ml_class_tab(const MLCtx<NL, NB, R>& c, const T* tab, int fl) {
  const int s = c.cls[fl];
  if constexpr (NB == 7) {
    if (s < 0) {
      if constexpr (std::is_same<T, R>::value) tab = c.gtab;
      else tab = c.gtab64;
      return tab + ~s * ml_class_stride(NL, NB, sizeof(T));
    }
  }
  return tab + s * ml_class_stride(NL, NB, sizeof(T));
}

// y[q] = (A x)_(i + q) of facet f on the leading BS modes, for the ml_modes(BS) modes of a lane
template <int NL, int NB, int BS, typename R, typename T>
__device__ __forceinline__ void ml_apply_row(const MLCtx<NL, NB, R>& c, const T* tab, int f, int i, const T* x, int vs,
                                             T (&y)[ml_modes(BS)]) {
  constexpr int MP = ml_modes(BS);
  const int fl = f - c.f0;
  int g[NB];
  g[0] = f;
#pragma unroll
  for (int b = 1; b < NB; ++b) g[b] = c.nbr[fl * (NB - 1) + b - 1];
  T xs[NB][BS];
#pragma unroll
  for (int b = 0; b < NB; ++b) ld_row<BS>(x + size_t(g[b]) * vs, xs[b]);
#pragma unroll
  for (int q = 0; q < MP; ++q) y[q] = T(0);
  if (c.classes) {
    const T* t = ml_class_tab<NL, NB, R, T>(c, tab, fl) + i * c.RS;
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int q = 0; q < MP; ++q) {
        T a[BS];
        ld_tab<BS>(t + (b * NL + q) * c.RS, a);
#pragma unroll
        for (int j = 0; j < BS; ++j) y[q] += a[j] * xs[b][j];
      }
  } else {
    const T* t = tab + size_t(f) * c.LP + i;
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int j = 0; j < BS; ++j)
#pragma unroll
        for (int q = 0; q < MP; ++q) y[q] += __ldg(t + size_t(b * NL + j) * c.n * c.LP + q) * xs[b][j];
  }
}

// t[q] = (B v)_(i + q) on BS modes: v is spread over the facet's lanes
template <int NL, int NB, int BS, typename R>
__device__ __forceinline__ void ml_binv_row(const MLCtx<NL, NB, R>& c, int f, int i, const R (&v)[ml_modes(BS)],
                                            R (&t)[ml_modes(BS)]) {
  constexpr int MP = ml_modes(BS), LB = ml_lanes(BS);
  if constexpr (BS == 1) {
    t[0] = c.classes ? ml_class_tab<NL, NB, R, R>(c, c.tab, f - c.f0)[c.BLK + NL * c.RS + 4] * v[0]
                     : __ldg(c.tab + size_t(c.n) * ((NB + 1) * NL * c.LP + 4) + f) * v[0];
  } else {
    R w[BS];
#pragma unroll
    for (int j = 0; j < BS; ++j) w[j] = __shfl_sync(0xffffffffu, v[j % MP], j / MP, LB);
#pragma unroll
    for (int q = 0; q < MP; ++q) {
      R a[BS];
      if (c.classes) {
        const R* o = ml_class_tab<NL, NB, R, R>(c, c.tab, f - c.f0) + c.BLK;
        if constexpr (BS == NL) ld_tab<BS>(o + (i + q) * c.RS, a);
        else ld_tab<BS>(o + NL * c.RS + (i + q) * 2, a);
      } else {
        const R* o = c.tab + size_t(c.n) * NB * NL * c.LP + (BS == NL ? 0 : size_t(c.n) * NL * c.LP);
#pragma unroll
        for (int j = 0; j < BS; ++j) a[j] = __ldg(o + (size_t(j) * c.n + f) * (LB * MP) + i + q);
      }
      t[q] = R(0);
#pragma unroll
      for (int j = 0; j < BS; ++j) t[q] += a[j] * w[j];
    }
  }
}

// Loop over the block's facets, LB lanes each, i the lane's first mode: fn(f, i, live). Lanes past
// the last facet or past the last mode (i is then clamped) run along with live = false, so that
// fn may shuffle over the warp; warps past the last facet leave (an FP64 instruction costs its 64
// cycles whether its lanes are live or not).
template <int BS, typename Ctx, typename F>
__device__ __forceinline__ void ml_facets(const Ctx& c, F&& fn) {
  constexpr int LB = ml_lanes(BS);
  const int i0 = (threadIdx.x & (LB - 1)) * ml_modes(BS), i = i0 < BS ? i0 : BS - 1;
  const int step = threadIdx.x / LB, warp0 = (threadIdx.x & ~31) / LB;
  for (int fb = c.f0; fb + warp0 < c.f1; fb += int(blockDim.x) / LB) {
    const int f = fb + step;
    fn(f < c.f1 ? f : c.f1 - 1, i, f < c.f1 && i0 < BS);
  }
}

// Rows of a CSR level in groups of G lanes of one warp, G = the largest power of two <= 32 with
// G n <= the grid's threads: the lanes of a group split a row's sum (dot(i, lane, G), a strided
// partial sum) and add their partials by shuffles, then lane 0 of the group calls f(i, sum).
template <typename R, typename Dot, typename F>
__device__ __forceinline__ void rows_grouped(int n, Dot&& dot, F&& f) {
  const int gtid = blockIdx.x * blockDim.x + threadIdx.x, gsz = gridDim.x * blockDim.x;
  int G = 1;
  while (G < 32 && 2 * G * n <= gsz) G *= 2;
  const int lane = threadIdx.x & (G - 1), grp = gtid / G, ngrp = gsz / G;
  for (int i0 = 0; i0 < n; i0 += ngrp) {
    const int i = i0 + grp;
    R s = i < n ? dot(i, lane, G) : R(0);
    for (int o = G >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (i < n && lane == 0) f(i, s);
  }
}

// Strided partial sum of a CSR row: sum over p = rp[i] + lane, + G, ... of v[p] x[ci[p]]
template <typename R>
__device__ __forceinline__ R csr_part(const int32_t* rp, const int32_t* ci, const R* v, const R* x, int i, int lane,
                                      int G) {
  R s = R(0);
  const int p1 = __ldg(&rp[i + 1]);
#pragma unroll 4
  for (int p = __ldg(&rp[i]) + lane; p < p1; p += G) s += __ldg(&v[p]) * x[__ldg(&ci[p])];
  return s;
}

// y = M x for a matrix in sliced rows (SellHost): a warp takes a slice, f(row, sum) on each row's
// first lane. Slices are dealt out to the blocks one by one: their lengths vary slowly along the
// rows, so that every block gets its share of long ones.
template <typename R, typename F>
__device__ __forceinline__ void sell_rows(int n, int G, const int32_t* __restrict__ ptr, const int32_t* __restrict__ ci,
                                          const R* __restrict__ v, const R* x, F&& f) {
  const int per = 32 / G, ns = (n + per - 1) / per, lane = threadIdx.x & 31;
  for (int s = blockIdx.x + (threadIdx.x >> 5) * gridDim.x; s < ns; s += gridDim.x * (blockDim.x / 32)) {
    const int p1 = __ldg(&ptr[s + 1]);
    R a = R(0);
#pragma unroll 8
    for (int p = __ldg(&ptr[s]); p < p1; ++p) {
      const size_t o = size_t(p) * 32 + lane;
      a += __ldg(&v[o]) * x[__ldg(&ci[o])];
    }
    for (int o = G >> 1; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    const int i = s * per + lane / G;
    if (i < n && (lane & (G - 1)) == 0) f(i, a);
  }
}

// x_c = pinv b_c, a warp per row (rows padded to ld, a multiple of four words)
template <typename R, typename F>
__device__ __forceinline__ void dense_rows(int nc, int ld, const R* __restrict__ A, const R* x, F&& f) {
  using V = typename std::conditional<std::is_same<R, float>::value, float4, double2>::type;
  constexpr int W = sizeof(V) / sizeof(R);
  const int lane = threadIdx.x & 31, nv = ld / W;
  const V* xv = reinterpret_cast<const V*>(x);
  for (int i = blockIdx.x + (threadIdx.x >> 5) * gridDim.x; i < nc; i += gridDim.x * (blockDim.x / 32)) {
    const V* row = reinterpret_cast<const V*>(A + size_t(i) * ld);
    R s = R(0);
#pragma unroll 4
    for (int j = lane; j < nv; j += 32) {
      const V a = __ldg(&row[j]), b = xv[j];
      if constexpr (W == 4) s += a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w;
      else s += a.x * b.x + a.y * b.y;
    }
    s = warp_sum(s);
    if (lane == 0) f(i, s);
  }
}

// [A] of a stencil level: second Chebyshev step from zero
template <int NL, int NB, int BS, typename R>
__device__ __forceinline__ void ml_phase_a(const MLCtx<NL, NB, R>& c, const MLLevelT<R>& L) {
  constexpr int VS = ml_vs<R>(BS), MP = ml_modes(BS);
  ml_facets<BS>(c, [&](int f, int i, bool live) {
    const size_t o = size_t(f) * VS + i;
    R y[MP], t[MP], d[MP];
    ml_apply_row<NL, NB, BS>(c, c.tab, f, i, static_cast<const R*>(L.d), VS, y);
#pragma unroll
    for (int q = 0; q < MP; ++q) {
      d[q] = L.d[o + q];
      y[q] = L.b[o + q] - y[q];
    }
    ml_binv_row<NL, NB, BS>(c, f, i, y, t);
    if (live)
#pragma unroll
      for (int q = 0; q < MP; ++q) L.x[o + q] = d[q] + L.c1 * d[q] + L.c2 * t[q];
  });
}

// [B]: residual; with an injected transfer the next level's right-hand side (bc for the coarsest)
// and, if that level is not fused, its first Chebyshev step from zero, d = c0 B b
template <int NL, int NB, int BS, typename R>
__device__ __forceinline__ void ml_phase_b(const MLCtx<NL, NB, R>& c, const MLLevelT<R>& L, const MLLevelT<R>* N, R* bc) {
  constexpr int VS = ml_vs<R>(BS), MP = ml_modes(BS);
  ml_facets<BS>(c, [&](int f, int i, bool live) {
    const size_t o = size_t(f) * VS + i;
    R r[MP];
    ml_apply_row<NL, NB, BS>(c, c.tab, f, i, static_cast<const R*>(L.x), VS, r);
#pragma unroll
    for (int q = 0; q < MP; ++q) r[q] = L.b[o + q] - r[q];
    if (!L.inject) {
      if (live)
#pragma unroll
        for (int q = 0; q < MP; ++q) L.r[o + q] = r[q];
      return;
    }
    const int bn = L.bs_next;
    R* nb = N ? N->b : bc;
#pragma unroll
    for (int q = 0; q < MP; ++q)
      if (live && i + q < bn) nb[size_t(f) * bn + i + q] = r[q];
    if (N && !N->fused) {
      if (bn == 2) {
        if constexpr (BS > 2 && MP == 1) {
          // B of the two-mode level on the lanes of modes 0 and 1 (others compute and drop)
          constexpr int LB = ml_lanes(BS);
          const int i2 = i & 1;
          R a[2];
          if (c.classes) {
            ld_tab<2>(ml_class_tab<NL, NB, R, R>(c, c.tab, f - c.f0) + c.BLK + NL * c.RS + i2 * 2, a);
          } else {
            const R* t = c.tab + size_t(c.n) * (NB + 1) * NL * c.LP;
            a[0] = __ldg(t + size_t(f) * 2 + i2);
            a[1] = __ldg(t + (size_t(c.n) + f) * 2 + i2);
          }
          const R t = a[0] * __shfl_sync(0xffffffffu, r[0], 0, LB) + a[1] * __shfl_sync(0xffffffffu, r[0], 1, LB);
          if (live && i < 2) N->d[size_t(f) * 2 + i] = N->c0 * t;
        }
      } else if (live && i == 0) {
        R t[1] = {r[0]};
        if (N->stencil) ml_binv_row<NL, NB, 1>(c, f, 0, t, t);
        else t[0] *= __ldg(&N->binv[f]);
        N->d[f] = N->c0 * t[0];
      }
    }
  });
}

// [Q] r = b - A x, d = c0 B r
template <int NL, int NB, int BS, typename R>
__device__ __forceinline__ void ml_phase_q(const MLCtx<NL, NB, R>& c, const MLLevelT<R>& L) {
  constexpr int VS = ml_vs<R>(BS), MP = ml_modes(BS);
  ml_facets<BS>(c, [&](int f, int i, bool live) {
    const size_t o = size_t(f) * VS + i;
    R r[MP], t[MP];
    ml_apply_row<NL, NB, BS>(c, c.tab, f, i, static_cast<const R*>(L.x), VS, r);
#pragma unroll
    for (int q = 0; q < MP; ++q) r[q] = L.b[o + q] - r[q];
    ml_binv_row<NL, NB, BS>(c, f, i, r, t);
    if (live)
#pragma unroll
      for (int q = 0; q < MP; ++q) {
        L.r[o + q] = r[q];
        L.d[o + q] = L.c0 * t[q];
      }
  });
}

// [R] x += d + c1 d + c2 B (r - A d): fin(f, i, x) takes the live lanes' results
template <int NL, int NB, int BS, typename R, typename F>
__device__ __forceinline__ void ml_phase_r(const MLCtx<NL, NB, R>& c, const MLLevelT<R>& L, F&& fin) {
  constexpr int VS = ml_vs<R>(BS), MP = ml_modes(BS);
  ml_facets<BS>(c, [&](int f, int i, bool live) {
    const size_t o = size_t(f) * VS + i;
    R y[MP], t[MP], x[MP];
    ml_apply_row<NL, NB, BS>(c, c.tab, f, i, static_cast<const R*>(L.d), VS, y);
#pragma unroll
    for (int q = 0; q < MP; ++q) {
      const R d = L.d[o + q];
      x[q] = L.x[o + q] + d + L.c1 * d;
      y[q] = L.r[o + q] - y[q];
    }
    ml_binv_row<NL, NB, BS>(c, f, i, y, t);
    if (live)
#pragma unroll
      for (int q = 0; q < MP; ++q) fin(f, i + q, x[q] + L.c2 * t[q]);
  });
}

// dispatch on the values per row of a stencil level: all NL modes, two, or one
#define ML_BS(bs, CALL)                                          \
  if ((bs) == NL) { constexpr int BS = NL; CALL; }               \
  else if ((bs) == 2) { constexpr int BS = 2; CALL; }            \
  else { constexpr int BS = 1; CALL; }

// One V-cycle: on entry lv[0].b holds the input (in FP64 the PCG residual r itself) and
// lv[0].d = c0 B b (set by the caller before a barrier, ml_start); on return every thread has
// written its rows of the output z (m.z; lv[0].x itself in FP64) and accumulated, over its rows,
// r.z, r.r and the sum of r's mode 0 into red[0..2], with r the PCG residual m.r. The caller's
// reduction is the closing barrier. (The mode-0 sum has a loop of its own, a facet a lane: in the
// loop over the modes its FP64 add would run at a quarter of the lanes.)
template <int NL, int NB, typename R>
__device__ bool ml_vcycle(const MLSys<R>& m, const MLCtx<NL, NB, R>& c, const MLLevelT<R>* lv, Barrier& bar,
                          double (&red)[3]) {
  const int nlev = m.nlev;
  for (int l = 0; l < nlev; ++l) {
    const MLLevelT<R>& L = lv[l];
    const bool last = l + 1 == nlev;
    const MLLevelT<R>* N = last ? nullptr : &lv[l + 1];
    if (L.fused) {
      R* out = last ? m.bc : N->b;
      sell_rows(L.n_next, L.dg, L.d_ptr, L.d_ci, L.d_v, static_cast<const R*>(L.b), [&](int i, R v) { out[i] = v; });
      if (!grid_sync(bar, m.stats)) return false;
      continue;
    }
    // [A] second Chebyshev step from zero
    if (L.stencil) {
      ML_BS(L.bs, (ml_phase_a<NL, NB, BS, R>(c, L)));
    } else {
      rows_grouped<R>(
          L.n, [&](int i, int lane, int G) { return csr_part<R>(L.a_rp, L.a_ci, L.a_v, L.d, i, lane, G); },
          [&](int i, R y) {
            const R t = __ldg(&L.binv[i]) * (L.b[i] - y);
            const R d = L.d[i];
            L.x[i] = d + L.c1 * d + L.c2 * t;
          });
    }
    if (!grid_sync(bar, m.stats)) return false;
    // [B] residual, injected restriction
    if (L.stencil) {
      ML_BS(L.bs, (ml_phase_b<NL, NB, BS, R>(c, L, N, m.bc)));
    } else {
      // CSR levels hold one value per row and transfer through R (phase [C])
      rows_grouped<R>(
          L.n, [&](int i, int lane, int G) { return csr_part<R>(L.a_rp, L.a_ci, L.a_v, L.x, i, lane, G); },
          [&](int i, R y) { L.r[i] = L.b[i] - y; });
    }
    if (!grid_sync(bar, m.stats)) return false;
    if (!L.inject) {
      // [C] CSR restriction b_next = R r
      rows_grouped<R>(
          L.n_next, [&](int j, int lane, int G) { return csr_part<R>(L.r_rp, L.r_ci, L.r_v, L.r, j, lane, G); },
          [&](int j, R v) {
            if (last) {
              m.bc[j] = v;
            } else {
              N->b[j] = v;
              if (!N->fused) N->d[j] = N->c0 * (__ldg(&N->binv[j]) * v);
            }
          });
      if (!grid_sync(bar, m.stats)) return false;
    }
  }
  // coarsest level: x_c = pinv b_c
  {
    const MLLevelT<R>& Lz = lv[nlev - 1];
    dense_rows(m.nc, m.ld, m.cpinv, static_cast<const R*>(m.bc), [&](int i, R v) {
      if (Lz.inject) Lz.x[size_t(i) * ml_vs<R>(Lz.bs)] += v;
      else m.xc[i] = v;
    });
    if (!grid_sync(bar, m.stats)) return false;
  }
  for (int l = nlev - 1; l >= 0; --l) {
    const MLLevelT<R>& L = lv[l];
    const MLLevelT<R>* F = l > 0 && lv[l - 1].inject ? &lv[l - 1] : nullptr;
    const int fvs = F ? ml_vs<R>(F->bs) : 0;
    if (L.fused) {
      // x = U [b; x_next], x_next right behind b
      sell_rows(L.n, L.ug, L.u_ptr, L.u_ci, L.u_v, static_cast<const R*>(L.b), [&](int i, R x) {
        if (F) F->x[size_t(i) * fvs] += x;
        else L.x[i] = x;
      });
      if (!grid_sync(bar, m.stats)) return false;
      continue;
    }
    if (!L.inject) {
      // [U] CSR prolongation x += P x_next
      const R* xn = (l + 1 == nlev) ? m.xc : lv[l + 1].x;
      rows_grouped<R>(
          L.n, [&](int i, int lane, int G) { return csr_part<R>(L.p_rp, L.p_ci, L.p_v, xn, i, lane, G); },
          [&](int i, R v) { L.x[i] += v; });
      if (!grid_sync(bar, m.stats)) return false;
    }
    if (!L.stencil) {
      // [Q], [R] of a CSR level
      rows_grouped<R>(
          L.n, [&](int i, int lane, int G) { return csr_part<R>(L.a_rp, L.a_ci, L.a_v, L.x, i, lane, G); },
          [&](int i, R y) {
            const R res = L.b[i] - y;
            L.r[i] = res;
            L.d[i] = L.c0 * (__ldg(&L.binv[i]) * res);
          });
      if (!grid_sync(bar, m.stats)) return false;
      rows_grouped<R>(
          L.n, [&](int i, int lane, int G) { return csr_part<R>(L.a_rp, L.a_ci, L.a_v, L.d, i, lane, G); },
          [&](int i, R y) {
            const R t = __ldg(&L.binv[i]) * (L.r[i] - y);
            const R d = L.d[i];
            const R x = L.x[i] + d + L.c1 * d + L.c2 * t;
            L.x[i] = x;
            if (F) F->x[size_t(i) * fvs] += x;   // injected into the finer level's mode 0
          });
      if (!grid_sync(bar, m.stats)) return false;
      continue;
    }
    // [Q] r = b - A x, d = c0 B r
    ML_BS(L.bs, (ml_phase_q<NL, NB, BS, R>(c, L)));
    if (!grid_sync(bar, m.stats)) return false;
    // [R]; at level 0 the output z and the PCG scalars, against the FP64 residual
    if (l == 0) {
      for (int f = c.f0 + threadIdx.x; f < c.f1; f += blockDim.x) red[2] += m.r[size_t(f) * NL];
      ml_phase_r<NL, NB, NL, R>(c, L, [&](int f, int i, R x) {
        const size_t o = size_t(f) * NL + i;
        const double z = double(x), b = m.r[o];
        m.z[o] = z;
        red[0] += b * z;
        red[1] += b * b;
      });
      return true;
    }
    ML_BS(L.bs, (ml_phase_r<NL, NB, BS, R>(c, L, [&](int f, int i, R x) {
            L.x[size_t(f) * ml_vs<R>(BS) + i] = x;
            if (F) F->x[size_t(f) * fvs + i] += x;
          })));
    if (!grid_sync(bar, m.stats)) return false;
  }
  return true;
}

// Level 0's input from the PCG residual: b = r (FP32: rounded) and its first Chebyshev step
// d = c0 B b, on the lanes of facet f, each holding its modes of r
template <int NL, int NB, typename R>
__device__ __forceinline__ void ml_start(const MLCtx<NL, NB, R>& c, const MLLevelT<R>& L0, int f, int i, bool live,
                                         const double (&r)[ml_modes(NL)]) {
  constexpr int VS = ml_vs<R>(NL), MP = ml_modes(NL);
  R b[MP], t[MP];
#pragma unroll
  for (int q = 0; q < MP; ++q) b[q] = R(r[q]);
  ml_binv_row<NL, NB, NL>(c, f, i, b, t);
  if (!live) return;
#pragma unroll
  for (int q = 0; q < MP; ++q) {
    if constexpr (!std::is_same<R, double>::value) L0.b[size_t(f) * VS + i + q] = b[q];
    L0.d[size_t(f) * VS + i + q] = L0.c0 * t[q];
  }
}

// Grid sums of N FP64 partials per thread, in a fixed order; thread 0 of every block then takes
// them to fn(sums), whose results other threads read from shared memory after the call. An FP64
// instruction occupies a quarter of an SM for 64 cycles, so a scalar step run by every warp of
// the block (a division, a square root) would cost microseconds, as would a butterfly over every
// warp: the partials go through shared memory, 64 threads a value add 16 each, one warp a value
// adds those 64 (about one add a partial).
template <int N, typename Sys, typename F>
__device__ bool ml_reduce(const Sys& m, Barrier& bar, int slot0, const double (&v)[N], double* scr, F&& fn) {
  constexpr int COLS = 64;
#pragma unroll
  for (int i = 0; i < N; ++i) scr[i * blockDim.x + threadIdx.x] = v[i];
  __syncthreads();
  double* part = scr + N * blockDim.x;
  if (threadIdx.x < N * COLS) {
    const double* p = scr + (threadIdx.x / COLS) * blockDim.x + threadIdx.x % COLS;
    double s0 = 0.0, s1 = 0.0;
    for (int k = 0; k < int(blockDim.x) / COLS; k += 2) {
      s0 += p[k * COLS];
      s1 += p[(k + 1) * COLS];
    }
    part[threadIdx.x] = s0 + s1;
  }
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w < N) {
    const double* p = part + w * COLS;
    const double s = warp_sum(p[lane] + p[lane + 32]);
    if (lane == 0) m.red[size_t(slot0 + w) * kMaxSolverBlocks + blockIdx.x] = s;
  }
  if (!grid_sync(bar, m.stats)) return false;
  if (w < N) {
    double a = 0.0;
    for (int b = lane; b < int(gridDim.x); b += 32) a += m.red[size_t(slot0 + w) * kMaxSolverBlocks + b];
    a = warp_sum(a);
    if (lane == 0) scr[w] = a;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t[N];
#pragma unroll
    for (int i = 0; i < N; ++i) t[i] = scr[i];
    fn(t);
  }
  __syncthreads();
  return true;
}

// Mode j of g at facet f: both sides' condensation output in the facet's canonical orientation
// and the boundary data (assemble_g, boundary_g in solver_common.cuh, one mode).
template <int NL>
__device__ __forceinline__ double ml_g_entry(const DevMesh& m, int f, int j, int homog) {
  double gv = 0.0;
  dfl acc(0);
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int t = __ldg(&m.facet_tri[size_t(f) * 2 + s]);
    if (t < 0) break;   // a wall has one side
    const int e = __ldg(&m.facet_loc[size_t(f) * 2 + s]);
    const bool neg = __ldg(&m.tri_orient[size_t(t) * 3 + e]) < 0 && (j & 1);
    const size_t o = size_t(t) * 3 * NL + e * NL + j;
    if (m.elem_df) {
      const dfl v = to_dfl(m.gl_df[o]);
      acc += neg ? -v : v;
    } else {
      gv += neg ? -m.gl[o] : m.gl[o];
    }
  }
  if (m.elem_df) gv = to_double(acc);
  if (m.facet_kind) {
    const int kd = __ldg(&m.facet_kind[f]);
    if (kd == kFacetOutflow) gv = 0.0;
    else if (kd == kFacetInflow && !homog) gv -= __ldg(&m.inflow_d[size_t(f) * NL + j]);
  }
  return gv;
}
// 3-D: canonical face basis, no orientation signs
template <int NL>
__device__ __forceinline__ double ml_g_entry(const DevMesh3& m, int f, int j, int) {
  const int t0 = __ldg(&m.face_tet[size_t(f) * 2]), t1 = __ldg(&m.face_tet[size_t(f) * 2 + 1]);
  const int e0 = __ldg(&m.face_loc[size_t(f) * 2]), e1 = __ldg(&m.face_loc[size_t(f) * 2 + 1]);
  return m.gl[size_t(t0) * 4 * NL + e0 * NL + j] + m.gl[size_t(t1) * 4 * NL + e1 * NL + j];
}

// Fills the block's context: operator tables and neighbour lists into shared memory. scr is the
// reductions' scratch, 3 kMLThreads + 192 doubles.
template <int NL, int NB, typename R>
__device__ void ml_context(const MLSys<R>& m, MLCtx<NL, NB, R>& c, MLLevelT<R>* lv, double*& scr) {
  extern __shared__ __align__(16) unsigned char ml_smem_raw[];
  scr = reinterpret_cast<double*>(ml_smem_raw);
  double* t64 = scr + 3 * kMLThreads + 192;
  c.n = m.n;
  const int share = (m.n + gridDim.x - 1) / gridDim.x;
  c.f0 = min(m.n, int(blockIdx.x) * share);
  c.f1 = min(m.n, c.f0 + share);
  c.classes = m.ncls > 0;
  c.tab64 = m.tab64;
  c.tab = m.tab;
  c.gtab64 = m.tab64;
  c.gtab = m.tab;
  unsigned char* next = reinterpret_cast<unsigned char*>(t64);
  // More classes than fit (faces of tetrahedra only): the block holds those of its own faces, in
  // the order of their numbers, as far as the slots go. map: class -> slot, or ~class (none left;
  // it reads the global table), in the reductions' scratch (ml_class_slots bounds ncls).
  int32_t* map = reinterpret_cast<int32_t*>(scr);
  const bool local = NB == 7 && m.nslot < m.ncls;
  if (local) {
    for (int i = threadIdx.x; i < m.ncls; i += blockDim.x) map[i] = 0;
    __syncthreads();
    for (int f = c.f0 + threadIdx.x; f < c.f1; f += blockDim.x) map[__ldg(&m.cls[f])] = 1;
    __syncthreads();
    if (threadIdx.x < 32) {
      int used = 0;
      for (int i0 = 0; i0 < m.ncls; i0 += 32) {
        const int i = i0 + threadIdx.x;
        const bool on = i < m.ncls && map[i];
        const unsigned b = __ballot_sync(0xffffffffu, on);
        const int slot = used + __popc(b & ((1u << threadIdx.x) - 1));
        if (i < m.ncls) map[i] = on && slot < m.nslot ? slot : ~i;
        used += __popc(b);
      }
    }
    __syncthreads();
  }
  if (c.classes) {
    const int w64 = m.nslot * ml_class_stride(NL, NB, 8);
    next += size_t(w64) * 8;
    auto fill = [&](auto* dst, const auto* src, int st) {
      if (!local) {
        for (int i = threadIdx.x; i < m.ncls * st; i += blockDim.x) dst[i] = __ldg(&src[i]);
      } else {
        for (int k = threadIdx.x >> 5; k < m.ncls; k += blockDim.x >> 5)
          if (map[k] >= 0)
            for (int i = threadIdx.x & 31; i < st; i += 32) dst[map[k] * st + i] = __ldg(&src[size_t(k) * st + i]);
      }
    };
    fill(t64, m.tab64, ml_class_stride(NL, NB, 8));
    c.tab64 = t64;
    if constexpr (std::is_same<R, float>::value) {
      float* t32 = reinterpret_cast<float*>(next);
      const int w32 = m.nslot * ml_class_stride(NL, NB, 4);
      fill(t32, m.tab, ml_class_stride(NL, NB, 4));
      c.tab = t32;
      next += size_t(w32) * 4;
    } else {
      c.tab = t64;
    }
  }
  c.nbr = m.nbr + size_t(c.f0) * (NB - 1);
  c.cls = m.cls + c.f0;
  if (m.idx_smem) {
    int32_t* idx = reinterpret_cast<int32_t*>(next);
    const int nf = c.f1 - c.f0;
    for (int i = threadIdx.x; i < nf * (NB - 1); i += blockDim.x) idx[i] = __ldg(&c.nbr[i]);
    for (int i = threadIdx.x; i < nf; i += blockDim.x) {
      const int k = __ldg(&c.cls[i]);
      idx[nf * (NB - 1) + i] = local ? map[k] : k;
    }
    c.nbr = idx;
    c.cls = idx + nf * (NB - 1);
  }
  for (int l = threadIdx.x; l < m.nlev; l += blockDim.x) lv[l] = m.lv[l];
  __syncthreads();
}

// Scalars of a solve: written by thread 0 of each block, identically in every block
struct MLScal {
  double c0, mean, alpha, beta;
  int zero, done;
};

// One solve: g assembled from the element sides, lam0 from the history or warm_scale * lam
// (warm_start_row), constant multiplier removed from g, then PCG with the V-cycle.
template <int NL, int NB, typename R, typename Mesh>
__global__ void __launch_bounds__((ml_threads<NL, R>()), 1) k_solve_ml(Mesh mesh, MLSys<R> m, SolveArgs a) {
  constexpr int MP = ml_modes(NL);
  __shared__ MLLevelT<R> lv[kMLMaxLevels];
  __shared__ MLScal sc;
  MLCtx<NL, NB, R> c;
  double* scr;
  ml_context<NL, NB, R>(m, c, lv, scr);
  Barrier bar(m.bar);
  double gg[2] = {0.0, 0.0};
  ml_facets<NL>(c, [&](int f, int i, bool live) {
    if (!live) return;
#pragma unroll
    for (int q = 0; q < MP; ++q) {
      const size_t o = size_t(f) * NL + i + q;
      const double gv = ml_g_entry<NL>(mesh, f, i + q, a.homog);
      m.g[o] = gv;
      gg[0] += gv * gv;
      if (i + q == 0) gg[1] += gv;
      warm_start_row<1>(m.lam, a, o);
    }
  });
  // thread 0's own (unused elsewhere): the solve's scalars
  double inv_nf = 0.0, gnorm = 0.0, stop2 = 0.0, floor2 = 0.0, rho = 0.0, rr = 0.0, best = 0.0;
  int it = 0, stall = 0;
  bool conv = false;
  if (!ml_reduce<2>(m, bar, 4, gg, scr, [&](const double (&t)[2]) {
        // with outflow facets S is definite: no constant component to remove (inv_nf = 0)
        inv_nf = m.has_kernel ? 1.0 / double(m.n) : 0.0;
        gnorm = sqrt(nonneg(t[0] - t[1] * t[1] * inv_nf));
        stop2 = (a.rtol * gnorm) * (a.rtol * gnorm);
        floor2 = (a.floor_rtol * gnorm) * (a.floor_rtol * gnorm);
        sc.c0 = t[1] * inv_nf;
        sc.zero = !(gnorm > 0.0);   // no data, or a NaN (a state that holds one): zero
      }))
    return;
  if (sc.zero) {
    ml_facets<NL>(c, [&](int f, int i, bool live) {
      if (live)
#pragma unroll
        for (int q = 0; q < MP; ++q) m.lam[size_t(f) * NL + i + q] = 0.0;
    });
    conv = true;
  } else {
    // The V-cycle, unlike S, does not annihilate the constant multiplier (mode 0 = 1 on every
    // facet, the kernel of S), and it amplifies that direction by about 1 / lambda_min(S):
    // rounding that leaves a constant component in r would soon dominate z. So r is kept in the
    // range of S: the mode-0 mean that it had at the last V-cycle is subtracted in the next
    // update (S p has none but its rounding, some 1e-16 of r).
    // r = (g - c0 1) - S lam, its mode-0 sum and square
    double r0s[2] = {0.0, 0.0};
    const double c0 = sc.c0;
    ml_facets<NL>(c, [&](int f, int i, bool live) {
      double y[MP];
      ml_apply_row<NL, NB, NL>(c, c.tab64, f, i, static_cast<const double*>(m.lam), NL, y);
      if (!live) return;
#pragma unroll
      for (int q = 0; q < MP; ++q) {
        const size_t o = size_t(f) * NL + i + q;
        const double r = (i + q == 0 ? m.g[o] - c0 : m.g[o]) - y[q];
        m.r[o] = r;
        if (i + q == 0) r0s[0] += r;
        r0s[1] += r * r;
      }
    });
    if (!ml_reduce<2>(m, bar, 0, r0s, scr, [&](const double (&t)[2]) {
          sc.done = drop_start(a, nonneg(t[1] - t[0] * t[0] * inv_nf), gnorm);
          sc.mean = sc.done ? 0.0 : t[0] * inv_nf;
        }))
      return;
    if (sc.done)
      ml_facets<NL>(c, [&](int f, int i, bool live) {
        if (live)
#pragma unroll
          for (int q = 0; q < MP; ++q) {
            const size_t o = size_t(f) * NL + i + q;
            m.lam[o] = 0.0;
            m.r[o] = i + q == 0 ? m.g[o] - c0 : m.g[o];
          }
      });
    // remove the constant component; first Chebyshev step of the V-cycle on r
    const double mean0 = sc.mean;
    ml_facets<NL>(c, [&](int f, int i, bool live) {
      const size_t o = size_t(f) * NL + i;
      double r[MP];
#pragma unroll
      for (int q = 0; q < MP; ++q) r[q] = m.r[o + q];
      if (i == 0) r[0] -= mean0;
      if (live && i == 0) m.r[o] = r[0];
      ml_start<NL, NB, R>(c, lv[0], f, i, live, r);
    });
    if (!grid_sync(bar, m.stats)) return;
    for (bool first = true;; first = false) {
      double red[3] = {0.0, 0.0, 0.0};
      if (!ml_vcycle<NL, NB, R>(m, c, lv, bar, red)) return;
      if (!ml_reduce<3>(m, bar, 1, red, scr, [&](const double (&t)[3]) {
            rr = nonneg(t[1] - t[2] * t[2] * inv_nf);
            sc.beta = first ? 0.0 : t[0] / rho;
            rho = t[0];
            sc.mean = t[2] * inv_nf;   // mode-0 mean of r as the V-cycle saw it
            if (first) best = rr;
            else ++it;
            // rounding floor: once 10 iterations in a row fail to halve the best residual, the
            // solve ends, converged if that residual is below floor_rtol (as in the other solvers)
            int done = 1;
            if (!isfinite(rr) || !isfinite(rho)) {
              if (blockIdx.x == 0) atomicOr(&m.stats->flags, kFlagNonFinite);
            } else if (rr <= stop2) {
              conv = true;
            } else if (!(rr < 0.25 * best) && ++stall >= 10) {
              conv = best <= floor2;
            } else if (it < a.maxit) {
              if (rr < 0.25 * best) {
                best = rr;
                stall = 0;
              }
              done = 0;
            }
            sc.done = done;
          }))
        return;
      if (sc.done) break;
      // p = z + beta p, q = S p = S z + beta q (each facet's own entries; no p of a neighbour is
      // needed, which halves the FP64 work of the pass); reduce p.q
      const double beta = sc.beta, cmean = sc.mean;
      double pq[1] = {0.0};
      ml_facets<NL>(c, [&](int f, int i, bool live) {
        double y[MP];
        ml_apply_row<NL, NB, NL>(c, c.tab64, f, i, static_cast<const double*>(m.z), NL, y);
        if (!live) return;
#pragma unroll
        for (int q = 0; q < MP; ++q) {
          const size_t o = size_t(f) * NL + i + q;
          double p = m.z[o];
          if (!first) {
            p += beta * m.pa[o];
            y[q] += beta * m.q[o];
          }
          m.pa[o] = p;
          m.q[o] = y[q];
          pq[0] += p * y[q];
        }
      });
      if (!ml_reduce<1>(m, bar, 6, pq, scr, [&](const double (&t)[1]) {
            const bool down = !(t[0] > 0.0);
            const double alpha = down ? -1.0 : rho / t[0];
            if (m.hist && blockIdx.x == 0 && it < kMLHist) {
              m.hist[4 * it + 0] = sqrt(rr) / gnorm;
              m.hist[4 * it + 1] = rho;
              m.hist[4 * it + 2] = t[0];
              m.hist[4 * it + 3] = alpha;
            }
            if (down && !isfinite(t[0]) && blockIdx.x == 0) atomicOr(&m.stats->flags, kFlagNonFinite);
            sc.alpha = alpha;
            sc.done = down;
          }))
        return;
      if (sc.done) break;
      // lam += alpha p, r -= alpha q and its last mean, first Chebyshev step on r
      const double alpha = sc.alpha;
      ml_facets<NL>(c, [&](int f, int i, bool live) {
        const size_t o = size_t(f) * NL + i;
        double r[MP];
#pragma unroll
        for (int q = 0; q < MP; ++q) r[q] = m.r[o + q] - alpha * m.q[o + q];
        if (i == 0) r[0] -= cmean;
        if (live)
#pragma unroll
          for (int q = 0; q < MP; ++q) {
            m.lam[o + q] += alpha * m.pa[o + q];
            m.r[o + q] = r[q];
          }
        ml_start<NL, NB, R>(c, lv[0], f, i, live, r);
      });
      if (!grid_sync(bar, m.stats)) return;
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

// One V-cycle z = M r on its own (test hook dg_test_multilevel_apply): r and z are facet-major
// [n_facet][k+1] in device memory. Uses the solver's level-0 vectors m.r and m.z.
template <int NL, int NB, typename R>
__global__ void __launch_bounds__((ml_threads<NL, R>()), 1) k_ml_apply(MLSys<R> m, const double* rin, double* zout) {
  __shared__ MLLevelT<R> lv[kMLMaxLevels];
  MLCtx<NL, NB, R> c;
  double* scr;
  ml_context<NL, NB, R>(m, c, lv, scr);
  Barrier bar(m.bar);
  ml_facets<NL>(c, [&](int f, int i, bool live) {
    const size_t o = size_t(f) * NL + i;
    double r[ml_modes(NL)];
#pragma unroll
    for (int q = 0; q < ml_modes(NL); ++q) {
      r[q] = rin[o + q];
      if (live) m.r[o + q] = r[q];
    }
    ml_start<NL, NB, R>(c, lv[0], f, i, live, r);
  });
  if (!grid_sync(bar, m.stats)) return;
  double red[3] = {0.0, 0.0, 0.0};
  if (!ml_vcycle<NL, NB, R>(m, c, lv, bar, red)) return;
  ml_facets<NL>(c, [&](int f, int i, bool live) {
    if (live)
#pragma unroll
      for (int q = 0; q < ml_modes(NL); ++q) zout[size_t(f) * NL + i + q] = m.z[size_t(f) * NL + i + q];
  });
}

// ---- launch

// shared memory of a block: reduction scratch, operator tables, neighbour lists (if they fit)
size_t ml_smem(int nl, int nb, bool fp32, int ncls, int n, int nblocks, int* idx) {
  size_t s = size_t(3 * kMLThreads + 192) * 8;
  if (ncls > 0) s += size_t(ncls) * (ml_class_stride(nl, nb, 8) * 8 + (fp32 ? ml_class_stride(nl, nb, 4) * 4 : 0));
  const size_t i = size_t((n + nblocks - 1) / nblocks) * nb * sizeof(int32_t);
  *idx = i <= size_t(kMLIdxMax);
  return s + (*idx ? i : 0);
}

template <typename R>
MLSys<R> ml_system(const DevMesh& v) {
  MLSys<R> s{};
  s.ncls = v.ml_ncls;
  s.nslot = v.ml_ncls;
  s.nlev = v.ml_nlev;
  s.nc = v.ml_nc;
  s.ld = v.ml_ld;
  s.tab64 = v.ml_tab;
  s.r = v.r;
  s.z = v.z;
  s.red = v.red;
  s.bar = v.bar;
  s.stats = v.stats;
  s.hist = v.ml_hist;
  if constexpr (std::is_same<R, float>::value) {
    s.tab = v.ml_tab_f;
    s.lv = v.ml_lv_f;
    s.cpinv = v.ml_cpinv_f;
    s.xc = v.ml_xc_f;
    s.bc = v.ml_bc_f;
  } else {
    s.tab = v.ml_tab;
    s.lv = v.ml_lv;
    s.cpinv = v.ml_cpinv;
    s.xc = v.ml_xc;
    s.bc = v.ml_bc;
  }
  return s;
}

template <typename R>
MLSys<R> ml_system(const DevMesh& m, const DevMesh&) {
  MLSys<R> s = ml_system<R>(m);
  s.n = m.n_facet;
  s.nbr = m.facet_nbr;
  s.cls = m.facet_stencil;
  s.has_kernel = m.has_kernel;
  s.lam = m.lam;
  s.g = m.g;
  s.pa = m.pa;
  s.q = m.q;
  return s;
}
template <typename R>
MLSys<R> ml_system(const DevMesh3& m, const DevMesh& v) {
  MLSys<R> s = ml_system<R>(v);
  s.n = m.n_face;
  s.nslot = m.ml_nslot;
  s.nbr = m.face_nbr;
  s.cls = m.face_stencil;
  s.has_kernel = 1;   // closed mesh: the constant multiplier is the kernel of S
  s.lam = m.lam;
  s.g = m.g;
  s.pa = m.pa;
  s.q = m.q;
  return s;
}

// Blocks of the solver's grid: one per SM, fewer on meshes that would leave a block less than
// two warps of facet lanes.
int ml_want_blocks(int nl, int n, int sms) {
  const int want = (n * ml_lanes(nl) + 63) / 64;
  return want < 1 ? 1 : (want < sms ? want : sms);
}

// The grid's blocks. Also lets the kernel use its shared memory. 0: it does not fit.
int ml_blocks(const void* fn, int threads, int nl, int nb, bool fp32, int ncls, int n, int* fit = nullptr) {
  int dev = 0, sms = 0, per_sm = 0, idx = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int blocks = ml_want_blocks(nl, n, sms);
  const size_t smem = ml_smem(nl, nb, fp32, ncls, n, blocks, &idx);
  if (!fn || cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMLSmemMax) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    return 0;
  }
  if (fit) *fit = sms;
  return blocks;
}

template <int NL, int NB, typename R, typename Mesh>
cudaError_t ml_launch(const Mesh& mesh, const DevMesh& v, const SolveArgs& a, int nblocks, cudaStream_t s) {
  MLSys<R> sys = ml_system<R>(mesh, v);
  const size_t smem = ml_smem(NL, NB, std::is_same<R, float>::value, sys.nslot, sys.n, nblocks, &sys.idx_smem);
  if (sys.nlev < 1 || sys.nlev > kMLMaxLevels || smem > size_t(kMLSmemMax)) return cudaErrorInvalidValue;
  // a block's own classes are numbered in its neighbour lists' shared memory
  if (sys.nslot < sys.ncls && (NB != 7 || !sys.idx_smem || sys.ncls > kMLMapMax)) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(sys.bar, 0, sizeof(GridBar), s);
  if (e != cudaSuccess) return e;
  Mesh mm = mesh;
  SolveArgs aa = a;
  void* args[] = {&mm, &sys, &aa};
  return cudaLaunchCooperativeKernel((const void*)k_solve_ml<NL, NB, R, Mesh>, dim3(nblocks),
                                     dim3(ml_threads<NL, R>()), args, smem, s);
}

template <int NL, typename R>
cudaError_t ml_launch_apply(const DevMesh& v, const double* r, double* z, int nblocks, cudaStream_t s) {
  MLSys<R> sys = ml_system<R>(v, v);
  const size_t smem = ml_smem(NL, 5, std::is_same<R, float>::value, sys.nslot, sys.n, nblocks, &sys.idx_smem);
  if (sys.nlev < 1 || sys.nlev > kMLMaxLevels || smem > size_t(kMLSmemMax)) return cudaErrorInvalidValue;
  const void* fn = (const void*)k_ml_apply<NL, 5, R>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMLSmemMax);
  if (e == cudaSuccess) e = cudaMemsetAsync(sys.bar, 0, sizeof(GridBar), s);
  if (e != cudaSuccess) return e;
  void* args[] = {&sys, (void*)&r, (void*)&z};
  return cudaLaunchCooperativeKernel(fn, dim3(nblocks), dim3(ml_threads<NL, R>()), args, smem, s);
}

}  // namespace

// The class tables of both precisions have to fit beside the scratch and the neighbour lists.
bool ml_class_tables_fit(int nl, int nb, bool fp32, int ncls) {
  int idx = 0;
  return ml_smem(nl, nb, fp32, ncls, 1, 1, &idx) + kMLIdxMax <= size_t(kMLSmemMax);
}

// Blocks' own class tables, where the tables of all classes don't fit. A periodic Kuhn cube has 120
// classes (the wrapped vertex ids order 48 kinds of tetrahedra), 437 KB at k = 2, but a block of
// 324 faces meets 12 to 60 of them, and some 45 fit. With a table per face a V-cycle and the product
// with S streamed 340 MB from HBM each iteration (ncu): 140 us, with the slots 110 (16^3, k = 2;
// 15.9 -> 13.3 ms a step).
// Slots a block, or 0 where this does not pay: where more than a quarter of some block's faces would
// have to read the global table, scattered over its lanes, the tables per face are read coalesced.
int ml_class_slots(int nl, int nb, bool fp32, int ncls, int n, const int32_t* cls) {
  int dev = 0, sms = 152, idx = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int blocks = ml_want_blocks(nl, n, sms), share = (n + blocks - 1) / blocks;
  const size_t none = ml_smem(nl, nb, fp32, 0, n, blocks, &idx), one = ml_smem(nl, nb, fp32, 1, n, blocks, &idx) - none;
  if (!idx || ncls > kMLMapMax || none + one > size_t(kMLSmemMax)) return 0;
  const int fit = int((size_t(kMLSmemMax) - none) / one);
  int most = 0;
  std::vector<int32_t> own;
  for (int f0 = 0; f0 < n; f0 += share) {
    own.assign(cls + f0, cls + std::min(n, f0 + share));
    std::sort(own.begin(), own.end());
    int used = 0, over = 0;
    for (size_t i = 0; i < own.size(); ++i) {
      used += i == 0 || own[i] != own[i - 1];
      over += used > fit;
    }
    if (over * 4 > int(own.size())) return 0;
    most = std::max(most, std::min(used, fit));
  }
  return most;
}

int ml_grid_threads() {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms * kMLThreads;
}

#define ML_K2(k, fp32, CALL)                                                                     \
  switch ((k) * 2 + ((fp32) ? 1 : 0)) {                                                          \
    case 2: { constexpr int NL = 2; using R = double; CALL; }                                    \
    case 3: { constexpr int NL = 2; using R = float; CALL; }                                     \
    case 4: { constexpr int NL = 3; using R = double; CALL; }                                    \
    case 5: { constexpr int NL = 3; using R = float; CALL; }                                     \
    case 6: { constexpr int NL = 4; using R = double; CALL; }                                    \
    case 7: { constexpr int NL = 4; using R = float; CALL; }                                     \
  }

cudaError_t launch_ml_apply(const DevMesh& m, const double* r, double* z, int nblocks, cudaStream_t s) {
  ML_K2(m.k, m.ml_lv_f != nullptr, return (ml_launch_apply<NL, R>(m, r, z, nblocks, s)));
  return cudaErrorInvalidValue;
}

int solver_ml_blocks(const DevMesh& m, int* fit) {
  const bool fp32 = m.ml_lv_f != nullptr;
  ML_K2(m.k, fp32, return ml_blocks((const void*)k_solve_ml<NL, 5, R, DevMesh>, ml_threads<NL, R>(), NL, 5, fp32,
                                m.ml_ncls, m.n_facet, fit));
  return 0;
}

cudaError_t launch_solve_ml(const DevMesh& m, const SolveArgs& a, int nblocks, cudaStream_t s) {
  ML_K2(m.k, m.ml_lv_f != nullptr, return (ml_launch<NL, 5, R>(m, m, a, nblocks, s)));
  return cudaErrorInvalidValue;
}

// the three-dimensional path runs its V-cycle in FP32
int solver3_ml_blocks(const DevMesh3& m, const DevMesh& mv) {
  if (m.k == 1) return ml_blocks((const void*)k_solve_ml<3, 7, float, DevMesh3>, ml_threads<3, float>(), 3, 7, true, m.ml_nslot, m.n_face);
  if (m.k == 2) return ml_blocks((const void*)k_solve_ml<6, 7, float, DevMesh3>, ml_threads<6, float>(), 6, 7, true, m.ml_nslot, m.n_face);
  return 0;
}

cudaError_t launch_solve3_ml(const DevMesh3& m, const DevMesh& mv, const SolveArgs& a, int nblocks, cudaStream_t s) {
  if (m.k == 1) return ml_launch<3, 7, float>(m, mv, a, nblocks, s);
  if (m.k == 2) return ml_launch<6, 7, float>(m, mv, a, nblocks, s);
  return cudaErrorInvalidValue;
}

}  // namespace dgdf
