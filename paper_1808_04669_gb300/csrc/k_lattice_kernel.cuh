// Facet-system solve on translation-invariant split-square meshes (the lattice
// path of the condensed hybrid-mixed system, eq. (12) of Sec. 2.4).
//
// On such a mesh the facet operator S is block circulant over the N x N cell
// grid: a 2-D discrete Fourier transform turns it into one Hermitian block
// S^(kappa) of size C = 3(k+1) per wavenumber, and S^+ r = IDFT(S^(kappa)^+ DFT(r))
// (pseudo-inverse at kappa = 0, the constant multiplier). The Fourier-space inverse B is S^+ up
// to rounding, so the solve is iterative refinement:
//   z = B r,  lam += z,  r -= S z   until |r| <= rtol |g|.
//   FP64 form : FP64 vectors, FP64 products, FP64 transforms (one iteration);
//   mixed form: double-float vectors and products on the FP32 units, FP32 transforms (two or
//               three iterations: each gains the FP32 rounding times cond(S), 1e4 at N = 256).
// Where an iteration gains less than a factor of ten, the solve goes on as PCG preconditioned by B
// (lat_pcg), which needs two more vectors, their traffic, two more reductions an iteration and a
// last row pass for nothing. The solve is bound by latency (16 warps an SM between grid barriers):
// 9 grid-wide phases at 2 iterations. N = 256, BDM_3, mixed form: 244 us as PCG with a thread a
// facet, 170 us now; FP64 form at N = 128: 222 -> 157 us; N = 8, BDM_2, FP64: 98 -> 55 us.
// The residual is real, so only the wavenumbers ki in [0, N/2] are transformed:
//   rows   : two facet rows j, j+1 packed as one complex row, FFT along i, split
//            into the two half spectra (Hermitian symmetry)
//   columns: per ki, FFT along j, multiply by S^(kappa)^+ (FP32: its near-singular
//            eigen-direction applied on its own plus the packed Hermitian remainder, so
//            FP32 rounding causes no cancellation), inverse FFT along j
//   rows   : inverse FFT along i of two rows packed the same way (scaled 1/N^2)
// with a grid barrier between the passes. Transforms run in shared memory: for N a
// power of two up to 1024 (FP32) / 256 (FP64) a two-pass FFT whose radix-sqrt(N)
// DFTs run in registers, self-sorting (Stockham) radix-2 passes for larger powers of
// two, a direct DFT otherwise. One persistent cooperative kernel per solve, two blocks
// per SM.
#pragma once

#include "device.cuh"
#include "dfloat.cuh"
#include "kcommon.cuh"
#include "solver_common.cuh"

namespace dgdf {
namespace {

constexpr int kLatThreads = 256;
constexpr int kLatTJ = 4;          // facet rows j per row-pass tile (two packed pairs)

template <bool MIXED>
struct LatT;
template <>
struct LatT<false> {   // FP64 form
  using R = double;
  using C2 = double2;
  using V = double;     // vector storage (lam, g, r, p, q)
  using A = double;     // arithmetic on vector values
  using Z = double;     // preconditioned residual z
  using Acc = double;
};
template <>
struct LatT<true> {    // mixed form
  using R = float;
  using C2 = float2;
  using V = float2;
  using A = dfl;
  using Z = float;
  using Acc = dacc;
};

// ---- typed vector access and accumulation
__device__ __forceinline__ double ldv(const double* p) { return __ldcg(p); }
__device__ __forceinline__ dfl ldv(const float2* p) { return to_dfl(__ldcg(p)); }
__device__ __forceinline__ double ldz(const double* p) { return __ldcg(p); }
__device__ __forceinline__ float ldz(const float* p) { return __ldcg(p); }
__device__ __forceinline__ void stv(double* p, double v) { *p = v; }
__device__ __forceinline__ void stv(float2* p, dfl v) { *p = to_float2(v); }
__device__ __forceinline__ void mad(double& a, double x, double y) { a = fma(x, y, a); }
__device__ __forceinline__ void acc_add(double& a, double v) { a += v; }
__device__ __forceinline__ void acc_add(dacc& a, dfl v) {
  float s, t;
  two_sum(a.s, v.hi, s, t);
  a.s = s;
  a.c += t + v.lo;
}
__device__ __forceinline__ double acc_zero(double) { return 0.0; }
__device__ __forceinline__ dacc acc_zero(dacc) { return dacc_zero(); }
__device__ __forceinline__ double acc_val(double a) { return a; }
__device__ __forceinline__ double acc_val(const dacc& a) { return double(a.s) + double(a.c); }
__device__ __forceinline__ double fin(double a) { return a; }
__device__ __forceinline__ dfl fin(const dacc& a) { return val(a); }
__device__ __forceinline__ double fft_in(double v) { return v; }
__device__ __forceinline__ float fft_in(dfl v) { return v.hi; }
__device__ __forceinline__ double as_a(double v) { return v; }
__device__ __forceinline__ double lead_d(double v) { return v; }
__device__ __forceinline__ double lead_d(dfl v) { return double(v.hi); }
__device__ __forceinline__ dfl as_a(float v) { return dfl(v, 0.f); }
__device__ __forceinline__ double stencil_entry(const DevMesh& m, size_t i, double) { return __ldg(&m.st_blk[i]); }
__device__ __forceinline__ dfl stencil_entry(const DevMesh& m, size_t i, dfl) { return to_dfl(__ldg(&m.st_blk_df[i])); }

template <typename C2>
__device__ __forceinline__ C2 cmul(C2 a, C2 b) {
  return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename C2>
__device__ __forceinline__ C2 cadd(C2 a, C2 b) {
  return {a.x + b.x, a.y + b.y};
}
template <typename C2>
__device__ __forceinline__ C2 csub(C2 a, C2 b) {
  return {a.x - b.x, a.y - b.y};
}
// a += h b
template <typename C2>
__device__ __forceinline__ void cmad(C2& a, C2 h, C2 b) {
  a.x += h.x * b.x - h.y * b.y;
  a.y += h.x * b.y + h.y * b.x;
}
// a += conj(h) b
template <typename C2>
__device__ __forceinline__ void cmad_conj(C2& a, C2 h, C2 b) {
  a.x += h.x * b.x + h.y * b.y;
  a.y += h.x * b.y - h.y * b.x;
}

// Self-sorting (Stockham) radix-2 FFT of `rows` rows of length n = 2^logn, natural
// order in and out, ping-ponging between a and b; returns the buffer holding the
// result. Stage s combines pairs (j, j + n/2) of the input into outputs
// (j / l) 2l + j % l and that + l, l = 2^s, with twiddle exp(-+2 pi i (j % l) / (2l)).
// tw[t] = exp(-2 pi i t / n).
template <typename C2>
__device__ C2* fft_stockham(C2* a, C2* b, int rows, int logn, const C2* tw, bool inverse) {
  const int n = 1 << logn, hn = n >> 1;
  for (int s = 0; s < logn; ++s) {
    const int l = 1 << s;
#pragma unroll 4
    for (int e = threadIdx.x; e < rows * hn; e += blockDim.x) {
      const int row = e >> (logn - 1), j = e & (hn - 1);
      const C2* x = a + row * n;
      C2* y = b + row * n;
      const int k = j & (l - 1);
      C2 w = tw[k << (logn - 1 - s)];
      if (inverse) w.y = -w.y;
      const C2 c0 = x[j], c1 = cmul(x[j + hn], w);
      const int d = ((j - k) << 1) + k;
      y[d] = cadd(c0, c1);
      y[d + l] = csub(c0, c1);
    }
    __syncthreads();
    C2* t = a;
    a = b;
    b = t;
  }
  return a;
}

// In-register DFT of size R (a power of two), natural order in and out: radix-2
// decimation in frequency with twiddles w^j = tw[j tstep] (w = exp(-+2 pi i / R)),
// then the bit-reversal permutation of the registers (resolved at compile time).
template <int R, typename C2>
__device__ __forceinline__ void reg_dft(C2 (&v)[R], const C2* tw, int tstep, bool inverse) {
#pragma unroll
  for (int half = R / 2; half >= 1; half >>= 1) {
#pragma unroll
    for (int blk = 0; blk < R; blk += 2 * half) {
#pragma unroll
      for (int j = 0; j < half; ++j) {
        const C2 a = v[blk + j], b = v[blk + j + half];
        v[blk + j] = cadd(a, b);
        const C2 d = csub(a, b);
        if (j == 0) {
          v[blk + j + half] = d;
        } else {
          C2 w = tw[j * (R / (2 * half)) * tstep];
          if (inverse) w.y = -w.y;
          v[blk + j + half] = cmul(d, w);
        }
      }
    }
  }
  C2 t[R];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    int b = 0;
#pragma unroll
    for (int q = 1; q < R; q <<= 1) b = (b << 1) | ((i / q) & 1);
    t[i] = v[b];
  }
#pragma unroll
  for (int i = 0; i < R; ++i) v[i] = t[i];
}

// Two-pass ("four-step") FFT of `rows` rows of length N = R1 R2 held in a (natural
// order, in place), through the scratch s (rows of stride R2 (R1 + 1), padded against
// bank conflicts): x[n1 + R1 n2] -> DFT over n2 (thread per (row, n1)) -> twiddle
// w_N^(n1 k2) -> DFT over n1 (thread per (row, k2)) -> X[k2 + R2 k1].
template <int R1, int R2, typename C2>
__device__ void fft_four_step(C2* a, C2* s, int rows, const C2* tw, bool inverse) {
  constexpr int N = R1 * R2, SR = R2 * (R1 + 1);
  for (int t = threadIdx.x; t < rows * R1; t += blockDim.x) {
    const int row = t / R1, n1 = t - row * R1;
    C2 v[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) v[n2] = a[row * N + n1 + R1 * n2];
    reg_dft<R2>(v, tw, R1, inverse);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) {
      C2 w = tw[n1 * k2];
      if (inverse) w.y = -w.y;
      s[row * SR + k2 * (R1 + 1) + n1] = k2 == 0 ? v[k2] : cmul(v[k2], w);
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < rows * R2; t += blockDim.x) {
    const int row = t / R2, k2 = t - row * R2;
    C2 v[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) v[n1] = s[row * SR + k2 * (R1 + 1) + n1];
    reg_dft<R1>(v, tw, R2, inverse);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) a[row * N + k2 + R2 * k1] = v[k1];
  }
  __syncthreads();
}

// Largest log2 N handled by the two-pass FFT (register budget of one radix-R pass).
template <typename C2>
struct FourStepMax;
template <>
struct FourStepMax<float2> {
  static constexpr int logn = 10;
};
template <>
struct FourStepMax<double2> {
  static constexpr int logn = 8;
};

// DFT of `rows` rows of any length N = R1 R2 held in a (natural order, in place) through the scratch
// s, as fft_four_step with direct sums in both passes: N (R1 + R2) multiply-adds a row instead of
// the N^2 of one sum (R1 = 1, a prime N). A thread forms kDftOut outputs at once, so that an input
// read from shared memory serves as many sums. tw[t] = exp(-2 pi i t / N), conjugated for the
// inverse. (N = 150, BDM_3, mixed form, 3.5 iterations: with this and the refinement a solve fell
// from 563 to 199 us; at the prime 127 only the shared inputs help.)
constexpr int kDftOut = 4;
template <typename C2>
__device__ void dft_two_factor(C2* a, C2* s, int rows, int N, int R1, const C2* tw, bool inverse) {
  const int R2 = N / R1;
  // out[j0 + u] = sum_t in[t is] w^(t step (j0 + u)), u < kDftOut (outputs past `n` are dropped)
  auto sums = [&](const C2* in, int is, int n, int step, int j0, C2 (&acc)[kDftOut]) {
    int idx[kDftOut], inc[kDftOut];
#pragma unroll
    for (int u = 0; u < kDftOut; ++u) {
      acc[u] = C2{0, 0};
      idx[u] = 0;
      inc[u] = j0 + u < n ? (j0 + u) * step : 0;   // < N
    }
    for (int t = 0; t < n; ++t) {
      const C2 x = in[t * is];
#pragma unroll
      for (int u = 0; u < kDftOut; ++u) {
        C2 w = tw[idx[u]];
        if (inverse) w.y = -w.y;
        cmad(acc[u], w, x);
        idx[u] += inc[u];
        if (idx[u] >= N) idx[u] -= N;
      }
    }
  };
  // pass 1: over n2 for each n1, then the twiddle w^(n1 k2): s[k2 R1 + n1]
  const int g2 = (R2 + kDftOut - 1) / kDftOut;
  for (int e = threadIdx.x; e < rows * R1 * g2; e += blockDim.x) {
    const int n1 = e % R1, rest = e / R1, k0 = (rest % g2) * kDftOut, row = rest / g2;
    C2 acc[kDftOut];
    sums(a + size_t(row) * N + n1, R1, R2, R1, k0, acc);
#pragma unroll
    for (int u = 0; u < kDftOut; ++u)
      if (k0 + u < R2) {
        C2 w = tw[n1 * (k0 + u)];
        if (inverse) w.y = -w.y;
        s[size_t(row) * N + (k0 + u) * R1 + n1] = cmul(acc[u], w);
      }
  }
  __syncthreads();
  // pass 2: over n1 for each k2: X[k2 + R2 k1]
  const int g1 = (R1 + kDftOut - 1) / kDftOut;
  for (int e = threadIdx.x; e < rows * R2 * g1; e += blockDim.x) {
    const int k2 = e % R2, rest = e / R2, k0 = (rest % g1) * kDftOut, row = rest / g1;
    C2 acc[kDftOut];
    sums(s + size_t(row) * N + k2 * R1, 1, R1, R2, k0, acc);
#pragma unroll
    for (int u = 0; u < kDftOut; ++u)
      if (k0 + u < R1) a[size_t(row) * N + k2 + R2 * (k0 + u)] = acc[u];
  }
  __syncthreads();
}

// the divisor of N nearest to its square root from below
__device__ __forceinline__ int dft_factor(int N) {
  int r = int(sqrtf(float(N)) + 0.5f);
  while (N % r) --r;
  return r;
}

template <int K, bool MIXED>
struct LatCtx {
  using T = LatT<MIXED>;
  using C2 = typename T::C2;
  static constexpr int NL = K + 1, C = 3 * NL;
  // facet stride of the solver vectors: padded to 4 for k = 2 in the mixed form, so that
  // every facet's values are one aligned 16- or 32-byte access
  static constexpr int VS = (MIXED && NL == 3) ? 4 : NL;
  // stored entries per wavenumber: FP32, the deflated eigen form (the eigenvector v1 of the
  // largest inverse eigenvalue, that eigenvalue, the packed upper triangle of the rest);
  // FP64, the full inverse block
  static constexpr int NP = MIXED ? C + 1 + C * (C + 1) / 2 : C * C;
  int N, logn, NK, ntj;   // NK = N/2 + 1 wavenumbers ki; ntj row tiles per facet type
  int grp;                // rows transformed at a time (the scratch holds grp rows)
  bool pow2;              // FFT (N a power of two) or two-factor DFT
  int r1;                 // its first factor
  C2* tw;                 // [N] exp(-2 pi i t / N)
  C2* bufa;               // transform data, max(C, 2(k+1)) rows of N
  C2* scr;                // scratch, grp rows of lattice_scratch_row(N)
  C2* X;                  // [C][NK][N] spectrum: half along i, full along j (then along kj)
  // split column pass (lattice_split): each column ki is two work items, the even and the
  // odd wavenumbers kj (one decimation-in-frequency step, then transforms of length N/2);
  // their inverse halves go to X2 and the inverse row pass adds them
  bool split;
  C2* tw2;                // [N/2] exp(-2 pi i t / (N/2))
  C2* X2;                 // [C][NK][N]: [0, N/2) the even half E, [N/2, N) w^-j times the odd half
  const C2* S;            // [NK][NP][N] S^(kappa)^+ (packed upper triangle or full), kj fastest
  // vectors, facet-major [n_facet][NL] in lattice order
  typename T::V *lam, *g, *r, *q;
  typename T::Z* z;
};

// Forward or inverse transform, in place, of `rows` natural-order rows held in a: groups
// of L.grp rows go through the scratch buffer. Powers of two up to FourStepMax: the
// two-pass FFT; larger powers of two: Stockham passes (a result left in the scratch is
// copied back); other N: the two-factor DFT.
template <int K, bool MIXED>
__device__ void xform(const LatCtx<K, MIXED>& L, typename LatT<MIXED>::C2* a, int rows, bool inverse) {
  using C2 = typename LatT<MIXED>::C2;
  const int N = L.N;
  for (int r0 = 0; r0 < rows; r0 += L.grp) {
    const int gr = min(L.grp, rows - r0);
    C2* d = a + size_t(r0) * N;
    if (L.pow2 && L.logn <= FourStepMax<C2>::logn) {
      switch (L.logn) {
        case 0: break;
        case 1: fft_four_step<2, 1>(d, L.scr, gr, L.tw, inverse); break;
        case 2: fft_four_step<2, 2>(d, L.scr, gr, L.tw, inverse); break;
        case 3: fft_four_step<4, 2>(d, L.scr, gr, L.tw, inverse); break;
        case 4: fft_four_step<4, 4>(d, L.scr, gr, L.tw, inverse); break;
        case 5: fft_four_step<8, 4>(d, L.scr, gr, L.tw, inverse); break;
        case 6: fft_four_step<8, 8>(d, L.scr, gr, L.tw, inverse); break;
        case 7: fft_four_step<16, 8>(d, L.scr, gr, L.tw, inverse); break;
        case 8: fft_four_step<16, 16>(d, L.scr, gr, L.tw, inverse); break;
        default:
          if constexpr (FourStepMax<C2>::logn >= 10) {
            if (L.logn == 9) fft_four_step<32, 16>(d, L.scr, gr, L.tw, inverse);
            else fft_four_step<32, 32>(d, L.scr, gr, L.tw, inverse);
          }
          break;
      }
      continue;
    }
    if (L.pow2) {
      const C2* res = fft_stockham(d, L.scr, gr, L.logn, L.tw, inverse);
      if (res != d) {
        for (int e = threadIdx.x; e < gr * N; e += blockDim.x) d[e] = res[e];
        __syncthreads();
      }
    } else {
      dft_two_factor(d, L.scr, gr, N, L.r1, L.tw, inverse);
    }
  }
}

// ---- one facet's NL values of a solver vector (facet stride VS), as aligned vector
// accesses where the stride allows (coherent L2 loads: the data was written by other
// blocks before the last grid barrier)
template <int NL, int VS>
__device__ __forceinline__ void ldf(const float2* p, dfl (&v)[NL]) {
  if constexpr (VS % 2 == 0) {
#pragma unroll
    for (int h = 0; h < VS / 2; ++h) {
      const float4 w = __ldcg(reinterpret_cast<const float4*>(p) + h);
      if (2 * h < NL) v[2 * h] = dfl(w.x, w.y);
      if (2 * h + 1 < NL) v[2 * h + 1] = dfl(w.z, w.w);
    }
  } else {
#pragma unroll
    for (int j = 0; j < NL; ++j) v[j] = to_dfl(__ldcg(p + j));
  }
}
template <int NL, int VS>
__device__ __forceinline__ void stf(float2* p, const dfl (&v)[NL]) {
  if constexpr (VS % 2 == 0) {
#pragma unroll
    for (int h = 0; h < VS / 2; ++h) {
      const dfl a = (2 * h < NL) ? v[2 * h] : dfl(0), b = (2 * h + 1 < NL) ? v[2 * h + 1] : dfl(0);
      reinterpret_cast<float4*>(p)[h] = make_float4(a.hi, a.lo, b.hi, b.lo);
    }
  } else {
#pragma unroll
    for (int j = 0; j < NL; ++j) p[j] = to_float2(v[j]);
  }
}
template <int NL, int VS>
__device__ __forceinline__ void ldf(const float* p, float (&v)[NL]) {
  if constexpr (VS == 4) {
    const float4 w = __ldcg(reinterpret_cast<const float4*>(p));
    const float t[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int j = 0; j < NL; ++j) v[j] = t[j];
  } else if constexpr (VS == 2) {
    const float2 w = __ldcg(reinterpret_cast<const float2*>(p));
    v[0] = w.x;
    v[NL - 1] = w.y;
  } else {
#pragma unroll
    for (int j = 0; j < NL; ++j) v[j] = __ldcg(p + j);
  }
}
template <int NL, int VS>
__device__ __forceinline__ void stf(float* p, const float (&v)[NL]) {
  if constexpr (VS == 4) {
    float t[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < NL; ++j) t[j] = v[j];
    *reinterpret_cast<float4*>(p) = make_float4(t[0], t[1], t[2], t[3]);
  } else if constexpr (VS == 2) {
    *reinterpret_cast<float2*>(p) = make_float2(v[0], v[NL - 1]);
  } else {
#pragma unroll
    for (int j = 0; j < NL; ++j) p[j] = v[j];
  }
}
template <int NL, int VS>
__device__ __forceinline__ void ldf(const double* p, double (&v)[NL]) {
  if constexpr (VS % 2 == 0) {
#pragma unroll
    for (int h = 0; h < VS / 2; ++h) {
      const double2 w = __ldcg(reinterpret_cast<const double2*>(p) + h);
      if (2 * h < NL) v[2 * h] = w.x;
      if (2 * h + 1 < NL) v[2 * h + 1] = w.y;
    }
  } else {
#pragma unroll
    for (int j = 0; j < NL; ++j) v[j] = __ldcg(p + j);
  }
}
template <int NL, int VS>
__device__ __forceinline__ void stf(double* p, const double (&v)[NL]) {
  if constexpr (VS % 2 == 0) {
#pragma unroll
    for (int h = 0; h < VS / 2; ++h) reinterpret_cast<double2*>(p)[h] = make_double2(v[2 * h], v[2 * h + 1]);
  } else {
#pragma unroll
    for (int j = 0; j < NL; ++j) p[j] = v[j];
  }
}

// Facets are numbered (type, j, i) on a lattice mesh, so a tile of kLatTJ rows of one
// facet type with all k+1 modes is one contiguous range of the facet-major vectors:
// DOF index ((type N + j) N + i) VS + m.

// Row pass, forward: per tile read r; src(o, rv) sees (and may change) the values of the facet that
// start at o; pack rows j0+2p (real part) and j0+2p+1 (imaginary part) per mode, FFT along i, split
// into the two rows' half spectra and store them in X.
template <int K, bool MIXED, typename Src>
__device__ __forceinline__ void rows_forward(const LatCtx<K, MIXED>& L, Src src) {
  using T = LatT<MIXED>;
  using C2 = typename T::C2;
  using R = typename T::R;
  using A = typename T::A;
  constexpr int NL = K + 1, VS = LatCtx<K, MIXED>::VS;
  const int N = L.N, NK = L.NK;
  const int ntiles = 3 * L.ntj;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int ty = tile / L.ntj, j0 = (tile - ty * L.ntj) * kLatTJ;
    const int rows = min(kLatTJ, N - j0), npair = (rows + 1) >> 1;
    const size_t base = (size_t(ty) * N + j0) * N * VS;
#pragma unroll 4
    for (int e = threadIdx.x; e < rows * N; e += blockDim.x) {   // one facet (row r_, column i)
      const int r_ = e / N, i = e - r_ * N;
      const size_t o = base + size_t(e) * VS;
      A rv[NL];
      ldf<NL, VS>(L.r + o, rv);
      src(o, rv);
#pragma unroll
      for (int mm = 0; mm < NL; ++mm) {
        C2* slot = &L.bufa[((r_ >> 1) * NL + mm) * N + i];
        if (r_ & 1) slot->y = fft_in(rv[mm]);
        else slot->x = fft_in(rv[mm]);
      }
    }
    if (rows & 1)   // the last pair has no odd row
      for (int e = threadIdx.x; e < NL * N; e += blockDim.x) L.bufa[((npair - 1) * NL) * N + e].y = R(0);
    __syncthreads();
    xform(L, L.bufa, npair * NL, false);
    const C2* res = L.bufa;
    // Z = X_even + i X_odd: X_even[k] = (Z[k] + conj Z[-k]) / 2, X_odd[k] = (Z[k] - conj Z[-k]) / (2i)
    for (int e = threadIdx.x; e < rows * NK * NL; e += blockDim.x) {
      const int r_ = e % rows, rest = e / rows;
      const int ki = rest % NK, mm = rest / NK;
      const C2* row = res + ((r_ >> 1) * NL + mm) * N;
      const C2 Z = row[ki], Zc = row[ki == 0 ? 0 : N - ki];
      C2 out;
      if (r_ & 1) {
        out.x = R(0.5) * (Z.y + Zc.y);
        out.y = R(-0.5) * (Z.x - Zc.x);
      } else {
        out.x = R(0.5) * (Z.x + Zc.x);
        out.y = R(0.5) * (Z.y - Zc.y);
      }
      L.X[(size_t(ty * NL + mm) * NK + ki) * N + j0 + r_] = out;
    }
    __syncthreads();
  }
}

// y = S^(kappa)^+ x for the C values x_b = cur[b rs + kc], in place; the symbol entry e is
// S[e N + ks] (mixed form: from its deflated eigen form, FP64: the full block).
template <int K, bool MIXED>
__device__ __forceinline__ void symbol_product(const typename LatT<MIXED>::C2* S, int N, int ks,
                                               typename LatT<MIXED>::C2* cur, int rs, int kc) {
  using C2 = typename LatT<MIXED>::C2;
  constexpr int C = LatCtx<K, MIXED>::C;
  if constexpr (MIXED) {
    // y = v1 (v1^H x) / mu1 + R x, R the packed Hermitian remainder (R_ba = conj R_ab)
    C2 x[C], y[C];
    C2 s1 = {0, 0};
#pragma unroll
    for (int b = 0; b < C; ++b) {
      x[b] = cur[b * rs + kc];
      cmad_conj(s1, __ldg(&S[size_t(b) * N + ks]), x[b]);
    }
    const typename LatT<MIXED>::R d1 = __ldg(&S[size_t(C) * N + ks]).x;
    s1.x *= d1;
    s1.y *= d1;
#pragma unroll
    for (int a = 0; a < C; ++a) y[a] = cmul(__ldg(&S[size_t(a) * N + ks]), s1);
    int pi = C + 1;
#pragma unroll
    for (int a = 0; a < C; ++a)
#pragma unroll
      for (int b = a; b < C; ++b, ++pi) {
        const C2 h = __ldg(&S[size_t(pi) * N + ks]);
        cmad(y[a], h, x[b]);
        if (b != a) cmad_conj(y[b], h, x[a]);
      }
#pragma unroll
    for (int a = 0; a < C; ++a) cur[a * rs + kc] = y[a];
  } else {
    C2 x[C], y[C];
#pragma unroll
    for (int b = 0; b < C; ++b) {
      x[b] = cur[b * rs + kc];
      y[b] = C2{0, 0};
    }
#pragma unroll
    for (int a = 0; a < C; ++a)
#pragma unroll
      for (int b = 0; b < C; ++b) cmad(y[a], __ldg(&S[size_t(a * C + b) * N + ks]), x[b]);
#pragma unroll
    for (int a = 0; a < C; ++a) cur[a * rs + kc] = y[a];
  }
}

// Column pass: per ki, FFT along j, y = S^(kappa)^+ x, inverse FFT along j.
// Split form (L.split): the work items are (ki, parity p). With h = N/2 and w = exp(-2 pi i/N),
// one decimation-in-frequency step gives the even wavenumbers X[2k] = DFT_h(x_j + x_(j+h)) and
// the odd ones X[2k+1] = DFT_h((x_j - x_(j+h)) w^j); after the product, item p keeps the
// inverse half E = IDFT_h(Y_even) (p = 0) or w^-j IDFT_h(Y_odd) (p = 1) in X2, and the inverse
// row pass takes y_j = E_j + O_j, y_(j+h) = E_j - O_j. The symbol is stored with the even kj
// first, then the odd ones, so that each item reads a contiguous half.
template <int K, bool MIXED>
__device__ void columns(const LatCtx<K, MIXED>& L) {
  using C2 = typename LatT<MIXED>::C2;
  constexpr int C = LatCtx<K, MIXED>::C;
  constexpr int NP = LatCtx<K, MIXED>::NP;
  const int N = L.N, NK = L.NK;
  if (L.split) {
    const int h = N / 2;
    LatCtx<K, MIXED> Lh = L;
    Lh.N = h;
    Lh.logn = L.logn - 1;
    Lh.pow2 = (h & (h - 1)) == 0;
    Lh.r1 = dft_factor(h);
    Lh.tw = L.tw2;
    for (int item = blockIdx.x; item < 2 * NK; item += gridDim.x) {
      const int ki = item >> 1, par = item & 1;
#pragma unroll 6
      for (int e = threadIdx.x; e < C * h; e += blockDim.x) {
        const int c = e / h, j = e - c * h;
        const C2* col = &L.X[(size_t(c) * NK + ki) * N];
        const C2 a = __ldcg(&col[j]), b = __ldcg(&col[j + h]);
        L.bufa[e] = par ? cmul(csub(a, b), L.tw[j]) : cadd(a, b);
      }
      __syncthreads();
      xform(Lh, L.bufa, C, false);
      const C2* S = L.S + size_t(ki) * NP * N;
      for (int k = threadIdx.x; k < h; k += blockDim.x) symbol_product<K, MIXED>(S, N, par * h + k, L.bufa, h, k);
      __syncthreads();
      xform(Lh, L.bufa, C, true);
      for (int e = threadIdx.x; e < C * h; e += blockDim.x) {
        const int c = e / h, j = e - c * h;
        C2 v = L.bufa[e];
        if (par) {
          C2 w = L.tw[j];
          w.y = -w.y;
          v = cmul(v, w);
        }
        L.X2[(size_t(c) * NK + ki) * N + par * h + j] = v;
      }
      __syncthreads();
    }
    return;
  }
  for (int ki = blockIdx.x; ki < NK; ki += gridDim.x) {
#pragma unroll 12
    for (int e = threadIdx.x; e < C * N; e += blockDim.x) {
      const int c = e / N, j = e - c * N;
      L.bufa[e] = __ldcg(&L.X[(size_t(c) * NK + ki) * N + j]);
    }
    __syncthreads();
    xform(L, L.bufa, C, false);
    const C2* S = L.S + size_t(ki) * NP * N;
    for (int kj = threadIdx.x; kj < N; kj += blockDim.x) symbol_product<K, MIXED>(S, N, kj, L.bufa, N, kj);
    __syncthreads();
    xform(L, L.bufa, C, true);
    const C2* res = L.bufa;
    for (int e = threadIdx.x; e < C * N; e += blockDim.x) {
      const int c = e / N, j = e - c * N;
      L.X[(size_t(c) * NK + ki) * N + j] = res[e];
    }
    __syncthreads();
  }
}

// Row pass, inverse: rebuild W = Y_even + i Y_odd over all k (Y[N-k] = conj Y[k]),
// inverse FFT along i, z = the real / imaginary parts scaled by 1/N^2 in facet order, stored and
// given to fin(o, zv).
template <int K, bool MIXED, typename Fin>
__device__ __forceinline__ void rows_inverse(const LatCtx<K, MIXED>& L, Fin fin) {
  using T = LatT<MIXED>;
  using C2 = typename T::C2;
  using R = typename T::R;
  using Z = typename T::Z;
  constexpr int NL = K + 1, VS = LatCtx<K, MIXED>::VS;
  const int N = L.N, NK = L.NK;
  const R scale = R(1.0 / (double(N) * double(N)));
  const int ntiles = 3 * L.ntj;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int ty = tile / L.ntj, j0 = (tile - ty * L.ntj) * kLatTJ;
    const int rows = min(kLatTJ, N - j0), npair = (rows + 1) >> 1;
#pragma unroll 8
    for (int e = threadIdx.x; e < npair * NK * NL; e += blockDim.x) {
      const int pr = e % npair, rest = e / npair;
      const int ki = rest % NK, mm = rest / NK;
      C2 ya, yb = C2{0, 0};
      if (L.split) {
        // y_j = E_j + O_j and y_(j+h) = E_j - O_j from the two halves of the split pass
        const int h = N >> 1;
        const C2* src = &L.X2[(size_t(ty * NL + mm) * NK + ki) * N];
        const int ja = j0 + 2 * pr, jb = ja + 1;
        const int ra = ja < h ? ja : ja - h, rb = jb < h ? jb : jb - h;
        const C2 ea = __ldcg(&src[ra]), oa = __ldcg(&src[h + ra]);
        ya = ja < h ? cadd(ea, oa) : csub(ea, oa);
        if (2 * pr + 1 < rows) {
          const C2 eb = __ldcg(&src[rb]), ob = __ldcg(&src[h + rb]);
          yb = jb < h ? cadd(eb, ob) : csub(eb, ob);
        }
      } else {
        const C2* src = &L.X[(size_t(ty * NL + mm) * NK + ki) * N + j0 + 2 * pr];
        ya = __ldcg(src);
        if (2 * pr + 1 < rows) yb = __ldcg(src + 1);
      }
      C2* w = L.bufa + (pr * NL + mm) * N;
      w[ki] = C2{ya.x - yb.y, ya.y + yb.x};
      if (ki > 0 && N - ki >= NK) w[N - ki] = C2{ya.x + yb.y, yb.x - ya.y};
    }
    __syncthreads();
    xform(L, L.bufa, npair * NL, true);
    const C2* res = L.bufa;
    const size_t base = (size_t(ty) * N + j0) * N * VS;
#pragma unroll 4
    for (int e = threadIdx.x; e < rows * N; e += blockDim.x) {
      const int r_ = e / N, i = e - r_ * N;
      const size_t o = base + size_t(e) * VS;
      Z zv[NL];
#pragma unroll
      for (int mm = 0; mm < NL; ++mm) {
        const C2 v = res[((r_ >> 1) * NL + mm) * N + i];
        zv[mm] = Z((r_ & 1) ? v.y : v.x) * Z(scale);
      }
      fin(o, zv);
      stf<NL, VS>(L.z + o, zv);
    }
    __syncthreads();
  }
}

// ---- loads of any vector type as the arithmetic type of its form
__device__ __forceinline__ double ldx(const double* p) { return __ldcg(p); }
__device__ __forceinline__ dfl ldx(const float2* p) { return to_dfl(__ldcg(p)); }
__device__ __forceinline__ float ldx(const float* p) { return __ldcg(p); }

// y = (S x)_f: the facet's own block and its four neighbours' (stencil class of f)
template <int NL, int VS, bool MIXED, typename X, typename XV>
__device__ __forceinline__ void spmv_lat(const DevMesh& m, int f, const X* x, XV, typename LatT<MIXED>::A (&y)[NL]) {
  using A = typename LatT<MIXED>::A;
  using Acc = typename LatT<MIXED>::Acc;
  int nb[5];
  facet_nbrs<NL>(m, f, nb);
  const size_t sb = size_t(__ldg(&m.facet_stencil[f])) * 5 * NL * NL;
  XV xs[5][NL];
#pragma unroll
  for (int b = 0; b < 5; ++b) ldf<NL, VS>(x + size_t(nb[b]) * VS, xs[b]);
  Acc acc[NL];
#pragma unroll
  for (int i = 0; i < NL; ++i) acc[i] = acc_zero(Acc{});
#pragma unroll
  for (int b = 0; b < 5; ++b)
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      const XV xv = xs[b][j];
#pragma unroll
      for (int i = 0; i < NL; ++i) mad(acc[i], stencil_entry(m, sb + (b * NL + i) * NL + j, A{}), xv);
    }
#pragma unroll
  for (int i = 0; i < NL; ++i) y[i] = fin(acc[i]);
}

// The warm start of a solve from the multiplier history and its image under S in one pass:
// lam0 = c1 h1 + c2 h2 (h2 read only if use2) at facet f and at its four stencil neighbours,
// y = (S lam0)_f. Every facet forms its own and its neighbours' lam0 with the same operations,
// so lam0 (returned for f) is the same bits wherever it is formed.
template <int NL, int VS, bool MIXED>
__device__ __forceinline__ void spmv_lat_hist(const DevMesh& m, int f, const typename LatT<MIXED>::V* h1,
                                              const typename LatT<MIXED>::V* h2, typename LatT<MIXED>::A c1,
                                              typename LatT<MIXED>::A c2, bool use2,
                                              typename LatT<MIXED>::A (&lam0)[NL], typename LatT<MIXED>::A (&y)[NL]) {
  using A = typename LatT<MIXED>::A;
  using Acc = typename LatT<MIXED>::Acc;
  int nb[5];
  facet_nbrs<NL>(m, f, nb);
  const size_t sb = size_t(__ldg(&m.facet_stencil[f])) * 5 * NL * NL;
  A xs[5][NL];
#pragma unroll
  for (int b = 0; b < 5; ++b) {
    const size_t o = size_t(nb[b]) * VS;
    ldf<NL, VS>(h1 + o, xs[b]);
    if (use2) {
      A t[NL];
      ldf<NL, VS>(h2 + o, t);
#pragma unroll
      for (int j = 0; j < NL; ++j) xs[b][j] = c1 * xs[b][j] + c2 * t[j];
    } else {
#pragma unroll
      for (int j = 0; j < NL; ++j) xs[b][j] = c1 * xs[b][j];
    }
  }
  Acc acc[NL];
#pragma unroll
  for (int i = 0; i < NL; ++i) acc[i] = acc_zero(Acc{});
#pragma unroll
  for (int b = 0; b < 5; ++b)
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      const A xv = xs[b][j];
#pragma unroll
      for (int i = 0; i < NL; ++i) mad(acc[i], stencil_entry(m, sb + (b * NL + i) * NL + j, A{}), xv);
    }
#pragma unroll
  for (int i = 0; i < NL; ++i) {
    y[i] = fin(acc[i]);
    lam0[i] = xs[0][i];
  }
}

// g of facet f in the arithmetic type of the form
template <int NL>
__device__ __forceinline__ void facet_g(const DevMesh& m, int f, double (&gv)[NL]) {
  assemble_g<NL>(m, f, gv);
}
template <int NL>
__device__ __forceinline__ void facet_g(const DevMesh& m, int f, dfl (&gv)[NL]) {
  assemble_g_df<NL>(m, f, gv);
}

// ---- grid reductions of the per-thread partials, in the accumulator's own arithmetic
// (FP32 TwoSum pairs in the mixed form: no FP64 pipe): warps, then warp 0 for the block;
// the block partial goes to m.red (a dacc pair occupies the 8 bytes of a double slot);
// after the barrier every thread loads at most a couple of block partials, and the same
// warp / block steps give the grid sum, broadcast through shared memory. Fixed order:
// bitwise reproducible and identical in every block.
__device__ __forceinline__ double acc_combine(double a, double b) { return a + b; }
__device__ __forceinline__ dacc acc_combine(dacc a, dacc b) {
  float s, t;
  two_sum(a.s, b.s, s, t);
  return dacc{s, a.c + b.c + t};
}
__device__ __forceinline__ double shfl_acc(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ dacc shfl_acc(dacc v, int o) {
  return dacc{__shfl_xor_sync(0xffffffffu, v.s, o), __shfl_xor_sync(0xffffffffu, v.c, o)};
}
template <typename Acc>
__device__ __forceinline__ Acc warp_acc(Acc v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = acc_combine(v, shfl_acc(v, o));
  return v;
}
__device__ __forceinline__ void red_store(double* p, double v) { *p = v; }
__device__ __forceinline__ void red_store(double* p, dacc v) { *reinterpret_cast<float2*>(p) = make_float2(v.s, v.c); }
__device__ __forceinline__ double red_load(const double* p, double) { return __ldcg(p); }
__device__ __forceinline__ dacc red_load(const double* p, dacc) {
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return dacc{v.x, v.y};
}

// Grid sums of N per-thread partials, in the accumulator's own arithmetic and in a fixed order;
// thread 0 of every block then takes them to fn(sums), whose results other threads read from shared
// memory after the call. FP64 instructions occupy a quarter of an SM for 64 cycles a warp, so the
// partials go through shared memory (one warp a sum, eight values a lane) instead of a butterfly
// over every warp, and no scalar is formed by more than one warp. scr: N rows of kLatThreads.
constexpr int kLatSums = 4;
template <int N, typename Acc, typename F>
__device__ __forceinline__ bool lat_reduce(const DevMesh& m, Barrier& bar, int slot0, const Acc (&v)[N],
                                           Acc (*scr)[kLatThreads], F&& fn) {
  static_assert(N <= kLatSums, "scratch rows");
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < N; ++i) scr[i][threadIdx.x] = v[i];
  __syncthreads();
  if (w < N) {
    Acc b = scr[w][l];
#pragma unroll
    for (int k = 1; k < kLatThreads / 32; ++k) b = acc_combine(b, scr[w][l + 32 * k]);
    b = warp_acc(b);
    if (l == 0) red_store(&m.red[size_t(slot0 + w) * kMaxSolverBlocks + blockIdx.x], b);
  }
  if (!grid_sync(bar, m.stats)) return false;
  if (w < N) {
    Acc g = acc_zero(Acc{});
    for (int k = l; k < int(gridDim.x); k += 32)
      g = acc_combine(g, red_load(&m.red[size_t(slot0 + w) * kMaxSolverBlocks + k], Acc{}));
    g = warp_acc(g);
    if (l == 0) scr[w][0] = g;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t[N];
#pragma unroll
    for (int i = 0; i < N; ++i) t[i] = acc_val(scr[i][0]);
    fn(t);
  }
  __syncthreads();
  return true;
}

// Scalars of the solve: written by thread 0 of each block (identically in every block), read by
// all after a block barrier.
template <typename A>
struct LatScal {
  A alpha, alpha_lam, beta, mean;
  double sum[2];
  float scale;
  int done, conv;
  double relres;
};

// ---- facet passes, a lane per value: LP lanes a facet (the last idle for three modes), lane i its
// mode i. Against a thread a facet this needs a quarter of the registers, so that a thread keeps
// the loads of several values in flight, and every access of a warp is a contiguous run.
template <int NL>
struct LatLanes {
  static constexpr int LP = NL == 2 ? 2 : 4;
};
// fn(f, i, live): lanes past the last facet or mode run along with live = false.
template <int NL, typename F>
__device__ __forceinline__ void lat_facets(int nF, F&& fn) {
  constexpr int LP = LatLanes<NL>::LP;
  const int i0 = threadIdx.x & (LP - 1), i = i0 < NL ? i0 : NL - 1;
  const int step = int(gridDim.x * blockDim.x) / LP;
  const int f0 = int(blockIdx.x * blockDim.x + threadIdx.x) / LP;
  const int w0 = int(blockIdx.x * blockDim.x + (threadIdx.x & ~31)) / LP;
#pragma unroll 2
  for (int d = 0; w0 + d < nF; d += step) {
    const int f = f0 + d;
    fn(f < nF ? f : nF - 1, i, f < nF && i0 < NL);
  }
}

__device__ __forceinline__ double shfl_lane(double v, int l, int w) { return __shfl_sync(0xffffffffu, v, l, w); }
__device__ __forceinline__ dfl shfl_lane(dfl v, int l, int w) {
  return dfl(__shfl_sync(0xffffffffu, v.hi, l, w), __shfl_sync(0xffffffffu, v.lo, l, w));
}

// an entry of the stencil classes' blocks, [class][5][NL][NL] in the vector type
template <int NL>
__device__ __forceinline__ double lat_entry(const double* S, int o, double) { return S[o]; }
template <int NL>
__device__ __forceinline__ dfl lat_entry(const float2* S, int o, dfl) { return to_dfl(S[o]); }

// Mode i of g at facet f from the packed offsets of its two sides' condensation outputs
// (m.lat_src: 2 x offset of the side's mode 0, + 1 where the side runs the facet backwards: odd
// Legendre modes change sign).
__device__ __forceinline__ double lat_g(const DevMesh& m, int f, int i, double) {
  const int2 s = __ldg(&m.lat_src[f]);
  const double a = __ldcg(&m.gl[(s.x >> 1) + i]), b = __ldcg(&m.gl[(s.y >> 1) + i]);
  return ((s.x & i & 1) ? -a : a) + ((s.y & i & 1) ? -b : b);
}
__device__ __forceinline__ dfl lat_g(const DevMesh& m, int f, int i, dfl) {
  const int2 s = __ldg(&m.lat_src[f]);
  const dfl a = to_dfl(__ldcg(&m.gl_df[(s.x >> 1) + i])), b = to_dfl(__ldcg(&m.gl_df[(s.y >> 1) + i]));
  return ((s.x & i & 1) ? -a : a) + ((s.y & i & 1) ? -b : b);
}

// The squares that give |g| and |r| are summed in double-float in the mixed form, of values scaled
// by a power of two against the ends of the FP32 exponents: 2^32 in the first pass, which does not
// know |g| yet, then the one that brings g to a root mean square in [1, 2). A sum above kLatSumMax,
// or a mean square at the stopping threshold (rtol |g|)^2 below kLatMeanMin (of the scaled values:
// there a square's trailing word would leave the exponents), is left to lat_pcg, which scales by |g|
// from the start. FP64: unscaled.
constexpr float kLatScale = 4294967296.f;
constexpr double kLatMeanMin = 1e-30, kLatSumMax = 1e36;
__device__ __forceinline__ void add_square(double& a, double v, float) { a = fma(v, v, a); }
__device__ __forceinline__ void add_square(dacc& a, dfl v, float scale) {
  const dfl x(v.hi * scale, v.lo * scale);
  mad(a, x, x);
}

// Iterative refinement. Returns 0 when the solve ended (st.conv, st.relres and it are set), -1 when
// a barrier's wait ran out, 1 when lat_pcg has to take the solve from its start, 2 when it has to
// go on from lam (the history has moved then). A start that is farther off than zero (multipliers of
// another state, or not finite) is dropped: against it rounding, eps |S lam0|, would stay in lam and
// the recursive residual would not show it.
template <int K, bool MIXED>
__device__ __forceinline__ int lat_refine(const DevMesh& m, const SolveArgs& a, const LatCtx<K, MIXED>& L,
                                          const typename LatT<MIXED>::V* S, Barrier& bar,
                                          LatScal<typename LatT<MIXED>::A>& sc,
                                          typename LatT<MIXED>::Acc (*scr)[kLatThreads], int& it) {
  using T = LatT<MIXED>;
  using V = typename T::V;
  using A = typename T::A;
  using Acc = typename T::Acc;
  using Z = typename T::Z;
  constexpr int NL = K + 1, VS = LatCtx<K, MIXED>::VS, LP = LatLanes<NL>::LP;
  const int nF = m.n_facet;
  const A warm = A(a.warm_scale), hc1 = A(a.c1), hc2 = A(a.c2);
  V* hist1 = static_cast<V*>(a.hist1);
  V* hist2 = static_cast<V*>(a.hist2);
  V* hnew = static_cast<V*>(a.hist_new);
  const bool use2 = a.c2 != 0.0;
  bool lam0 = hist1 || a.warm_scale != 0.0;   // false: start from zero
  // (S x)_i from the lanes' x of the five facets
  auto product = [&](const A (&x)[5], int cls, int i) {
    Acc acc = acc_zero(Acc{});
    const V* row = S + (cls * 5 * NL + i) * NL;
#pragma unroll
    for (int b = 0; b < 5; ++b)
#pragma unroll
      for (int j = 0; j < NL; ++j) mad(acc, lat_entry<NL>(row, b * NL * NL + j, A{}), shfl_lane(x[b], j, LP));
    return fin(acc);
  };
  // thread 0's own: the squared norms (scaled), without the constant-multiplier component
  double stop2 = 0.0, floor2 = 0.0, gg = 0.0, rr = 0.0;
  double f2 = MIXED ? double(kLatScale) * double(kLatScale) : 1.0;   // the scale's square
  // g from both sides of every facet, the warm start lam0 = c1 hist1 + c2 hist2 (or warm_scale lam,
  // or zero) and r = g - S lam0 in one pass: a facet forms its neighbours' lam0 from the history
  // with the same operations as they do, so that lam0 is the same bits wherever it is formed
  for (;; lam0 = false) {
    Acc s4[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) s4[i] = acc_zero(Acc{});
    lat_facets<NL>(nF, [&](int f, int i, bool live) {
      const size_t o = size_t(f) * VS + i;
      const A g = lat_g(m, f, i, A{});
      A r = g;
      if (lam0) {
        const int4 nb = __ldg(reinterpret_cast<const int4*>(m.facet_nbr) + f);
        const int n5[5] = {f, nb.x, nb.y, nb.z, nb.w};
        const int cls = __ldg(&m.facet_stencil[f]);
        const V* src = hist1 ? hist1 : L.lam;
        A x[5], x2[5];
#pragma unroll
        for (int b = 0; b < 5; ++b) x[b] = ldv(src + size_t(n5[b]) * VS + i);
        if (hist1 && use2) {
#pragma unroll
          for (int b = 0; b < 5; ++b) x2[b] = ldv(hist2 + size_t(n5[b]) * VS + i);
#pragma unroll
          for (int b = 0; b < 5; ++b) x[b] = hc1 * x[b] + hc2 * x2[b];
        } else {
          const A c = hist1 ? hc1 : warm;
#pragma unroll
          for (int b = 0; b < 5; ++b) x[b] = c * x[b];
        }
        r = g - product(x, cls, i);
        if (hist1 && live) stv(L.lam + o, x[0]);
      }
      if (!live) return;
      stv(L.r + o, r);
      add_square(s4[0], g, kLatScale);
      add_square(s4[1], r, kLatScale);
      if (i == 0) {
        acc_add(s4[2], g);
        acc_add(s4[3], r);
      }
    });
    // (a second pass sums in other slots: blocks may still read the first one's)
    if (!lat_reduce<4>(m, bar, lam0 ? 4 : 0, s4, scr, [&](const double (&t)[4]) {
          const double inv = 1.0 / double(nF);
          gg = t[0] - t[2] * t[2] * f2 * inv;
          rr = nonneg(t[1] - t[3] * t[3] * f2 * inv);
          stop2 = a.rtol * a.rtol * gg;
          floor2 = a.floor_rtol * a.floor_rtol * gg;
          sc.mean = A(t[3] * inv);
          sc.conv = 0;
          sc.done = 0;
          if (!(stop2 * (MIXED ? inv / NL : 1.0) >= (MIXED ? kLatMeanMin : 1e-280) &&
                gg <= (MIXED ? kLatSumMax : 1e280))) {
            sc.done = 3;   // out of range, zero or not finite
          } else if (lam0 && !(rr <= gg)) {
            sc.done = 4;
          } else if (rr <= stop2) {
            sc.done = sc.conv = 1;
            sc.relres = sqrt(rr / gg);
          } else if constexpr (MIXED) {
            const int e = ilogb(gg * inv / NL) >> 1;   // the root mean square of kLatScale g is 2^e to 2^(e+1)
            const double down = ldexp(1.0, -2 * e);
            sc.scale = ldexpf(kLatScale, -e);
            f2 *= down;
            gg *= down;
            rr *= down;
            stop2 *= down;
            floor2 *= down;
          }
        }))
      return -1;
    if (sc.done != 4) break;
  }
  if (sc.done == 3) return 1;
  const bool at_once = sc.done != 0;
  while (!sc.done) {
    const bool first = it == 0;
    // z = B r. The constant multiplier is in the kernel of S and of B: refinement cannot reduce r's
    // component along it, which only rounding feeds; it is left out of the norms and subtracted
    // from r in the next update.
    rows_forward<K, MIXED>(L, [](size_t, A (&)[NL]) {});
    if (!grid_sync(bar, m.stats)) return -1;
    columns<K, MIXED>(L);
    if (!grid_sync(bar, m.stats)) return -1;
    // lam += z; the first pass moves the history down one slot, every pass stores the new entry
    const A mean = sc.mean;
    const float scale = sc.scale;
    rows_inverse<K, MIXED>(L, [&](size_t o, const Z (&zv)[NL]) {
      A lv[NL];
      if (first && !lam0) {
#pragma unroll
        for (int j = 0; j < NL; ++j) lv[j] = as_a(zv[j]);
      } else {
        ldf<NL, VS>(L.lam + o, lv);
#pragma unroll
        for (int j = 0; j < NL; ++j) lv[j] = (first && !hist1 ? warm * lv[j] : lv[j]) + as_a(zv[j]);
      }
      stf<NL, VS>(L.lam + o, lv);
      if (first && hist1) {
        A hv[NL];
        ldf<NL, VS>(hist1 + o, hv);
        stf<NL, VS>(hist2 + o, hv);
      }
      if (hnew) stf<NL, VS>(hnew + o, lv);
    });
    if (!grid_sync(bar, m.stats)) return -1;
    // r -= S z and its constant component
    Acc s2[2] = {acc_zero(Acc{}), acc_zero(Acc{})};
    lat_facets<NL>(nF, [&](int f, int i, bool live) {
      const size_t o = size_t(f) * VS + i;
      const int4 nb = __ldg(reinterpret_cast<const int4*>(m.facet_nbr) + f);
      const int n5[5] = {f, nb.x, nb.y, nb.z, nb.w};
      const int cls = __ldg(&m.facet_stencil[f]);
      A r = ldv(L.r + o);
      Z z[5][NL];
#pragma unroll
      for (int b = 0; b < 5; ++b) ldf<NL, VS>(L.z + size_t(n5[b]) * VS, z[b]);
      Acc acc = acc_zero(Acc{});
      const V* row = S + (cls * 5 * NL + i) * NL;
#pragma unroll
      for (int b = 0; b < 5; ++b)
#pragma unroll
        for (int j = 0; j < NL; ++j) mad(acc, lat_entry<NL>(row, b * NL * NL + j, A{}), z[b][j]);
      r = r - fin(acc);
      if (i == 0) r = r - mean;
      if (!live) return;
      stv(L.r + o, r);
      add_square(s2[0], r, scale);
      if (i == 0) acc_add(s2[1], r);
    });
    ++it;
    const int n = it;
    if (!lat_reduce<2>(m, bar, n & 1 ? 0 : 2, s2, scr, [&](const double (&t)[2]) {
          const double inv = 1.0 / double(nF), prev = rr;
          rr = nonneg(t[0] - t[1] * t[1] * f2 * inv);
          sc.mean = A(t[1] * inv);
          sc.relres = sqrt(rr / gg);
          if (!isfinite(rr)) {
            if (blockIdx.x == 0) atomicOr(&m.stats->flags, kFlagNonFinite);
            sc.done = 1;
          } else if (rr <= stop2 || (rr <= floor2 && rr > 0.25 * prev)) {
            // converged, or at the rounding floor (an iteration no longer halves the residual)
            sc.done = sc.conv = 1;
          } else if (n >= a.maxit) {
            sc.done = 1;
          } else if (!(rr <= a.gain * prev)) {
            sc.done = 3;
          }
        }))
      return -1;
  }
  if (sc.done == 3) return 2;
  if (at_once) {   // no pass has moved the history or stored lam
    const int gsz = gridDim.x * blockDim.x;
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < nF; f += gsz) {
      const size_t o = size_t(f) * VS;
      A lv[NL], hv[NL];
      if (hist1) {
        ldf<NL, VS>(hist1 + o, hv);
        stf<NL, VS>(hist2 + o, hv);
      }
      if (!(hist1 && lam0)) {
#pragma unroll
        for (int j = 0; j < NL; ++j) lv[j] = A(0);
        if (lam0) {
          ldf<NL, VS>(L.lam + o, lv);
#pragma unroll
          for (int j = 0; j < NL; ++j) lv[j] = warm * lv[j];
        }
        stf<NL, VS>(L.lam + o, lv);
      } else {
        ldf<NL, VS>(L.lam + o, lv);
      }
      if (hnew) stf<NL, VS>(hnew + o, lv);
    }
  }
  return 0;
}

// lat_reduce with the sums in every thread
template <int N, typename Acc, typename A>
__device__ __forceinline__ bool lat_sums(const DevMesh& m, Barrier& bar, int slot0, const Acc (&v)[N],
                                         Acc (*scr)[kLatThreads], LatScal<A>& sc, double (&out)[N]) {
  if (!lat_reduce<N>(m, bar, slot0, v, scr, [&](const double (&t)[N]) {
#pragma unroll
        for (int i = 0; i < N; ++i) sc.sum[i] = t[i];
      }))
    return false;
#pragma unroll
  for (int i = 0; i < N; ++i) out[i] = sc.sum[i];
  return true;
}

__device__ __forceinline__ bool grid_reduce_pair(const DevMesh& m, Barrier& bar, int slot0, double a, double b,
                                                 double (&out)[2]) {
  out[0] = a;
  out[1] = b;
  return grid_reduce<2>(m, slot0, out, bar);
}

// The solve as PCG preconditioned by B, on the system scaled by the size of g: for systems where
// refinement gains too little, or whose size is outside the range of its sums. Returns 0 when the
// solve ended, -1 when a barrier's wait ran out, 1 when the start is farther off than zero (the
// history has moved; call again without it).
template <int K, bool MIXED>
__device__ __noinline__ int lat_pcg(const DevMesh& m, const SolveArgs& a, const LatCtx<K, MIXED>& L,
                                     typename LatT<MIXED>::V* p, Barrier& bar, LatScal<typename LatT<MIXED>::A>& sc,
                                     typename LatT<MIXED>::Acc (*scr)[kLatThreads], int& it) {
  using T = LatT<MIXED>;
  using V = typename T::V;
  using A = typename T::A;
  using Acc = typename T::Acc;
  using Z = typename T::Z;
  constexpr int NL = K + 1, VS = LatCtx<K, MIXED>::VS;
  const int nF = m.n_facet;
  const int gtid = blockIdx.x * blockDim.x + threadIdx.x, gsz = gridDim.x * blockDim.x;
  // g from both sides of every facet and the warm start lam0. With a history (the same stage
  // of earlier steps), lam0 = c1 hist1 + c2 hist2 and r = g - S lam0 in the same pass (every
  // facet forms its neighbours' lam0 from the history, which this launch only reads until
  // the first row pass moves it down one slot); otherwise lam0 = warm_scale lam (or zero),
  // and r = g - S lam0 takes a pass of its own after a grid barrier.
  const A warm = A(a.warm_scale), hc1 = A(a.c1), hc2 = A(a.c2);
  V* hist1 = static_cast<V*>(a.hist1);
  V* hist2 = static_cast<V*>(a.hist2);
  const bool use2 = a.c2 != 0.0;
  double ga = 0.0;
  Acc g0 = acc_zero(Acc{});
#pragma unroll 4
  for (int f = gtid; f < nF; f += gsz) {
    const size_t o = size_t(f) * VS;
    A gv[NL], lv[NL];
    facet_g<NL>(m, f, gv);
    if (hist1) {
      A y[NL];
      spmv_lat_hist<NL, VS, MIXED>(m, f, hist1, hist2, hc1, hc2, use2, lv, y);
#pragma unroll
      for (int j = 0; j < NL; ++j) y[j] = gv[j] - y[j];
      stf<NL, VS>(L.r + o, y);
    } else {
      if (a.warm_scale != 0.0) {
        ldf<NL, VS>(L.lam + o, lv);
#pragma unroll
        for (int j = 0; j < NL; ++j) lv[j] = warm * lv[j];
      } else {
#pragma unroll
        for (int j = 0; j < NL; ++j) lv[j] = A(0);
      }
      stf<NL, VS>(L.g + o, gv);
    }
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      const double lead = lead_d(gv[j]);
      ga = fma(lead, lead, ga);
    }
    stf<NL, VS>(L.lam + o, lv);
    acc_add(g0, gv[0]);
  }
  double gg[2];
  {
    // FP64 sums (the squares of any g fit), through the double slots of the scratch
    if (!grid_reduce_pair(m, bar, 4, ga, acc_val(g0), gg)) return -1;
  }
  const double c0 = gg[1] / double(nF);
  const double gnorm0 = sqrt(nonneg(gg[0] - gg[1] * gg[1] / double(nF)));
  // PCG runs on the system scaled by sigma = 2^-e, e the exponent of the RMS entry of g
  // (exact in any precision): residuals and dot products stay near 1 whatever the size
  // of g, away from the FP32 exponent limits of the double-float form. r and p are
  // scaled, lam is not: lam += (alpha / sigma) p.
  const double sigma = gnorm0 > 0.0 ? ldexp(1.0, -ilogb(gnorm0 / sqrt(double(nF) * NL))) : 1.0;
  const double gnorm = sigma * gnorm0;
  const double stop2 = (a.rtol * gnorm) * (a.rtol * gnorm);
  // rounding floor: the recursive residual stops decreasing near eps * cond(S) relative
  // (double-float vectors: 1e-14..1e-12 on large meshes; FP64: near 1e-13 at N = 1024);
  // once an iteration no longer halves the residual and it is below floor_rtol, the
  // solve is accepted there
  const double floor2 = (a.floor_rtol * gnorm) * (a.floor_rtol * gnorm);
  bool conv = false;
  double relres = 0.0;
  if (!(gnorm0 > 0.0)) {   // no data, or a NaN (a state that holds one): zero
    for (int f = gtid; f < nF; f += gsz) {
      const size_t o = size_t(f) * VS;
      A zero[NL];
#pragma unroll
      for (int j = 0; j < NL; ++j) zero[j] = A(0);
      stf<NL, VS>(L.lam + o, zero);
      if (hist1) {
        A hv[NL];
        ldf<NL, VS>(hist1 + o, hv);
        stf<NL, VS>(hist2 + o, hv);
      }
    }
    conv = true;
  } else {
    if (!hist1) {
      // r = g - S lam0
#pragma unroll 4
      for (int f = gtid; f < nF; f += gsz) {
        const size_t o = size_t(f) * VS;
        A y[NL], gv[NL];
        spmv_lat<NL, VS, MIXED>(m, f, L.lam, A{}, y);
        ldf<NL, VS>(L.g + o, gv);
#pragma unroll
        for (int j = 0; j < NL; ++j) y[j] = gv[j] - y[j];
        stf<NL, VS>(L.r + o, y);
      }
      if (!grid_sync(bar, m.stats)) return -1;
    }
    // z = M r
    // The constant multiplier is in the kernel of S and of the preconditioner, so PCG cannot
    // reduce r's component along it; rounding in every update adds to it (relative size
    // eps times the cancellation in S q). It is measured with r.r (the sum of the mode-0
    // entries), left out of the convergence test, and subtracted from r in the next update.
    // The first row pass scales r by sigma and removes the constant component of g from it:
    // r = sigma (g - c0 1 - S lam0).
    Acc rra[2] = {acc_zero(Acc{}), acc_zero(Acc{})};
    {
      const A cm = A(c0), scale = A(sigma);
      rows_forward<K, MIXED>(L, [&](size_t o, A (&rv)[NL]) {
        rv[0] = rv[0] - cm;
#pragma unroll
        for (int j = 0; j < NL; ++j) {
          rv[j] = scale * rv[j];
          mad(rra[0], rv[j], rv[j]);
        }
        acc_add(rra[1], rv[0]);
        stf<NL, VS>(L.r + o, rv);
        if (hist1) {
          A hv[NL];
          ldf<NL, VS>(hist1 + o, hv);
          stf<NL, VS>(hist2 + o, hv);
        }
      });
    }
    double rr[2];
    if (!lat_sums<2>(m, bar, 6, rra, scr, sc, rr)) return -1;
    double cmode = rr[1] / double(nF);
    rr[0] = nonneg(rr[0] - rr[1] * rr[1] / double(nF));
    // (gnorm is that of g's leading words: up to its rounding)
    if ((hist1 || a.warm_scale != 0.0) && !(rr[0] <= gnorm * gnorm * 1.0001)) return 1;
    columns<K, MIXED>(L);
    if (!grid_sync(bar, m.stats)) return -1;
    Acc rza[2] = {acc_zero(Acc{}), acc_zero(Acc{})};
    rows_inverse<K, MIXED>(L, [&](size_t o, const Z (&zv)[NL]) {
      A rv[NL];
      ldf<NL, VS>(L.r + o, rv);
#pragma unroll
      for (int j = 0; j < NL; ++j) mad(rza[0], rv[j], zv[j]);
    });
    double rz[2];
    {
      const Acc rz1[1] = {rza[0]};
      double rzt[1];
      if (!lat_sums<1>(m, bar, 1, rz1, scr, sc, rzt)) return -1;
      rz[0] = rzt[0];
    }
    double rho = rz[0], rrv = rr[0];
    double beta = 0.0;
    for (int n = 0;; ++it, ++n) {
      // convergence and the scalars of this step, once per block
      if (threadIdx.x == 0) {
        sc.done = 0;
        sc.conv = 0;
        sc.relres = sqrt(rrv) / gnorm;
        if (!isfinite(rrv) || !isfinite(rho)) {
          if (blockIdx.x == 0) atomicOr(&m.stats->flags, kFlagNonFinite);
          sc.done = 1;
        } else if (rrv <= stop2) {
          sc.done = sc.conv = 1;
        } else if (it >= a.maxit) {
          sc.done = 1;
        }
        sc.beta = A(beta);
      }
      __syncthreads();
      relres = sc.relres;
      if (sc.done) {
        conv = sc.conv != 0;
        break;
      }
      // p = z + beta p, q = S p = S z + beta q (each facet updates only its own entries)
      const A bt = sc.beta;
      Acc pqa[1] = {acc_zero(Acc{})};
#pragma unroll 4
      for (int f = gtid; f < nF; f += gsz) {
        const size_t o = size_t(f) * VS;
        A y[NL], pv[NL], qv[NL];
        Z zz[NL];
        spmv_lat<NL, VS, MIXED>(m, f, L.z, Z{}, y);
        ldf<NL, VS>(L.z + o, zz);
        if (n > 0) {
          ldf<NL, VS>(p + o, pv);
          ldf<NL, VS>(L.q + o, qv);
        }
#pragma unroll
        for (int j = 0; j < NL; ++j) {
          const A zv = as_a(zz[j]);
          pv[j] = (n == 0) ? zv : zv + bt * pv[j];
          qv[j] = (n == 0) ? y[j] : y[j] + bt * qv[j];
          mad(pqa[0], pv[j], qv[j]);
        }
        stf<NL, VS>(p + o, pv);
        stf<NL, VS>(L.q + o, qv);
      }
      double pq[1];
      if (!lat_sums<1>(m, bar, 0, pqa, scr, sc, pq)) return -1;
      if (threadIdx.x == 0) {
        sc.done = 0;
        if (!(pq[0] > 0.0)) {
          if (!isfinite(pq[0]) && blockIdx.x == 0) atomicOr(&m.stats->flags, kFlagNonFinite);
          sc.done = 1;
        } else {
          const double alpha = rho / pq[0];
          sc.alpha = A(alpha);
          sc.alpha_lam = A(alpha / sigma);
        }
      }
      __syncthreads();
      if (sc.done) break;
      // r -= alpha q, lam += alpha p, and the forward row pass of z = M r
      rra[0] = acc_zero(Acc{});
      rra[1] = acc_zero(Acc{});
      {
        const A al = sc.alpha, all = sc.alpha_lam, cm = A(cmode);
        rows_forward<K, MIXED>(L, [&](size_t o, A (&rv)[NL]) {
          A qv[NL], lv[NL], pv[NL];
          ldf<NL, VS>(L.q + o, qv);
          ldf<NL, VS>(L.lam + o, lv);
          ldf<NL, VS>(p + o, pv);
#pragma unroll
          for (int j = 0; j < NL; ++j) {
            rv[j] = rv[j] - al * qv[j];
            lv[j] = lv[j] + all * pv[j];
          }
          rv[0] = rv[0] - cm;   // the constant-multiplier component measured last pass
#pragma unroll
          for (int j = 0; j < NL; ++j) mad(rra[0], rv[j], rv[j]);
          acc_add(rra[1], rv[0]);
          stf<NL, VS>(L.r + o, rv);
          stf<NL, VS>(L.lam + o, lv);
        });
      }
      if (!lat_sums<2>(m, bar, 6, rra, scr, sc, rr)) return -1;
      cmode = rr[1] / double(nF);
      const double rr_prev = rrv;
      rrv = nonneg(rr[0] - rr[1] * rr[1] / double(nF));
      if (threadIdx.x == 0) {
        sc.done = 0;
        sc.conv = 0;
        const bool stagnated = rrv <= floor2 && rrv > 0.25 * rr_prev;
        if (rrv <= stop2 || !isfinite(rrv) || stagnated) {
          sc.done = 1;
          sc.relres = sqrt(rrv) / gnorm;
          sc.conv = isfinite(rrv) ? 1 : 0;
          if (!sc.conv && blockIdx.x == 0) atomicOr(&m.stats->flags, kFlagNonFinite);
        }
      }
      __syncthreads();
      if (sc.done) {
        ++it;
        relres = sc.relres;
        conv = sc.conv != 0;
        break;
      }
      columns<K, MIXED>(L);
      if (!grid_sync(bar, m.stats)) return -1;
      rza[0] = acc_zero(Acc{});
      rza[1] = acc_zero(Acc{});
      rows_inverse<K, MIXED>(L, [&](size_t o, const Z (&zv)[NL]) {
        A rv[NL];
        Z zo[NL];
        ldf<NL, VS>(L.r + o, rv);
        ldf<NL, VS>(L.z + o, zo);
#pragma unroll
        for (int j = 0; j < NL; ++j) {
          mad(rza[1], rv[j], zo[j]);
          mad(rza[0], rv[j], zv[j]);
        }
      });
      if (!lat_sums<2>(m, bar, 1, rza, scr, sc, rz)) return -1;
      // flexible (Polak-Ribiere) beta: the FP32 preconditioner is symmetric only up to rounding
      beta = (rz[0] - rz[1]) / rho;
      rho = rz[0];
    }
  }
  if (a.hist_new) {
    V* hnew = static_cast<V*>(a.hist_new);
    if (!grid_sync(bar, m.stats)) return -1;
    for (int f = gtid; f < nF; f += gsz) {
      A lv[NL];
      ldf<NL, VS>(L.lam + size_t(f) * VS, lv);
      stf<NL, VS>(hnew + size_t(f) * VS, lv);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    sc.conv = conv ? 1 : 0;
    sc.relres = relres;
  }
  return 0;
}

// One solve: refinement, and PCG where it does not do.
template <int K, bool MIXED>
__global__ void __launch_bounds__(kLatThreads, 2) k_solve_lat(DevMesh m, SolveArgs a) {
  using T = LatT<MIXED>;
  using C2 = typename T::C2;
  using R = typename T::R;
  using V = typename T::V;
  using A = typename T::A;
  using Acc = typename T::Acc;
  constexpr int NL = K + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ LatScal<A> sc;
  __shared__ __align__(16) V stencil[kLatStencils * 5 * NL * NL];
  LatCtx<K, MIXED> L;
  L.N = m.lat_N;
  L.logn = m.lat_logn;
  L.NK = L.N / 2 + 1;
  L.ntj = (L.N + kLatTJ - 1) / kLatTJ;
  L.pow2 = (L.N & (L.N - 1)) == 0;
  L.r1 = dft_factor(L.N);
  L.grp = m.lat_grp;
  L.tw = reinterpret_cast<C2*>(smem_raw);
  L.bufa = L.tw + L.N;
  L.scr = L.bufa + m.lat_bufsz;
  // the reductions run while the transform buffers are free
  Acc(*scr)[kLatThreads] = reinterpret_cast<Acc(*)[kLatThreads]>(L.bufa);
  L.X = reinterpret_cast<C2*>(m.lat_x);
  L.S = reinterpret_cast<const C2*>(m.lat_sinv);
  L.split = m.lat_split != 0;
  L.tw2 = reinterpret_cast<C2*>(smem_raw) + m.lat_tw2_off;
  L.X2 = reinterpret_cast<C2*>(m.lat_x2);
  V* p;
  if constexpr (MIXED) {
    L.lam = m.lam_df;
    L.g = m.lv_g;
    L.r = m.lv_r;
    L.q = m.lv_q;
    L.z = m.lv_z;
    p = m.lv_p;
  } else {
    L.lam = m.lam;
    L.g = m.g;
    L.r = m.r;
    L.q = m.q;
    L.z = m.z;
    p = m.pa;
  }
  for (int t = threadIdx.x; t < L.N; t += blockDim.x) L.tw[t] = C2{R(m.lat_tw[2 * t]), R(m.lat_tw[2 * t + 1])};
  if (L.split)
    for (int t = threadIdx.x; t < L.N / 2; t += blockDim.x)
      L.tw2[t] = C2{R(m.lat_tw[4 * t]), R(m.lat_tw[4 * t + 1])};
  const V* S;   // (a uniform torus has three classes; more are read from global memory)
  if constexpr (MIXED) S = m.st_blk_df;
  else S = m.st_blk;
  if (m.n_stencil <= kLatStencils) {
    for (int t = threadIdx.x; t < m.n_stencil * 5 * NL * NL; t += blockDim.x) stencil[t] = __ldg(&S[t]);
    S = stencil;
  }
  __syncthreads();
  Barrier bar(m.bar);
  int it = 0;
  const int how = lat_refine<K, MIXED>(m, a, L, S, bar, sc, scr, it);
  if (how < 0) return;
  if (how > 0) {
    SolveArgs b = a;
    if (how == 2) {
      b.hist1 = nullptr;
      b.warm_scale = 1.0;
    }
    if (!grid_sync(bar, m.stats)) return;
    for (;;) {
      const int left = lat_pcg<K, MIXED>(m, b, L, p, bar, sc, scr, it);
      if (left < 0) return;
      if (left == 0) break;
      b.hist1 = nullptr;
      b.warm_scale = 0.0;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    DevStats* st = m.stats;
    st->last_iters = it;
    st->total_iters += it;
    st->solves += 1;
    st->last_relres = sc.relres;
    st->last_sweeps = 1;
    st->total_sweeps += 1;
    if (!sc.conv) atomicOr(&st->flags, kFlagNotConverged);
  }
}

}  // namespace
}  // namespace dgdf
