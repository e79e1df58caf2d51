// Compact right side F of the sixth-order scheme for separable sources (FP64): sums of
// Gaussian sources, or any f = sum_t c_t X_t(x) Y_t(y) Z_t(z) given by 1D derivative tables.
//
// Interior (Eq. scheme right side, h^2-scaled; the mixed fourth derivatives carry the
// total weight h^4/90 that makes the scheme sixth order):
//   F = h^2 [ cf f + q1 lap f + (h^4/360) sum_a f_aaaa + (h^4/90) sum_{a<b} f_aabb ] + h^2 cf eta
//   cf = 1 - k^2h^2/12 + k^4h^4/360,  q1 = (h^2/12)(1 - k^2h^2/30).
// Neumann face rows (Eq. 3DN, homogeneous data, minus sign on the 7h^5/180 term):
//   F -= D_N,  D_N = dn1 f_n + dn3 f_nnn + dnm (f_ntt + f_nss)
// Sommerfeld-like face rows (Eq. 3DDISCS), fbar = exp(ik n) f in the inward normal n:
//   F -= D_S,  D_S = -e^{ikh} mu3 [ 2h Fbar + mu1 (h^5/3)(fbar_ntt + fbar_nss) ].
// Each separable term contributes products of its factors' 1D derivatives X^(m)(x),
// m = 0..4, tabulated (complex) per axis at the unknown nodes by the host.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "helm6_internal.h"

#include <climits>

namespace helm6 {

namespace {

struct RhsCoef {
  double h;
  c64d cf, q1;         // interior
  c64d dn1;            // Neumann: coefficient of f_n
  double dn3, dnm;     // Neumann: f_nnn and f_ntt + f_nss
  c64d ik;             // Sommerfeld-like: i k
  c64d a1, a2;         // Fbar = a1 fb_n + a2 fb_nn + a3 (fb_nnn - fb_ntt - fb_nss)
  double a3;
  c64d e1mu3, mu1h5;   // D_S = -e1mu3 (2h Fbar + mu1h5 (fb_ntt + fb_nss))
};

using Z = cpx<double>;

__device__ __forceinline__ Z zc(c64d a) { return Z{a.re, a.im}; }

// Table values of a separable term: real (Gaussian factors) or complex.
struct Re {
  double v;
};
__device__ __forceinline__ Re operator*(Re a, Re b) { return Re{a.v * b.v}; }
__device__ __forceinline__ Re operator+(Re a, Re b) { return Re{a.v + b.v}; }
__device__ __forceinline__ Z operator*(Z a, Re b) { return Z{a.re * b.v, a.im * b.v}; }
// a + w x
__device__ __forceinline__ Z mad(Z w, Re x, Z a) { return Z{fma(w.re, x.v, a.re), fma(w.im, x.v, a.im)}; }
__device__ __forceinline__ Z mad(Z w, Z x, Z a) { return cfma(w, x, a); }
template <bool REAL>
struct TabT {
  using t = Z;
  static __device__ __forceinline__ Z ld(const double* p, int64_t o) { return Z{p[2 * o], p[2 * o + 1]}; }
};
template <>
struct TabT<true> {
  using t = Re;
  static __device__ __forceinline__ Re ld(const double* p, int64_t o) { return Re{p[o]}; }
};

// Nodes [lo, hi) of each axis outside which every derivative of a term's factor is exactly 0
// (a Gaussian's tails underflow); a term is skipped where its product is an exact zero.
struct TermRange {
  int lo[3], hi[3];
};

// Element idx of a complex array: 16 bytes at once where the arrays are aligned to that, else (a caller's
// own buffers may be aligned to a double only) two doubles.
__device__ __forceinline__ Z ldc(const double* p, int64_t idx, bool wide) {
  if (!wide) return Z{p[2 * idx], p[2 * idx + 1]};
  const double2 v = ((const double2*)p)[idx];
  return Z{v.x, v.y};
}
__device__ __forceinline__ void stc(double* p, int64_t idx, const Z& v, bool wide) {
  if (wide) {
    ((double2*)p)[idx] = make_double2(v.re, v.im);
  } else {
    p[2 * idx] = v.re;
    p[2 * idx + 1] = v.im;
  }
}

constexpr int RHS_WARPS = 4, RHS_ROWS = 16, RHS_TERMS = 32;  // warps and x rows of a block, terms per pass

// A Neumann or Sommerfeld-like face's data term is, per separable term with normal factor
// derivatives N0..N3 (N in the inward normal: odd ones change sign at the upper face) and
// tangential factors S, T,   F -= c0 S0 T0 + c2 (S2 T0 + S0 T2)
// with   Neumann      c0 = dn1 N1 + dn3 N3,  c2 = dnm N1
//        Sommerfeld   c0 = -e1mu3 2h [a1 b1 + a2 b2 + a3 b3],  c2 = -e1mu3 (mu1h5 - 2h a3) b1,
//        b1 = ik N0 + N1, b2 = (ik)^2 N0 + 2 ik N1 + N2, b3 = (ik)^3 N0 + 3 (ik)^2 N1 + 3 ik N2 + N3.
template <bool REAL>
__device__ __forceinline__ void face_pair(const RhsCoef& c, int kind, int side, const double* tab, int64_t o, int mmax,
                                          Z& c0, Z& c2) {
  using TT = TabT<REAL>;
  const Z one{1.0, 0.0};
  const Z n0 = one * TT::ld(tab, o), n2 = one * TT::ld(tab, o + 2 * (int64_t)mmax);
  Z n1 = one * TT::ld(tab, o + mmax), n3 = one * TT::ld(tab, o + 3 * (int64_t)mmax);
  if (side) {
    n1 = -1.0 * n1;
    n3 = -1.0 * n3;
  }
  if (kind == HELM6_NEUMANN) {
    c0 = zc(c.dn1) * n1 + c.dn3 * n3;
    c2 = c.dnm * n1;
  } else {
    const Z ik = zc(c.ik), ik2 = ik * ik, ik3 = ik2 * ik;
    const Z b1 = ik * n0 + n1;
    const Z b2 = ik2 * n0 + 2.0 * (ik * n1) + n2;
    const Z b3 = ik3 * n0 + 3.0 * (ik2 * n1) + 3.0 * (ik * n2) + n3;
    const Z e = -1.0 * zc(c.e1mu3);
    c0 = e * ((2.0 * c.h) * (zc(c.a1) * b1 + zc(c.a2) * b2 + c.a3 * b3));
    c2 = e * ((zc(c.mu1h5) - Z{2.0 * c.h * c.a3, 0.0}) * b1);
  }
}

// A block takes RHS_ROWS x rows (j, l).  The compact right side of a separable term is, along a
// row, a combination of the three even derivatives of its x factor alone,
//     F(i) = sum_t A_t X_t(i) + B_t X_t^(2)(i) + C_t X_t^(4)(i)  (+ the x faces' terms at the ends),
// whose coefficients hold the y and z factors, the amplitude and the y and z faces' terms.  The
// block forms them first, one thread per (row, term) and 32 terms at a time, then a warp walks
// a row at 3 FMAs per term and component (real factors) instead of the products of every
// derivative pair.  FP64 arithmetic bounds the kernel, and an FP64 instruction costs the same
// with one lane as with 32: hence the coefficients of several rows at once.  At 256 x 258 x 258
// with eight sources and noise the call takes 0.66 ms, a third of it the host's tables; every
// derivative product at every point took 27.3 ms (the warp forming its own row's coefficients: 0.81).
template <bool REAL>
__global__ void __launch_bounds__(32 * RHS_WARPS) rhs_kernel(Geom g, RhsCoef c, int nterm, int mmax,
                                                             const double* __restrict__ tab,
                                                             const double* __restrict__ amps,
                                                             const TermRange* __restrict__ rng,
                                                             const double* __restrict__ noise, double* __restrict__ F, bool wide) {
  using TT = TabT<REAL>;
  __shared__ Z sA[RHS_ROWS][RHS_TERMS], sB[RHS_ROWS][RHS_TERMS], sC[RHS_ROWS][RHS_TERMS], sE[RHS_ROWS][2][RHS_TERMS];
  __shared__ short2 sR[RHS_ROWS][RHS_TERMS];  // the term's nonzero x nodes (empty: skipped on this row)
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t rows = (int64_t)g.my * g.mz, row0 = (int64_t)blockIdx.x * RHS_ROWS;
  const int nrow = (int)min((int64_t)RHS_ROWS, rows - row0);
  const double h2 = c.h * c.h, h4 = h2 * h2;
  const Z h2cf = h2 * zc(c.cf);
  for (int t0 = 0; t0 == 0 || t0 < nterm; t0 += RHS_TERMS) {
    const int nt = min(RHS_TERMS, nterm - t0);
    for (int e = threadIdx.x; e < nrow * nt; e += 32 * RHS_WARPS) {
      const int r = e / nt, s = e - r * nt, t = t0 + s;
      const int j = (int)((row0 + r) % g.my), l = (int)((row0 + r) / g.my);
      const TermRange q = rng[t];
      const bool on = j >= q.lo[1] && j < q.hi[1] && l >= q.lo[2] && l < q.hi[2];
      sR[r][s] = on ? make_short2((short)q.lo[0], (short)q.hi[0]) : make_short2(0, 0);
      if (!on) continue;
      const Z h2q1 = h2 * zc(c.q1);
      const double p4 = h2 * (h4 / 360.0), m4 = h2 * (h4 / 90.0);
      const int64_t ox = (int64_t)t * 15 * mmax, oy = ox + 5 * (int64_t)mmax + j, oz = ox + 10 * (int64_t)mmax + l;
      const auto y0 = TT::ld(tab, oy), y2 = TT::ld(tab, oy + 2 * (int64_t)mmax), y4 = TT::ld(tab, oy + 4 * (int64_t)mmax);
      const auto z0 = TT::ld(tab, oz), z2 = TT::ld(tab, oz + 2 * (int64_t)mmax), z4 = TT::ld(tab, oz + 4 * (int64_t)mmax);
      const Z am{amps[2 * t], amps[2 * t + 1]};
      const auto yz = y0 * z0, l2 = y2 * z0 + y0 * z2;
      Z A = (h2cf * yz) + (h2q1 * l2) + (Z{p4, 0.0} * (y4 * z0 + y0 * z4)) + (Z{m4, 0.0} * (y2 * z2));
      Z B = (h2q1 * yz) + (Z{m4, 0.0} * l2);
      const Z C = Z{p4, 0.0} * yz;
      Z c0, c2;
      for (int side = 0; side < 2; ++side) {
        if (g.face[2 + side] != HELM6_DIRICHLET && j == (side ? g.my - 1 : 0)) {
          face_pair<REAL>(c, g.face[2 + side], side, tab, oy, mmax, c0, c2);
          A = A - (c0 * z0 + c2 * z2);
          B = B - c2 * z0;
        }
        if (g.face[4 + side] != HELM6_DIRICHLET && l == (side ? g.mz - 1 : 0)) {
          face_pair<REAL>(c, g.face[4 + side], side, tab, oz, mmax, c0, c2);
          A = A - (c0 * y0 + c2 * y2);
          B = B - c2 * y0;
        }
      }
      for (int side = 0; side < 2; ++side) {
        Z x{0.0, 0.0};
        if (g.face[side] != HELM6_DIRICHLET) {
          face_pair<REAL>(c, g.face[side], side, tab, ox + (side ? g.mx - 1 : 0), mmax, c0, c2);
          x = am * (c0 * yz + c2 * l2);
        }
        sE[r][side][s] = x;
      }
      sA[r][s] = am * A;
      sB[r][s] = am * B;
      sC[r][s] = am * C;
    }
    __syncthreads();
    for (int r = w; r < nrow; r += RHS_WARPS) {
      for (int i = lane; i < g.mx; i += 32) {
        const int64_t idx = (row0 + r) * g.mx + i;
        Z v{0.0, 0.0};
        if (t0 > 0)
          v = ldc(F, idx, wide);
        else if (noise)
          v = h2cf * ldc(noise, idx, wide);
        for (int s = 0; s < nt; ++s) {
          const short2 q = sR[r][s];
          if (i < q.x || i >= q.y) continue;
          const int64_t o = (int64_t)(t0 + s) * 15 * mmax + i;
          v = mad(sA[r][s], TT::ld(tab, o), v);
          v = mad(sB[r][s], TT::ld(tab, o + 2 * (int64_t)mmax), v);
          v = mad(sC[r][s], TT::ld(tab, o + 4 * (int64_t)mmax), v);
          if (i == 0) v = v - sE[r][0][s];
          if (i == g.mx - 1) v = v - sE[r][1][s];
        }
        stc(F, idx, v, wide);
      }
    }
    __syncthreads();
  }
}

}  // namespace

// Upload the tables (real [nterm][3][5][mmax] doubles or complex pairs of that shape), the
// coefficients and the terms' nonzero ranges in one buffer, launch, free.
int launch_rhs(const Geom& g, double h, cd k, int nterm, int mmax, const double* tab, bool real, const double* coef,
               const double* noise, double* F, cudaStream_t s) {
  const size_t per = (size_t)15 * mmax * (real ? 1 : 2), ntab = per * nterm;
  const size_t nrng = ((size_t)nterm * sizeof(TermRange) + 7) / 8;
  std::vector<double> buf(std::max<size_t>(ntab + 2 * (size_t)nterm + nrng, 1));
  if (nterm > 0) {
    std::copy(tab, tab + ntab, buf.begin());
    std::copy(coef, coef + 2 * (size_t)nterm, buf.begin() + ntab);
  }
  const int mdim[3] = {g.mx, g.my, g.mz};
  // a non-finite amplitude or table value reaches every point (0 * Inf): nothing is skipped then
  std::vector<TermRange> rg((size_t)nterm);
  for (int t = 0; t < nterm; ++t) {
    bool finite = std::isfinite(coef[2 * t]) && std::isfinite(coef[2 * t + 1]);
    const double* tt = tab + (size_t)t * per;
    const int e = real ? 1 : 2;
    for (int a = 0; a < 3; ++a) {
      int lo = mdim[a], hi = 0;
      for (int m = 0; m < 5; ++m) {
        const double* p = tt + (size_t)(a * 5 + m) * mmax * e;
        for (int i = 0; i < mdim[a] * e; ++i) {
          if (!std::isfinite(p[i])) finite = false;
          if (p[i] != 0.0) {
            lo = std::min(lo, i / e);
            hi = std::max(hi, i / e + 1);
          }
        }
      }
      rg[t].lo[a] = lo;
      rg[t].hi[a] = hi;
    }
    if (!finite)
      for (int a = 0; a < 3; ++a) {
        rg[t].lo[a] = 0;
        rg[t].hi[a] = mdim[a];
      }
  }
  if (nterm > 0) std::memcpy(buf.data() + ntab + 2 * (size_t)nterm, rg.data(), (size_t)nterm * sizeof(TermRange));
  double* dbuf = nullptr;
  if (cudaMallocAsync((void**)&dbuf, buf.size() * sizeof(double), s) != cudaSuccess) {
    cudaGetLastError();
    return HELM6_ERR_NOMEM;
  }
  cudaMemcpyAsync(dbuf, buf.data(), buf.size() * sizeof(double), cudaMemcpyHostToDevice, s);

  RhsCoef c;
  const cd I(0.0, 1.0);
  const cd kh2 = k * k * h * h;
  const double h2 = h * h, h3 = h2 * h, h4 = h2 * h2, h5 = h4 * h;
  c.h = h;
  c.cf = to_pod(1.0 - kh2 / 12.0 + kh2 * kh2 / 360.0);
  c.q1 = to_pod((h2 / 12.0) * (1.0 - kh2 / 30.0));
  c.dn1 = to_pod(-(h3 / 3.0) * (1.0 - kh2 / 20.0));
  c.dn3 = -h5 / 60.0;
  c.dnm = -7.0 * h5 / 180.0;
  const cd ik = I * k;
  c.ik = to_pod(ik);
  const cd mu3 = 1.0 / (1.0 + (2.0 * ik * h / 3.0) * (1.0 + 2.0 * kh2 / 15.0));
  const cd mu1 = (ik * h / 90.0 + (1.0 + kh2 / 30.0) / (6.0 * mu3)) / (1.0 + 2.0 * ik * h / 3.0);
  c.a1 = to_pod(h2 / 6.0 + k * k * h4 / 45.0);
  c.a2 = to_pod(-ik * h4 / 90.0);
  c.a3 = h4 / 120.0;
  c.e1mu3 = to_pod(std::exp(ik * h) * mu3);
  c.mu1h5 = to_pod(mu1 * h5 / 3.0);

  const int64_t rows = (int64_t)g.my * g.mz;
  const unsigned grid = (unsigned)((rows + RHS_ROWS - 1) / RHS_ROWS);
  const double* damp = dbuf + ntab;
  const TermRange* drng = (const TermRange*)(damp + 2 * (size_t)nterm);
  const bool wide = ((uintptr_t)F | (uintptr_t)noise) % 16 == 0;
  note_launch();
  if (real)
    rhs_kernel<true><<<grid, 32 * RHS_WARPS, 0, s>>>(g, c, nterm, mmax, dbuf, damp, drng, noise, F, wide);
  else
    rhs_kernel<false><<<grid, 32 * RHS_WARPS, 0, s>>>(g, c, nterm, mmax, dbuf, damp, drng, noise, F, wide);
  cudaFreeAsync(dbuf, s);
  return cudaGetLastError() == cudaSuccess ? HELM6_OK : HELM6_ERR_CUDA;
}

// Gaussian sources: 1D derivative tables G^(m)(x) = (-1/sigma)^m He_m(t) exp(-t^2/2),
// t = (x-c)/sigma, with He the probabilists' Hermite polynomials, at the unknown nodes of
// each axis (real).
int rhs_gaussians(const Geom& g, double h, cd k, int nsrc, const double* centers, const double* amps,
                  double sigma, const double* noise, double* F, cudaStream_t s) {
  const int mmax = std::max(g.mx, std::max(g.my, g.mz));
  const int mdim[3] = {g.mx, g.my, g.mz};
  std::vector<double> tab((size_t)nsrc * 15 * mmax, 0.0);
  for (int src = 0; src < nsrc; ++src) {
    for (int ax = 0; ax < 3; ++ax) {
      const int start = (g.face[2 * ax] == HELM6_DIRICHLET) ? 1 : 0;
      for (int p = 0; p < mdim[ax]; ++p) {
        const double x = (start + p) * h;
        const double t = (x - centers[3 * src + ax]) / sigma;
        const double e = std::exp(-0.5 * t * t);
        double he[5];
        he[0] = 1.0;
        he[1] = t;
        for (int m = 1; m < 4; ++m) he[m + 1] = t * he[m] - m * he[m - 1];
        double sc = 1.0;
        for (int m = 0; m < 5; ++m) {
          tab[(((size_t)src * 3 + ax) * 5 + m) * mmax + (size_t)p] = sc * he[m] * e;
          sc *= -1.0 / sigma;
        }
      }
    }
  }
  return launch_rhs(g, h, k, nsrc, mmax, tab.data(), true, amps, noise, F, s);
}

// Separable source given by the caller's complex tables [nterm][3][5][mmax] (mmax the
// largest axis length), entry p of an axis = the factor's derivative at its p-th unknown.
int rhs_separable(const Geom& g, double h, cd k, int nterm, const double* coef, const double* tables, double* F,
                  cudaStream_t s) {
  const int mmax = std::max(g.mx, std::max(g.my, g.mz));
  return launch_rhs(g, h, k, nterm, mmax, tables, false, coef, nullptr, F, s);
}

namespace {

// Lifting of inhomogeneous Dirichlet data on a z face: the face's nodes are known, so their
// contribution to the neighbouring plane's rows moves to the right side,
//   F(l, j, i) -= sum over the 3 x 3 face nodes around (i, j) of w(di, dj) u_b,
// w = the interior rows' weights of the z +- 1 plane (centre c1, 4 neighbours c2, 4
// diagonals c3 of Eq. scheme).  ub: (my + 2) x (mx + 2) complex128 values on the face's
// node layer, ring included (the nodes of the neighbouring faces' ghost columns and rows).
// Rows next to a Dirichlet face with known values u_b: the face's nodes enter those rows
// through the 27-point weights of the row (interior, or the Sommerfeld-like face rows on z),
// F -= sum over the face's nodes in the row's 3 x 3 window of w * u_b.  A node's weight is the
// row's class weight for its offset: the plane offset along z and the number of nonzero
// in-plane (x, y) offsets (the interior weights are the same for any axis).  The face data
// holds a ring in the tangential axes that are padded before the face's own axis (x, then y,
// then z), so an edge node belongs to exactly one face: x faces [mz][my], y faces
// [mz][mx + 2], z faces [my + 2][mx + 2].
__global__ void lift_face_kernel(Geom g, RowWeights win, RowWeights wlo, RowWeights whi, int axis, int side,
                                 const double* __restrict__ ub, double* __restrict__ F) {
  const int m[3] = {g.mx, g.my, g.mz};
  const int a1 = axis == 0 ? 1 : 0, a2 = axis == 2 ? 1 : 2;  // tangential axes, a1 < a2
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)m[a1] * m[a2]) return;
  const int u1 = (int)(t % m[a1]), u2 = (int)(t / m[a1]);
  int c[3];
  c[axis] = side ? m[axis] - 1 : 0;
  c[a1] = u1;
  c[a2] = u2;
  const RowWeights& W = (c[2] == 0 && g.face[4] == HELM6_SOMMERFELD)            ? wlo
                        : (c[2] == m[2] - 1 && g.face[5] == HELM6_SOMMERFELD) ? whi
                                                                              : win;
  const int r1 = a1 < axis ? 1 : 0, r2 = a2 < axis ? 1 : 0;
  const int ld = m[a1] + 2 * r1;
  // a node beyond the data along a tangential axis: a Neumann face there reflects the ghost
  // onto the data (U_{-1} = U_1); otherwise it belongs to another face's data or is zero
  auto fold = [&](int q, int a, int ring) -> int {
    if (q >= -ring && q < m[a] + ring) return q;
    if (q < 0) return g.face[2 * a] == HELM6_NEUMANN ? 1 : INT_MIN;
    return g.face[2 * a + 1] == HELM6_NEUMANN ? m[a] - 2 : INT_MIN;
  };
  Z s{0.0, 0.0};
  for (int d2 = -1; d2 <= 1; ++d2)
    for (int d1 = -1; d1 <= 1; ++d1) {
      const int p1 = fold(u1 + d1, a1, r1), p2 = fold(u2 + d2, a2, r2);
      if (p1 == INT_MIN || p2 == INT_MIN) continue;
      int o[3];
      o[axis] = side ? 1 : -1;
      o[a1] = d1;
      o[a2] = d2;
      const int cls = (o[0] != 0) + (o[1] != 0);
      const int64_t q = (int64_t)(p2 + r2) * ld + (p1 + r1);
      s = s + zc(W.w[o[2] + 1][cls]) * Z{ub[2 * q], ub[2 * q + 1]};
    }
  const int64_t o = ((int64_t)c[2] * m[1] + c[1]) * m[0] + c[0];
  F[2 * o] -= s.re;
  F[2 * o + 1] -= s.im;
}

}  // namespace

int lift_dirichlet(const Geom& g, const StencilCoef& coef, int face, const double* ub, double* F, cudaStream_t s) {
  const int axis = face / 2, side = face % 2;
  const int m[3] = {g.mx, g.my, g.mz};
  const int64_t n = (int64_t)m[axis == 0 ? 1 : 0] * m[axis == 2 ? 1 : 2];
  note_launch();
  lift_face_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(g, coef.interior, coef.s_lo, coef.s_hi, axis, side,
                                                                ub, F);
  return cudaGetLastError() == cudaSuccess ? (int)HELM6_OK : (int)HELM6_ERR_CUDA;
}

}  // namespace helm6
