// The sixth-order compact 27-point operator (Eq. scheme) with the Neumann (Eq. 3DN) and
// Sommerfeld-like (Eq. 3DDISCS) face rows, applied matrix-free on planar complex data.
//
// Every row is   sum_{dz=-1,0,1}  wc[dz] C(l+dz) + wn[dz] Nb(l+dz) + wd[dz] Dg(l+dz)
// where for z-plane p, C(p) is the value at (i, j), Nb(p) the sum of the 4 in-plane
// neighbours and Dg(p) the sum of the 4 in-plane diagonals.  Interior rows use the four
// class weights c0..c3 of Eq. scheme; a Sommerfeld-like face row has no ghost plane and
// carries G0 on its own plane and G1 on the next plane inward (Eq. 3DDISCS).  Ghost values
// across x/y faces and across Neumann z faces are even reflections (U_{-1} = U_1);
// across Dirichlet faces they are zero.
//
// A thread block takes an (x, y) tile and marches over a chunk of z planes.  Each plane tile plus a
// one-point halo is staged in shared memory by asynchronous copies issued two or three planes ahead
// into a ring of buffers (one barrier per plane), and the plane's sums are combined with those of its
// neighbours in registers, so every input value is read from global memory once per chunk.
#include <algorithm>

#include "helm6_internal.h"

namespace helm6 {

namespace {

constexpr int ZCH = 32;  // most z planes per block

// FP32: planes per block for `tiles` (x, y) tiles of mz planes: 32 where that leaves `per_sm` blocks per
// SM, else half as many, down to 2 (a block reads two planes more than it computes).  A block
// marches plane by plane, so on small grids its length is the kernel's time; on large ones longer
// blocks read less twice.  Measured, 32 planes a block against this rule: 34 -> 9 us at 32^3,
// 35 -> 19 at 128^3, unchanged at 256^3 (16 planes there: 85 against 82).
constexpr int ZB32 = 3;  // blocks per SM asked for (best of 2 to 32 planes at 64^3 to 256^3)
// share: problems running side by side, which fill the SMs together (6 problems of 96 to 160
// points a side in one batch: 26.5 ms with each block length chosen as if alone, 25.3 so).
int z_chunk(int tiles, int mz, int per_sm, int share = 1) {
  static int sms = 0;
  if (!sms) sms = device_sm_count();
  int z = ZCH;
  while (z > 2 && (int64_t)tiles * ((mz + z - 1) / z) * share < (int64_t)per_sm * sms) z /= 2;
  return z;
}

template <typename T>
struct Sums {
  cpx<T> c, n, d;
};

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Asynchronous 4- or 8-byte copy global -> shared; src_bytes = 0 zero-fills (ghost = 0).
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src, int src_bytes) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(d), "l"(src), "n"(BYTES), "r"(src_bytes)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

__device__ __forceinline__ int ghost_index(int gi, int m, int lo_neumann, int hi_neumann) {
  if (gi < 0) return lo_neumann ? 1 : -1;
  if (gi >= m) return (hi_neumann && gi == m) ? m - 2 : -1;
  return gi;
}

// FP64: a 16 x 32 (x, y) tile, 16 x 16 threads with 2 y-adjacent points each.
//
// Bound by the FP64 pipe (two operations per clock and SM), so what counts is operations per
// point, those of idle lanes included.  The x-neighbour sums of the four halo rows are shared by
// the thread's two points (5 operations per point and component for the in-plane sums), and the
// planes are combined as they arrive: plane p gives
//     G(p) = c1 C + c2 Nb + c3 Dg   to rows p - 1 and p + 1,   c0 C + c1 Nb + c2 Dg   to row p,
// so a row is one sum of three fused chains, 7 operations with real weights, instead of the nine
// of adding up its 27 points class by class; two values per point and component are kept instead of
// three planes' sums.  Tiles are 16 points wide and a warp (4 rows) beyond the grid's edge skips the
// arithmetic, so little of it is spent on padding.  15 -> 12 operations; with the
// blocks chosen below, on a caller's arrays: A x 1214 -> 837 us at 256^3 (FP64 pipe at 12 operations:
// 745), 529 -> 394 at 192^3, 189 -> 107 at 100^3 (complex k); F - A x with its norm 1520 -> 1015 at 256^3.
//
// IL: x, f and y are interleaved complex arrays (a caller's own, or of a call without workspace)
// instead of planar ones.  RW: the interior class weights are real (a real wavenumber); the products
// with the imaginary parts, exact zeros, then drop out.
constexpr int DX = 16, DTY = 16, DLD = DX + 2, DNT = DX * DTY;

template <bool RW>
__device__ __forceinline__ cpx<double> wfma(const cpx<double>& c, const cpx<double>& v, const cpx<double>& a) {
  if constexpr (RW)
    return mk(fmx(c.re, v.re, a.re), fmx(c.re, v.im, a.im));
  else
    return cfma(c, v, a);
}
template <int MODE, bool NORM, bool RW, bool IL, int DR>
__global__ void __launch_bounds__(DNT, 3)
    stencil64_kernel(Geom g, const __grid_constant__ StencilCoef coef, const double* __restrict__ x,
                     double* __restrict__ y, const double* f, double* __restrict__ sumsq, int zch) {
  using Z = cpx<double>;
  // ring of NBUF staged planes; plane p + DIST is requested while plane p is used
  constexpr int DY = DTY * DR, DROWS = DY + 2;
  constexpr int DIST = 2, NBUF = DIST + 2, HALO = DROWS * DLD, PER = (HALO + DNT - 1) / DNT;
  __shared__ __align__(16) double2 sb[NBUF][DROWS][DLD];
  __shared__ double red[DNT / 32];

  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * DX + tx;
  const int i = blockIdx.x * DX + tx, j0 = blockIdx.y * DY + DR * ty;
  const int l0 = blockIdx.z * zch;
  const int l1 = min(l0 + zch, g.mz);
  const int64_t plane = (int64_t)g.mx * g.my;

  // halo elements tid, tid + DNT, ... of every plane: the in-plane source (reflection across
  // Neumann x/y faces) or -1 for a zero ghost, computed once
  int hoff[PER];
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int t = tid + k * DNT;
    hoff[k] = -1;
    if (t < HALO) {
      const int sy = t / DLD, sx = t - sy * DLD;
      const int gi = ghost_index(blockIdx.x * DX + sx - 1, g.mx, g.face[0] == HELM6_NEUMANN, g.face[1] == HELM6_NEUMANN);
      const int gj = ghost_index(blockIdx.y * DY + sy - 1, g.my, g.face[2] == HELM6_NEUMANN, g.face[3] == HELM6_NEUMANN);
      if (gi >= 0 && gj >= 0) hoff[k] = gj * g.mx + gi;
    }
  }
  // the halo tile of the plane feeding position p (ghost planes: reflection across a Neumann z
  // face, zero otherwise) into ring slot `slot`
  auto stage = [&](int p, int slot) {
    int src = p;
    bool zplane = false;
    if (p < 0) {
      if (g.face[4] == HELM6_NEUMANN) src = 1; else zplane = true;
    } else if (p >= g.mz) {
      if (g.face[5] == HELM6_NEUMANN) src = g.mz - 2; else zplane = true;
    }
    const int64_t pbase = (int64_t)src * plane;
    double2* d = &sb[slot][0][0];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int t = tid + k * DNT;
      if (t < HALO) {
        const bool ok = !zplane && hoff[k] >= 0;
        const int64_t idx = ok ? pbase + hoff[k] : 0;
        if constexpr (IL) {
          const uint32_t da = (uint32_t)__cvta_generic_to_shared(d + t);
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(da), "l"((const double2*)x + idx),
                       "r"(ok ? 16 : 0)
                       : "memory");
        } else {
          cp_async<8>(&d[t].x, x + idx, ok ? 8 : 0);
          cp_async<8>(&d[t].y, x + g.N + idx, ok ? 8 : 0);
        }
      }
    }
  };

  const Z c0 = cast<double>(coef.interior.w[1][0]), c1 = cast<double>(coef.interior.w[1][1]);
  const Z c2 = cast<double>(coef.interior.w[1][2]);
  const double c3 = coef.interior.w[0][2].re;  // 1/30: real whatever the wavenumber
  // the Sommerfeld-like face rows, with weights of their own: 1 (low), 2 (high); 0 any other row
  auto face_row = [&](int l) {
    if (l == 0 && g.face[4] == HELM6_SOMMERFELD) return 1;
    if (l == g.mz - 1 && g.face[5] == HELM6_SOMMERFELD) return 2;
    return 0;
  };
  // whether any of the warp's rows (its lanes take two thread rows) lies in the grid
  const bool warp_on = (int)(blockIdx.y * DY + DR * (ty & ~1)) < g.my;
  const Z zero = {0.0, 0.0};
  Z below[DR], part[DR];  // G of the last plane; the row of the last plane without what is above it
#pragma unroll
  for (int q = 0; q < DR; ++q) below[q] = part[q] = zero;
  double acc = 0.0;

  const int pfirst = l0 - 1;
  for (int d = 0; d < DIST; ++d) {
    if (pfirst + d <= l1) stage(pfirst + d, d);
    cp_commit();
  }
  for (int p = pfirst; p <= l1; ++p) {
    const int k = p - pfirst, l = p - 1;  // row l is complete with plane p
    if (p + DIST <= l1) stage(p + DIST, (k + DIST) % NBUF);
    cp_commit();
    Z fv[DR];
    if constexpr (MODE != 0) {
#pragma unroll
      for (int q = 0; q < DR; ++q) {
        fv[q] = zero;
        if (l >= l0 && i < g.mx && j0 + q < g.my) {
          const int64_t idx = (int64_t)l * plane + (int64_t)(j0 + q) * g.mx + i;
          if constexpr (IL) {
            const double2 v = ((const double2*)f)[idx];
            fv[q] = mk(v.x, v.y);
          } else {
            fv[q] = mk(f[idx], f[g.N + idx]);
          }
        }
      }
    }
    cp_wait<DIST>();  // the group of plane p has landed
    __syncthreads();
    if (!warp_on) continue;
    const double2* t0 = &sb[k % NBUF][DR * ty][tx];
    Z c[DR + 2], h[DR + 2];
#pragma unroll
    for (int q = 0; q < DR + 2; ++q) {
      const double2 a = t0[q * DLD], b = t0[q * DLD + 1], e = t0[q * DLD + 2];
      c[q] = mk(b.x, b.y);
      h[q] = mk(a.x + e.x, a.y + e.y);
    }
    const int fl = face_row(l), fp = face_row(p), fn = face_row(p + 1);
#pragma unroll
    for (int q = 0; q < DR; ++q) {
      const Z C = c[q + 1], n = h[q + 1] + (c[q] + c[q + 2]), d = h[q] + h[q + 2];
      const Z G = wfma<RW>(c2, n, wfma<RW>(c1, C, c3 * d));
      auto face = [&](int fc, int a, const Z& base) {  // plane p's part of a face row
        const RowWeights& W = fc == 1 ? coef.s_lo : coef.s_hi;
        return cfma(cast<double>(W.w[a][2]), d, cfma(cast<double>(W.w[a][1]), n, cfma(cast<double>(W.w[a][0]), C, base)));
      };
      Z out = fl ? face(fl, 2, part[q]) : part[q] + G;
      if (p >= l0 && p < l1) part[q] = fp ? face(fp, 1, below[q]) : wfma<RW>(c2, d, wfma<RW>(c1, n, wfma<RW>(c0, C, below[q])));
      below[q] = fn ? face(fn, 0, zero) : G;
      if (l >= l0 && i < g.mx && j0 + q < g.my) {
        const int64_t idx = (int64_t)l * plane + (int64_t)(j0 + q) * g.mx + i;
        if (MODE == 1) out = fv[q] - out;
        if (MODE == 2) out = fv[q] + out;
        if constexpr (IL) {
          ((double2*)y)[idx] = make_double2(out.re, out.im);
        } else {
          y[idx] = out.re;
          y[g.N + idx] = out.im;
        }
        if (NORM) acc += out.re * out.re + out.im * out.im;
      }
    }
  }
  cp_wait<0>();

  if (NORM) {
    acc = warp_sum(acc);
    if ((tid & 31) == 0) red[tid >> 5] = acc;
    __syncthreads();
    if (tid < 32) {
      double v = (tid < DNT / 32) ? red[tid] : 0.0;
      v = warp_sum(v);
      if (tid == 0) {
        const int64_t b = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        sumsq[b] = v;
      }
    }
  }
}

// FP32 variant for the Krylov bulk: 32 x 16 (x, y) tile, a 32 x 4 thread block, each
// thread computing 4 y-adjacent points from 6 x 3 shared-memory loads per component.  A
// halo row is staged in shared memory as [unused x3 | left ghost | 32 points | right ghost]
// (stride 40 floats) so that the 32-point middle is 16-byte aligned and can be copied in
// 16-byte chunks when mx % 4 == 0; the two edge columns, and everything when a chunk would
// cross the field's x extent, are copied element by element with the ghost rules.
constexpr int T4X = 32, T4Y = 16, T4R = 4, T4ROWS = T4Y + 2, T4LD = 40;
constexpr int T4SLOTS = 2 * T4ROWS * 10;  // components x rows x (8 chunks + 2 edges)

// The FP32 kernel's weights, rounded to FP32 once on the host (a conversion per thread and
// weight would run on the FP64 pipe): the four interior class weights and the two
// Sommerfeld-like face rows.
struct StencilCoef32 {
  cpx<float> c[4];
  cpx<float> lo[3][3], hi[3][3];
};

// NORM: accumulate the block's |y|^2 (FP64) into sumsq; a compile-time flag so that the
// FP32 path carries no FP64 arithmetic when no norm is wanted.
// RW: the interior weights are real (a real wavenumber), so each class term is two real
// FMAs instead of a complex multiply-add.
template <int MODE, bool NORM, bool RW>
__global__ void __launch_bounds__(T4X* T4Y / T4R)
    stencil4_kernel(Geom g, StencilCoef32 coef, const float* __restrict__ x, float* __restrict__ y,
                    const float* __restrict__ f, double* __restrict__ sumsq, int zch) {
  constexpr int DIST = 3, NBUF = DIST + 2;
  constexpr int NT = T4X * T4Y / T4R;  // 128 threads
  __shared__ __align__(16) float sbuf[NBUF][2][T4ROWS][T4LD];
  __shared__ double red[NT / 32];

  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * T4X + tx;
  const int x0 = blockIdx.x * T4X, y0 = blockIdx.y * T4Y;
  const int i = x0 + tx;
  const int l0 = blockIdx.z * zch;
  const int l1 = min(l0 + zch, g.mz);
  const int64_t plane = (int64_t)g.mx * g.my;
  const bool xn0 = g.face[0] == HELM6_NEUMANN, xn1 = g.face[1] == HELM6_NEUMANN;
  const bool yn0 = g.face[2] == HELM6_NEUMANN, yn1 = g.face[3] == HELM6_NEUMANN;
  const bool vec_ok = (g.mx & 3) == 0;

  // per-thread staging slots (fixed for every plane): component, halo row, slot kind
  int soff[3], sdst[3], skind[3];  // skind: 0 none, 1 vector chunk, 2 scalar x4, 3 scalar edge
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int t = tid + k * NT;
    skind[k] = 0;
    soff[k] = -1;
    sdst[k] = 0;
    if (t < T4SLOTS) {
      const int comp = t / (T4ROWS * 10), rem = t - comp * (T4ROWS * 10);
      const int sy = rem / 10, sl = rem - sy * 10;
      const int gj = ghost_index(y0 + sy - 1, g.my, yn0, yn1);
      sdst[k] = (comp * T4ROWS + sy) * T4LD;  // start of the row in one ring slot
      if (sl < 8) {
        const int xs = x0 + 4 * sl;
        sdst[k] += 4 + 4 * sl;
        skind[k] = (vec_ok && xs + 3 < g.mx) ? 1 : 2;
        soff[k] = (gj < 0) ? -1 : gj * g.mx + xs;  // row offset of the chunk's first point
      } else {
        const int gi = ghost_index(sl == 8 ? x0 - 1 : x0 + T4X, g.mx, xn0, xn1);
        sdst[k] += (sl == 8) ? 3 : 4 + T4X;
        skind[k] = 3;
        soff[k] = (gj < 0 || gi < 0) ? -1 : gj * g.mx + gi;
      }
      soff[k] = (soff[k] < 0) ? -1 : soff[k];
      // component offset in the source is added at staging time
      skind[k] |= comp << 4;
      // for scalar chunks keep the row index for per-element ghost mapping
      if ((skind[k] & 15) == 2) soff[k] = (gj < 0) ? -1 : gj;  // row only
    }
  }

  auto stage = [&](int p, int slot) {
    int src = p;
    bool zplane = false;
    if (p < 0) {
      if (g.face[4] == HELM6_NEUMANN) src = 1; else zplane = true;
    } else if (p >= g.mz) {
      if (g.face[5] == HELM6_NEUMANN) src = g.mz - 2; else zplane = true;
    }
    const int64_t pbase = (int64_t)src * plane;
    float* sl_base = &sbuf[slot][0][0][0];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int kind = skind[k] & 15;
      if (kind == 0) continue;
      const int comp = skind[k] >> 4;
      const float* xb = x + (comp ? g.N : 0) + pbase;
      float* d = sl_base + sdst[k];
      if (kind == 1) {
        const bool ok = !zplane && soff[k] >= 0;
        const uint32_t da = (uint32_t)__cvta_generic_to_shared(d);
        const float* sp = ok ? xb + soff[k] : x;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(da), "l"(sp), "r"(ok ? 16 : 0)
                     : "memory");
      } else if (kind == 2) {
        // the 4 points of the chunk one by one (x extent not a multiple of 4, or partial tile)
        const int sl = ((sdst[k] % T4LD) - 4) / 4;
        for (int e = 0; e < 4; ++e) {
          const int gi = ghost_index(x0 + 4 * sl + e, g.mx, xn0, xn1);
          const bool ok = !zplane && soff[k] >= 0 && gi >= 0;
          const float* sp = ok ? xb + (int64_t)soff[k] * g.mx + gi : x;
          cp_async<4>(d + e, sp, ok ? 4 : 0);
        }
      } else {
        const bool ok = !zplane && soff[k] >= 0;
        cp_async<4>(d, ok ? xb + soff[k] : x, ok ? 4 : 0);
      }
    }
  };

  const cpx<float> c0 = coef.c[0], c1 = coef.c[1], c2 = coef.c[2], c3 = coef.c[3];
  const cpx<float> zero = {0.f, 0.f};
  // plane sums of three consecutive planes, rotated by renaming: the loop below is
  // unrolled by three so that no register moves are needed
  Sums<float> SA[T4R], SB[T4R], SC[T4R];
#pragma unroll
  for (int r = 0; r < T4R; ++r) SA[r] = SB[r] = SC[r] = Sums<float>{zero, zero, zero};
  double acc = 0.0;

  const int pfirst = l0 - 1;
  for (int d = 0; d < DIST; ++d) {
    if (pfirst + d <= l1) stage(pfirst + d, d);
    cp_commit();
  }
  // step p: the sums of plane p go to PN; rows of plane p - 1 use P0 (plane p - 2), P1
  // (plane p - 1) and PN (plane p)
  auto step = [&](int p, Sums<float>(&PN)[T4R], Sums<float>(&P0)[T4R], Sums<float>(&P1)[T4R]) {
    const int k = p - pfirst;
    if (p + DIST <= l1) stage(p + DIST, (k + DIST) % NBUF);
    cp_commit();
    cp_wait<DIST>();
    __syncthreads();
    const int buf = k % NBUF;
    // 6 halo rows x 3 columns per component for this thread's 4 points
    float vr[T4R + 2][3], vi[T4R + 2][3];
#pragma unroll
    for (int rr = 0; rr < T4R + 2; ++rr) {
#pragma unroll
      for (int cc = 0; cc < 3; ++cc) {
        vr[rr][cc] = sbuf[buf][0][T4R * ty + rr][tx + 3 + cc];
        vi[rr][cc] = sbuf[buf][1][T4R * ty + rr][tx + 3 + cc];
      }
    }
    // x-neighbour sums of the six halo rows, shared by the four points' face and diagonal sums
    float hr[T4R + 2], hi[T4R + 2];
#pragma unroll
    for (int rr = 0; rr < T4R + 2; ++rr) {
      hr[rr] = vr[rr][0] + vr[rr][2];
      hi[rr] = vi[rr][0] + vi[rr][2];
    }
#pragma unroll
    for (int r = 0; r < T4R; ++r) {
      Sums<float> cur;
      cur.c = mk(vr[r + 1][1], vi[r + 1][1]);
      cur.n = mk(hr[r + 1] + vr[r][1] + vr[r + 2][1], hi[r + 1] + vi[r][1] + vi[r + 2][1]);
      cur.d = mk(hr[r] + hr[r + 2], hi[r] + hi[r + 2]);
      PN[r] = cur;
    }
    const int l = p - 1;
    if (l >= l0 && i < g.mx) {
      const bool slo = (l == 0) && (g.face[4] == HELM6_SOMMERFELD);
      const bool shi = (l == g.mz - 1) && (g.face[5] == HELM6_SOMMERFELD);
#pragma unroll
      for (int r = 0; r < T4R; ++r) {
        const int j = y0 + T4R * ty + r;
        if (j >= g.my) continue;
        cpx<float> out;
        if (!slo && !shi) {
          const cpx<float> s1 = P1[r].n + P0[r].c + PN[r].c, s2 = P1[r].d + P0[r].n + PN[r].n,
                           s3 = P0[r].d + PN[r].d;
          if constexpr (RW) {
            out.re = fmaf(c3.re, s3.re, fmaf(c2.re, s2.re, fmaf(c1.re, s1.re, c0.re * P1[r].c.re)));
            out.im = fmaf(c3.re, s3.im, fmaf(c2.re, s2.im, fmaf(c1.re, s1.im, c0.re * P1[r].c.im)));
          } else {
            out = c0 * P1[r].c;
            out = cfma(c1, s1, out);
            out = cfma(c2, s2, out);
            out = cfma(c3, s3, out);
          }
        } else {
          out = zero;
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const cpx<float> wc = slo ? coef.lo[0][a] : coef.hi[0][a];
            const cpx<float> wm = slo ? coef.lo[1][a] : coef.hi[1][a];
            const cpx<float> wp = slo ? coef.lo[2][a] : coef.hi[2][a];
            const cpx<float> s0 = (a == 0) ? P0[r].c : (a == 1) ? P0[r].n : P0[r].d;
            const cpx<float> s1 = (a == 0) ? P1[r].c : (a == 1) ? P1[r].n : P1[r].d;
            const cpx<float> s2 = (a == 0) ? PN[r].c : (a == 1) ? PN[r].n : PN[r].d;
            out = cfma(wc, s0, out);
            out = cfma(wm, s1, out);
            out = cfma(wp, s2, out);
          }
        }
        const int64_t idx = (int64_t)l * plane + (int64_t)j * g.mx + i;
        if (MODE == 1) {
          out = mk(f[idx] - out.re, f[g.N + idx] - out.im);
        } else if (MODE == 2) {
          out = mk(f[idx] + out.re, f[g.N + idx] + out.im);
        }
        y[idx] = out.re;
        y[g.N + idx] = out.im;
        if (NORM) acc += (double)out.re * out.re + (double)out.im * out.im;
      }
    }
  };
  for (int p = pfirst; p <= l1; p += 3) {
    step(p, SA, SB, SC);
    if (p + 1 <= l1) step(p + 1, SB, SC, SA);
    if (p + 2 <= l1) step(p + 2, SC, SA, SB);
  }
  cp_wait<0>();
  if (NORM) {
    acc = warp_sum(acc);
    if ((tid & 31) == 0) red[tid >> 5] = acc;
    __syncthreads();
    if (tid < 32) {
      double v = (tid < NT / 32) ? red[tid] : 0.0;
      v = warp_sum(v);
      if (tid == 0) {
        const int64_t b = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        sumsq[b] = v;
      }
    }
  }
}

}  // namespace

namespace {

// Points per thread (1 or 2) and planes per block: the pair with the least arithmetic on the fullest
// SM.  The FP64 pipe is the bound however many blocks share it, so what counts is whole blocks per SM,
// times planes (a block's first and last plane take half the work), times 13 or 23 operations per
// thread; partial tiles and the last chunk fill the SMs left over by the whole ones or add to
// them (a partial tile of at most four warps 0.6 of a whole one), and no SM does less than the mean.
// Against the best of all pairs tried at eight sizes from 32^3 to 300^3 (apply_A): within 2.6 %; 32
// planes, halved until every SM had four blocks of two points per thread, was up to 60 % off (21 us
// instead of 13 at 32^3, 45 instead of 30 at 64^3, 123 instead of 111 at 100^3).
struct Grid64 {
  int dr, zch;
  dim3 grid;
};
Grid64 grid64(const Geom& g) {
  static int sms = 0;
  if (!sms) sms = device_sm_count();
  auto up = [](int64_t a, int64_t b) { return (a + b - 1) / b; };
  Grid64 b{};
  double best = 1e300;
  for (int dr = 1; dr <= 2; ++dr) {
    const int dy = DTY * dr;
    const int64_t tx = up(g.mx, DX), left_rows = g.my % dy;
    const bool part = left_rows > 0 && left_rows <= dy / 2;  // a tile of at most four warps
    const int64_t ty = g.my / dy + (left_rows > dy / 2), tyf = std::max<int64_t>(1, ty);
    for (int z = 1; z <= 64 && (z == 1 || z < 2 * g.mz); ++z) {
      const int64_t nzf = std::max(1, g.mz / z), rz = g.mz > z ? g.mz % z : 0;
      const double whole = std::min(z, g.mz) + 1, rest = rz ? rz + 1 : 0;
      const int64_t n1 = tx * tyf * nzf, n2 = (rz ? tx * tyf : 0) + (part && ty ? tx * nzf : 0);
      const int64_t rounds = up(n1, sms), spare = rounds * sms - n1;
      const double extra = std::max(rest, part && ty ? 0.6 * whole : 0.0);
      const double full = rounds * whole + (n2 > spare ? extra * up(n2 - spare, sms) : 0.0);
      const double mean = tx * (tyf + (part && ty ? 0.5 : 0.0)) * (nzf * whole + rest) / sms;
      const double cost = std::max(full, mean) * (dr == 1 ? 13 : 23);
      if (cost < best) {
        best = cost;
        b.dr = dr;
        b.zch = z;
        b.grid = dim3((unsigned)tx, (unsigned)up(g.my, dy), (unsigned)up(g.mz, z));
      }
    }
  }
  return b;
}

bool real_weights(const StencilCoef& c) {
  return c.interior.w[1][0].im == 0.0 && c.interior.w[1][1].im == 0.0 && c.interior.w[1][2].im == 0.0;
}

template <int MODE, bool NORM, bool IL>
int run64(const Geom& g, const StencilCoef& c, const double* x, double* y, const double* f, double* sumsq,
          cudaStream_t s) {
  const Grid64 b = grid64(g);
  const dim3 block(DX, DTY);
  const bool rw = real_weights(c);
  note_launch();
  if (rw && b.dr == 1)
    stencil64_kernel<MODE, NORM, true, IL, 1><<<b.grid, block, 0, s>>>(g, c, x, y, f, sumsq, b.zch);
  else if (rw)
    stencil64_kernel<MODE, NORM, true, IL, 2><<<b.grid, block, 0, s>>>(g, c, x, y, f, sumsq, b.zch);
  else if (b.dr == 1)
    stencil64_kernel<MODE, NORM, false, IL, 1><<<b.grid, block, 0, s>>>(g, c, x, y, f, sumsq, b.zch);
  else
    stencil64_kernel<MODE, NORM, false, IL, 2><<<b.grid, block, 0, s>>>(g, c, x, y, f, sumsq, b.zch);
  return (int)(b.grid.x * b.grid.y * b.grid.z);
}

}  // namespace

int stencil_blocks(const Geom& g) {
  // the larger of the two kernels' grids
  const dim3 d = grid64(g).grid;
  const int t16 = ((g.mx + T4X - 1) / T4X) * ((g.my + T4Y - 1) / T4Y);
  const int z16 = z_chunk(t16, g.mz, ZB32);
  return std::max((int)(d.x * d.y * d.z), t16 * ((g.mz + z16 - 1) / z16));
}

void launch_apply64_il(const Geom& g, const StencilCoef& c, const double* x, double* y, cudaStream_t s) {
  run64<0, false, true>(g, c, x, y, nullptr, nullptr, s);
}

int launch_residual64_il(const Geom& g, const StencilCoef& c, const double* F, const double* u, double* r,
                         double* partials, cudaStream_t s) {
  return run64<1, true, true>(g, c, u, r, F, partials, s);
}

template <typename T>
void launch_stencil(const Geom& g, const StencilCoef& c, const T* x, T* y, const T* f, T* r,
                    int mode, double* sumsq, int* nblk, cudaStream_t s, int share) {
  (void)r;
  if (sizeof(T) == 4) {
    dim3 block(T4X, T4Y / T4R);
    dim3 grid((g.mx + T4X - 1) / T4X, (g.my + T4Y - 1) / T4Y);
    // (a norm's partial sums follow the blocks: the same for every caller)
    const int zch = z_chunk((int)(grid.x * grid.y), g.mz, ZB32, sumsq ? 1 : share);
    grid.z = (g.mz + zch - 1) / zch;
    if (nblk) *nblk = (int)(grid.x * grid.y * grid.z);
    note_launch();
    const float* xf = (const float*)x;
    float* yf = (float*)y;
    const float* ff = (const float*)f;
    StencilCoef32 c32;
    const c64d* cw[4] = {&c.interior.w[1][0], &c.interior.w[1][1], &c.interior.w[1][2], &c.interior.w[0][2]};
    for (int q = 0; q < 4; ++q) c32.c[q] = cpx<float>{(float)cw[q]->re, (float)cw[q]->im};
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b) {
        c32.lo[a][b] = cpx<float>{(float)c.s_lo.w[a][b].re, (float)c.s_lo.w[a][b].im};
        c32.hi[a][b] = cpx<float>{(float)c.s_hi.w[a][b].re, (float)c.s_hi.w[a][b].im};
      }
    const bool nrm = sumsq != nullptr;
    const bool rw = c.interior.w[1][0].im == 0.0 && c.interior.w[1][1].im == 0.0 &&
                    c.interior.w[1][2].im == 0.0 && c.interior.w[0][2].im == 0.0;
#define HELM6_S4(M, N)                                                                   \
  do {                                                                                   \
    if (rw)                                                                              \
      stencil4_kernel<M, N, true><<<grid, block, 0, s>>>(g, c32, xf, yf, ff, N ? sumsq : nullptr, zch);  \
    else                                                                                 \
      stencil4_kernel<M, N, false><<<grid, block, 0, s>>>(g, c32, xf, yf, ff, N ? sumsq : nullptr, zch); \
  } while (0)
    if (mode == 0 && !nrm)
      HELM6_S4(0, false);
    else if (mode == 0)
      HELM6_S4(0, true);
    else if (mode == 1 && !nrm)
      HELM6_S4(1, false);
    else if (mode == 1)
      HELM6_S4(1, true);
    else
      HELM6_S4(2, false);
#undef HELM6_S4
    return;
  }
  const double *xd = (const double*)x, *fd = (const double*)f;
  double* yd = (double*)y;
  int nb;
  if (mode == 0)
    nb = sumsq ? run64<0, true, false>(g, c, xd, yd, fd, sumsq, s) : run64<0, false, false>(g, c, xd, yd, fd, nullptr, s);
  else if (mode == 1)
    nb = sumsq ? run64<1, true, false>(g, c, xd, yd, fd, sumsq, s) : run64<1, false, false>(g, c, xd, yd, fd, nullptr, s);
  else
    nb = run64<2, false, false>(g, c, xd, yd, fd, nullptr, s);
  if (nblk) *nblk = nb;
}

template void launch_stencil<float>(const Geom&, const StencilCoef&, const float*, float*,
                                    const float*, float*, int, double*, int*, cudaStream_t, int);
template void launch_stencil<double>(const Geom&, const StencilCoef&, const double*, double*,
                                     const double*, double*, int, double*, int*, cudaStream_t, int);

}  // namespace helm6
