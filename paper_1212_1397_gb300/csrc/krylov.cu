// Vector kernels of the Krylov solvers: classical Gram-Schmidt dot products and updates,
// norms, linear combinations, precision conversions, and the FP64 Givens least-squares
// update of GMRES, all on the device.  Dot products accumulate per thread in the vector
// precision and combine block partials in FP64.
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "helm6_internal.h"

namespace helm6 {

namespace {

constexpr int RB = 256;  // threads per block of the reduction kernels

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum a per-thread double over the block; result valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* sh) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  v = (threadIdx.x < (blockDim.x >> 5)) ? sh[threadIdx.x] : 0.0;
  if (w == 0) v = warp_sum(v);
  return v;
}

template <typename T>
__global__ void __launch_bounds__(RB) sumsq_kernel(const T* __restrict__ x, int64_t N,
                                                   double* __restrict__ partial) {
  __shared__ double sh[RB / 32];
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  T a = T(0);
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < 2 * N; idx += stride) {
    const T v = x[idx];
    a = fmx(v, v, a);
  }
  const double s = block_sum((double)a, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

template <typename T>
__global__ void scale_copy_kernel(const T* __restrict__ x, T* __restrict__ y, int64_t n2,
                                  const double* __restrict__ inv_dev, double host_scale) {
  const T s = (T)(inv_dev ? *inv_dev : host_scale);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n2; idx += stride)
    y[idx] = x[idx] * s;
}

template <typename T>
struct V2;
template <>
struct V2<float> {
  using t = float2;
};
template <>
struct V2<double> {
  using t = double2;
};

// out (+)= scale * sum_i V_i y_i, y complex double.  Two points per thread (vector loads
// when the planes allow) and the basis read 8 vectors at a time, so that each thread has
// 16 independent loads in flight; sums in the input precision, widened once.
template <typename TI, typename TO, bool VEC>
__global__ void __launch_bounds__(RB) lincomb_kernel(const TI* __restrict__ V, int64_t vstride, int count,
                                                     const double* __restrict__ y, double scale,
                                                     TO* __restrict__ out, int64_t N, int accumulate,
                                                     const int* __restrict__ count_dev,
                                                     const double* __restrict__ scale_dev) {
  __shared__ TI yr[64], yi[64];
  if (count_dev) count = *count_dev;  // device-driven solves: the cycle's column count
  if (scale_dev) scale = *scale_dev;
  for (int c = threadIdx.x; c < count; c += blockDim.x) {
    yr[c] = (TI)(y[2 * c] * scale);
    yi[c] = (TI)(y[2 * c + 1] * scale);
  }
  __syncthreads();
  constexpr int P = VEC ? 2 : 1;
  constexpr int UB = 8;
  using TV = typename V2<TI>::t;
  const int64_t npts = N / P;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < npts; q += stride) {
    TI sr[P], si[P];
#pragma unroll
    for (int k = 0; k < P; ++k) sr[k] = si[k] = TI(0);
    for (int c0 = 0; c0 < count; c0 += UB) {
      TI vr[UB][P], vi[UB][P];
#pragma unroll
      for (int u = 0; u < UB; ++u) {
        if (c0 + u < count) {
          const TI* v = V + (int64_t)(c0 + u) * vstride;
          if constexpr (VEC) {
            const TV a = ((const TV*)v)[q], b = ((const TV*)(v + N))[q];
            vr[u][0] = a.x;
            vr[u][1 % P] = a.y;
            vi[u][0] = b.x;
            vi[u][1 % P] = b.y;
          } else {
            vr[u][0] = v[q];
            vi[u][0] = v[N + q];
          }
        }
      }
#pragma unroll
      for (int u = 0; u < UB; ++u) {
        if (c0 + u < count) {
          const TI a = yr[c0 + u], b = yi[c0 + u];
#pragma unroll
          for (int k = 0; k < P; ++k) {
            sr[k] = fmx(vr[u][k], a, fmx(-vi[u][k], b, sr[k]));
            si[k] = fmx(vr[u][k], b, fmx(vi[u][k], a, si[k]));
          }
        }
      }
    }
#pragma unroll
    for (int k = 0; k < P; ++k) {
      const int64_t idx = q * P + k;
      if (accumulate) {
        out[idx] += (TO)sr[k];
        out[N + idx] += (TO)si[k];
      } else {
        out[idx] = (TO)sr[k];
        out[N + idx] = (TO)si[k];
      }
    }
  }
}

template <typename TI, typename TO>
__global__ void convert_kernel(const TI* __restrict__ x, TO* __restrict__ y, int64_t n2, double scale,
                               const double* __restrict__ scale_dev) {
  if (scale_dev) scale = *scale_dev;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n2; idx += stride)
    y[idx] = (TO)((double)x[idx] * scale);
}

__global__ void inter_to_planar_kernel(const double2* __restrict__ z, double* __restrict__ out, int64_t N) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += stride) {
    const double2 v = z[idx];
    out[idx] = v.x;
    out[N + idx] = v.y;
  }
}

__global__ void planar_to_inter_kernel(const double* __restrict__ in, double2* __restrict__ z, int64_t N) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += stride)
    z[idx] = make_double2(in[idx], in[N + idx]);
}

// Index in the caller's array of the internal point idx when the caller's axis xaxis
// (0 = x, 1 = y) is the internal z axis (and the internal z axis is the caller's xaxis):
// internal (i, j, l) is the caller's (l, j, i) for xaxis 0 and (i, l, j) for xaxis 1.
__device__ __forceinline__ int64_t caller_index(int64_t idx, int mx, int my, int mz, int xaxis) {
  const int64_t i = idx % mx, j = (idx / mx) % my, l = idx / ((int64_t)mx * my);
  return xaxis == 0 ? (i * my + j) * mz + l : (j * mz + l) * mx + i;
}

__global__ void inter_to_planar_x_kernel(const double2* __restrict__ z, double* __restrict__ out, int mx, int my,
                                         int mz, int xaxis) {
  const int64_t N = (int64_t)mx * my * mz, stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += stride) {
    const double2 v = z[caller_index(idx, mx, my, mz, xaxis)];
    out[idx] = v.x;
    out[N + idx] = v.y;
  }
}

__global__ void planar_to_inter_x_kernel(const double* __restrict__ in, double2* __restrict__ z, int mx, int my,
                                         int mz, int xaxis) {
  const int64_t N = (int64_t)mx * my * mz, stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += stride)
    z[caller_index(idx, mx, my, mz, xaxis)] = make_double2(in[idx], in[N + idx]);
}

__global__ void reduce_sum_kernel(const double* __restrict__ partial, int n, double* __restrict__ out) {
  __shared__ double sh[RB / 32];
  double v = 0.0;
  for (int b = threadIdx.x; b < n; b += blockDim.x) v += partial[b];
  v = block_sum(v, sh);
  if (threadIdx.x == 0) *out = v;
}

// ---- Arnoldi with delayed classical Gram-Schmidt (one reduction + one update per step) ----
// Vector traits for 2-point loads of a planar field.

// Most basis vectors per warp group of the reduction pass (4 accumulators each).  FP64: 4, so that two
// blocks share an SM, one's loads behind the other's arithmetic (eight vectors, one block: 341 us
// instead of 301 per pass at 127^3, 198 and 183 at 101^3, 756 either way at 192^3).
template <typename T>
constexpr int CHD = sizeof(T) == 8 ? 4 : 8;

// P consecutive values of one plane, starting at point q * P, widened to the arithmetic
// type T.  S is the storage type: T itself (P = 1, 2, or 4 for float) or __half (P = 1, 2
// or 4).
template <typename T, int P, typename S>
__device__ __forceinline__ void ldpts(const S* p, int64_t q, T* o) {
  if constexpr (std::is_same<S, T>::value) {
    if constexpr (P == 1) {
      o[0] = p[q];
    } else if constexpr (P == 2) {
      const typename V2<T>::t v = ((const typename V2<T>::t*)p)[q];
      o[0] = v.x;
      o[1] = v.y;
    } else if constexpr (P == 4) {
      static_assert(std::is_same<T, float>::value, "4-point loads are FP32 or FP16");
      const float4 v = ((const float4*)p)[q];
      o[0] = v.x;
      o[1] = v.y;
      o[2] = v.z;
      o[3] = v.w;
    } else {
      static_assert(P == 8 && std::is_same<T, float>::value, "8-point loads are FP32 or FP16");
      const float4 a = ((const float4*)p)[2 * q], b = ((const float4*)p)[2 * q + 1];
      o[0] = a.x;
      o[1] = a.y;
      o[2] = a.z;
      o[3] = a.w;
      o[4] = b.x;
      o[5] = b.y;
      o[6] = b.z;
      o[7] = b.w;
    }
  } else {
    static_assert(std::is_same<S, __half>::value && std::is_same<T, float>::value, "FP16 storage, FP32 arithmetic");
    if constexpr (P == 1) {
      o[0] = __half2float(p[q]);
    } else if constexpr (P == 2) {
      const float2 a = __half22float2(((const __half2*)p)[q]);
      o[0] = a.x;
      o[1] = a.y;
    } else {
      static_assert(P == 4, "FP16 loads are 1, 2 or 4 points");
      const uint2 raw = ((const uint2*)p)[q];
      const float2 a = __half22float2(*(const __half2*)&raw.x), b = __half22float2(*(const __half2*)&raw.y);
      o[0] = a.x;
      o[1] = a.y;
      o[2] = b.x;
      o[3] = b.y;
    }
  }
}

// The store matching ldpts: values rounded to S (round to nearest even).
template <typename T, int P, typename S>
__device__ __forceinline__ void stpts(S* p, int64_t q, const T* v) {
  if constexpr (std::is_same<S, T>::value) {
    if constexpr (P == 1) {
      p[q] = v[0];
    } else if constexpr (P == 2) {
      ((typename V2<T>::t*)p)[q] = typename V2<T>::t{v[0], v[1]};
    } else if constexpr (P == 4) {
      ((float4*)p)[q] = float4{v[0], v[1], v[2], v[3]};
    } else {
      static_assert(P == 8, "stores of 1, 2, 4 or 8 points");
      ((float4*)p)[2 * q] = float4{v[0], v[1], v[2], v[3]};
      ((float4*)p)[2 * q + 1] = float4{v[4], v[5], v[6], v[7]};
    }
  } else {
    if constexpr (P == 1) {
      p[q] = __float2half_rn(v[0]);
    } else if constexpr (P == 2) {
      ((__half2*)p)[q] = __floats2half2_rn(v[0], v[1]);
    } else if constexpr (P == 4) {
      const __half2 a = __floats2half2_rn(v[0], v[1]), b = __floats2half2_rn(v[2], v[3]);
      uint2 raw;
      raw.x = *(const uint32_t*)&a;
      raw.y = *(const uint32_t*)&b;
      ((uint2*)p)[q] = raw;
    } else {
      static_assert(P == 8, "stores of 1, 2, 4 or 8 points");
      const __half2 a = __floats2half2_rn(v[0], v[1]), b = __floats2half2_rn(v[2], v[3]);
      const __half2 c = __floats2half2_rn(v[4], v[5]), d = __floats2half2_rn(v[6], v[7]);
      uint4 raw;
      raw.x = *(const uint32_t*)&a;
      raw.y = *(const uint32_t*)&b;
      raw.z = *(const uint32_t*)&c;
      raw.w = *(const uint32_t*)&d;
      ((uint4*)p)[q] = raw;
    }
  }
}

// P points of one plane held in registers as loaded: widened on use (get), so that an FP16
// basis takes one register per two points.
template <typename T, int P, typename S>
struct PtsReg {
  T v[P];
  __device__ __forceinline__ void load(const S* p, int64_t q) { ldpts<T, P, S>(p, q, v); }
  __device__ __forceinline__ T get(int k) const { return v[k]; }
};
template <>
struct PtsReg<float, 1, __half> {
  __half r;
  __device__ __forceinline__ void load(const __half* p, int64_t q) { r = p[q]; }
  __device__ __forceinline__ float get(int) const { return __half2float(r); }
};
template <>
struct PtsReg<float, 4, __half> {
  uint2 r;
  __device__ __forceinline__ void load(const __half* p, int64_t q) { r = ((const uint2*)p)[q]; }
  __device__ __forceinline__ float get(int k) const {
    const __half2 h = *(const __half2*)(k < 2 ? &r.x : &r.y);
    return (k & 1) ? __high2float(h) : __low2float(h);
  }
};
template <>
struct PtsReg<float, 8, __half> {
  uint4 r;
  __device__ __forceinline__ void load(const __half* p, int64_t q) { r = ((const uint4*)p)[q]; }
  __device__ __forceinline__ float get(int k) const {
    const uint32_t w = k < 2 ? r.x : k < 4 ? r.y : k < 6 ? r.z : r.w;
    const __half2 h = *(const __half2*)&w;
    return (k & 1) ? __high2float(h) : __low2float(h);
  }
};
template <>
struct PtsReg<float, 2, __half> {
  __half2 r;
  __device__ __forceinline__ void load(const __half* p, int64_t q) { r = ((const __half2*)p)[q]; }
  __device__ __forceinline__ float get(int k) const { return k == 0 ? __low2float(r) : __high2float(r); }
};

// x rounded to the storage type S and back (x itself when S is the arithmetic type).
template <typename T, typename S>
__device__ __forceinline__ T round_to(T x) {
  if constexpr (std::is_same<S, T>::value)
    return x;
  else
    return __half2float(__float2half_rn(x));
}

// The warp's sums of M values per lane (M a power of two up to 32): value c in lane c (and c + M, ...).
// Each exchange halves the values a lane is left with: M - 1 additions and a few for M < 32,
// instead of 5 M (in FP64 an addition takes a warp's scheduler 64 cycles: 35 sums by five additions
// each were 12 us per block of a reduction pass).
template <typename T, int M>
__device__ __forceinline__ T warp_sums(T (&r)[M], int lane) {
#pragma unroll
  for (int h = M / 2; h > 0; h /= 2) {
    const bool up = lane & h;
#pragma unroll
    for (int c = 0; c < h; ++c) {
      const T give = up ? r[c] : r[c + h], keep = up ? r[c + h] : r[c];
      r[c] = keep + __shfl_xor_sync(0xffffffffu, give, h);
    }
  }
  T v = r[0];
#pragma unroll
  for (int o = M; o < 32; o *= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// One reduction pass over the basis V_0..V_{count-1}, u and (optionally) w.  Per block:
//   s_i = sum conj(V_i) u,  t_i = sum conj(V_i) w  (i < count),
//   a = sum |u|^2,  b = sum conj(u) w.
// Partial layout per block (ncol = 4 count + 3 doubles): s (2 count), t (2 count), a, b (2).
// The basis is stored in TV (T, or FP16 holding vscale V_i with vscale a power of two), so
// the s and t sums are multiplied by vinv = 1 / vscale in the block epilogue.
// The block's warps form G = 1, 2, 4 or 8 groups (the fewest with at most CH basis vectors
// each); all groups walk the same points, each reducing its own share of the basis, so u
// and w come from DRAM once (the other groups' loads of them hit L1) however many vectors
// there are.  More than G * CH vectors (restarts beyond 32) take further rounds.  At the
// end of a round every accumulator is reduced by warp shuffles and one shared-memory
// exchange.
template <typename T, int PTS, typename TV, int CH>
__global__ void __launch_bounds__(RB, 2) dcgs_dot_kernel(const TV* __restrict__ V, int64_t vs, int count,
                                                         const T* __restrict__ u, const T* __restrict__ w,
                                                         int64_t N, double* __restrict__ partial, double vinv) {
  constexpr int NW = RB / 32;
  constexpr int NACC = 4 * CH + 3;
  __shared__ T sh[NW][NACC];
  const int ncol = 4 * count + 3;
  const bool hw = (w != nullptr);
  const int64_t npts = N / PTS;
  double* out = partial + (int64_t)blockIdx.x * ncol;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int G = 1;
  while (G < NW && (count + G - 1) / G > CH) G *= 2;
  const int wpg = NW / G;                     // warps per group
  const int grp = warp / wpg;
  const int tig = (warp % wpg) * 32 + lane;   // thread within the group
  const int64_t tpg = (int64_t)wpg * 32;
  const int64_t stride = (int64_t)gridDim.x * tpg;
  const int nround = count > 0 ? (count + G * CH - 1) / (G * CH) : 1;
  for (int rd = 0; rd < nround; ++rd) {
    const int rbase = rd * G * CH;
    const int rcount = min(G * CH, count - rbase);
    // group g reduces vectors [g rcount / G, (g + 1) rcount / G) of the round: shares
    // differ by at most one, the larger ones last (group 0 also forms a and b)
    const int base = rbase + grp * rcount / G;
    const int nc = rbase + (grp + 1) * rcount / G - base;
    const bool own = (rd == 0 && grp == 0);   // this group also forms a and b
    T acc[NACC];
#pragma unroll
    for (int c = 0; c < NACC; ++c) acc[c] = T(0);
    for (int64_t q = (int64_t)blockIdx.x * tpg + tig; q < npts; q += stride) {
      T ur[PTS], ui[PTS], wr[PTS], wi[PTS];
      ldpts<T, PTS, T>(u, q, ur);
      ldpts<T, PTS, T>(u + N, q, ui);
#pragma unroll
      for (int k = 0; k < PTS; ++k) wr[k] = wi[k] = T(0);
      if (hw) {
        ldpts<T, PTS, T>(w, q, wr);
        ldpts<T, PTS, T>(w + N, q, wi);
      }
      PtsReg<T, PTS, TV> vr[CH], vi[CH];
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        if (c < nc) {
          const TV* v = V + (int64_t)(base + c) * vs;
          vr[c].load(v, q);
          vi[c].load(v + N, q);
        }
      }
      if (own) {
#pragma unroll
        for (int k = 0; k < PTS; ++k) {
          acc[4 * CH] = fmx(ur[k], ur[k], fmx(ui[k], ui[k], acc[4 * CH]));
          acc[4 * CH + 1] = fmx(ur[k], wr[k], fmx(ui[k], wi[k], acc[4 * CH + 1]));
          acc[4 * CH + 2] = fmx(ur[k], wi[k], fmx(-ui[k], wr[k], acc[4 * CH + 2]));
        }
      }
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        if (c < nc) {
#pragma unroll
          for (int k = 0; k < PTS; ++k) {
            const T a = vr[c].get(k), b = vi[c].get(k);
            acc[4 * c] = fmx(a, ur[k], fmx(b, ui[k], acc[4 * c]));
            acc[4 * c + 1] = fmx(a, ui[k], fmx(-b, ur[k], acc[4 * c + 1]));
            acc[4 * c + 2] = fmx(a, wr[k], fmx(b, wi[k], acc[4 * c + 2]));
            acc[4 * c + 3] = fmx(a, wi[k], fmx(-b, wr[k], acc[4 * c + 3]));
          }
        }
      }
    }
    {
      constexpr int M = 4 * CH <= 4 ? 4 : 4 * CH <= 8 ? 8 : 4 * CH <= 16 ? 16 : 32;
      T r[M];
#pragma unroll
      for (int c = 0; c < M; ++c) r[c] = c < 4 * CH ? acc[c] : T(0);
      const T v = warp_sums<T, M>(r, lane);
      if (lane < 4 * CH) sh[warp][lane] = v;
      if (own) {
#pragma unroll
        for (int c = 4 * CH; c < NACC; ++c) {
          T v3 = acc[c];
          for (int o = 16; o > 0; o >>= 1) v3 += __shfl_xor_sync(0xffffffffu, v3, o);
          if (lane == 0) sh[warp][c] = v3;
        }
      } else if (lane < 3) {
        sh[warp][4 * CH + lane] = T(0);
      }
    }
    __syncthreads();
    // group gg's sums over its wpg warps; column c of its accumulators
    for (int e = threadIdx.x; e < G * NACC; e += blockDim.x) {
      const int gg = e / NACC, c = e - gg * NACC;
      double sum = 0.0;
      for (int ww = 0; ww < wpg; ++ww) sum += (double)sh[gg * wpg + ww][c];
      const int gbase = rbase + gg * rcount / G;
      const int gnc = rbase + (gg + 1) * rcount / G - gbase;
      if (c < 4 * CH) {
        const int cc = c >> 2, kind = c & 3;
        if (cc < gnc) out[(kind < 2 ? 0 : 2 * count) + 2 * (gbase + cc) + (kind & 1)] = sum * vinv;
      } else if (rd == 0 && gg == 0) {
        out[4 * count + (c - 4 * CH)] = sum;
      }
    }
    __syncthreads();
  }
}

// x cut to 24 bits, by integer operations (a conversion takes the FP64 pipe as long as a product);
// |x| < 2^127, below 2^-126: 0.
__device__ __forceinline__ float cut32(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), m = (hi & 0x7fffffffu) - 0x38000000u;  // exponent bias 1023 -> 127
  const uint32_t f = __funnelshift_l((uint32_t)__double2loint(x), m, 3);
  return __uint_as_float((int)m < 0x00100000 ? 0u : (f | (hi & 0x80000000u)));
}

// One update pass.  coef (complex double unless noted): s[count], t[count], c, inv (real).
//   v_new = (u - sum_i V_i s_i) inv          -> written to v_out (the basis slot `count`)
//   u     = (w - sum_i V_i t_i - v_new c) inv -> written over u (in place)
// With the basis stored in FP16 as vscale V_i, the coefficients are divided by vscale, v_out
// receives vscale v_new rounded to FP16, and the correction of u uses that rounded vector,
// so that u is orthogonalised against the basis as stored.  PTS points per thread; the basis
// is read UB vectors at a time, all loads of a group issued before its FMAs.
//
// FP64 arithmetic is bound by the FP64 pipe, eight operations per point and vector.  Half of them
// form sum_i V_i s_i, the correction of a vector that is orthogonal to the basis up to rounding
// already: |s_i| is around 2^-52 of the vector.  Where every |s_i| is below 2^-36 of it (else
// the general form runs), that sum is formed in FP32 from the vectors' leading 24 bits, cut by
// integer operations, and taken from u once: a term's error is below 2^-23 2^-36 of the vector,
// where the general form rounds u itself (2^-53) with every term.  FP32's exponents reach all that
// counts for alpha from 2^-64 to 2^64 (other alpha, and a breakdown: the general form).  Error of v
// against extended precision, in 2^-53 |u|, largest of 4096 points: 1.6 with 30 and with 64 vectors, the
// general form 12 and 20.  192^3 FP64 GMRES: 908 -> 667 us.
template <typename T, int PTS, typename TV, int UB = 8>
__global__ void __launch_bounds__(RB) dcgs_update_kernel(const TV* __restrict__ V, int64_t vs, int count,
                                                         T* u, const T* __restrict__ w, TV* __restrict__ v_out,
                                                         int64_t N, const double* __restrict__ coef, double vscale) {
  __shared__ T s_r[64], s_i[64], t_r[64], t_i[64];
  __shared__ T cc[3];
  const double vinv = 1.0 / vscale;
  for (int c = threadIdx.x; c < count; c += blockDim.x) {
    s_r[c] = (T)(coef[2 * c] * vinv);
    s_i[c] = (T)(coef[2 * c + 1] * vinv);
    t_r[c] = (T)(coef[2 * count + 2 * c] * vinv);
    t_i[c] = (T)(coef[2 * count + 2 * c + 1] * vinv);
  }
  if (threadIdx.x == 0) {
    cc[0] = (T)coef[4 * count];
    cc[1] = (T)coef[4 * count + 1];
    cc[2] = (T)coef[4 * count + 2];
  }
  bool low = false;  // the correction of u is small enough for FP32
  __shared__ float s32[sizeof(T) == 8 ? 64 : 1][2];
  if constexpr (sizeof(T) == 8) {
    const double alpha = 1.0 / coef[4 * count + 2];
    bool ok = alpha >= 5.421010862427522e-20 && alpha <= 18446744073709551616.0;  // 2^-64 .. 2^64
    for (int c = threadIdx.x; c < count; c += blockDim.x) {
      ok = ok && fabs(s_r[c]) + fabs(s_i[c]) < 1.4551915228366852e-11 * alpha;  // 2^-36
      s32[c][0] = (float)s_r[c];
      s32[c][1] = (float)s_i[c];
    }
    low = __syncthreads_and(ok);
  }
  __syncthreads();
  const T cr = cc[0], ci = cc[1], inv = cc[2];
  const T vsc = (T)vscale, vin = (T)vinv;  // powers of two: exact in T
  const int64_t npts = N / PTS;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < npts; q += stride) {
    T ur[PTS], ui[PTS], wr[PTS], wi[PTS];
    ldpts<T, PTS, T>(u, q, ur);
    ldpts<T, PTS, T>(u + N, q, ui);
    ldpts<T, PTS, T>(w, q, wr);
    ldpts<T, PTS, T>(w + N, q, wi);
    float fr[sizeof(T) == 8 ? PTS : 1], fi[sizeof(T) == 8 ? PTS : 1];  // low: the correction of u
    if constexpr (sizeof(T) == 8)
#pragma unroll
      for (int k = 0; k < PTS; ++k) fr[k] = fi[k] = 0.f;
    for (int c0 = 0; c0 < count; c0 += UB) {
      PtsReg<T, PTS, TV> vr[UB], vi[UB];
#pragma unroll
      for (int e = 0; e < UB; ++e) {
        if (c0 + e < count) {
          const TV* v = V + (int64_t)(c0 + e) * vs;
          vr[e].load(v, q);
          vi[e].load(v + N, q);
        }
      }
      if constexpr (sizeof(T) == 8) {
        if (low) {
#pragma unroll
          for (int e = 0; e < UB; ++e) {
            if (c0 + e < count) {
              const int c = c0 + e;
              const float sr = s32[c][0], si = s32[c][1];
#pragma unroll
              for (int k = 0; k < PTS; ++k) {
                const double a = vr[e].get(k), b = vi[e].get(k);
                const float a32 = cut32(a), b32 = cut32(b);
                fr[k] = fmaf(-a32, sr, fmaf(b32, si, fr[k]));
                fi[k] = fmaf(-a32, si, fmaf(-b32, sr, fi[k]));
                wr[k] = fma(-a, t_r[c], fma(b, t_i[c], wr[k]));
                wi[k] = fma(-a, t_i[c], fma(-b, t_r[c], wi[k]));
              }
            }
          }
          continue;
        }
      }
#pragma unroll
      for (int e = 0; e < UB; ++e) {
        if (c0 + e < count) {
          const int c = c0 + e;
#pragma unroll
          for (int k = 0; k < PTS; ++k) {
            const T a = vr[e].get(k), b = vi[e].get(k);
            ur[k] = fmx(-a, s_r[c], fmx(b, s_i[c], ur[k]));
            ui[k] = fmx(-a, s_i[c], fmx(-b, s_r[c], ui[k]));
            wr[k] = fmx(-a, t_r[c], fmx(b, t_i[c], wr[k]));
            wi[k] = fmx(-a, t_i[c], fmx(-b, t_r[c], wi[k]));
          }
        }
      }
    }
    if constexpr (sizeof(T) == 8)
#pragma unroll
      for (int k = 0; k < PTS; ++k) {  // (zero in the general form)
        ur[k] += (double)fr[k];
        ui[k] += (double)fi[k];
      }
    T nr[PTS], ni[PTS];
#pragma unroll
    for (int k = 0; k < PTS; ++k) {
      nr[k] = ur[k] * inv * vsc;
      ni[k] = ui[k] * inv * vsc;
    }
    stpts<T, PTS, TV>(v_out, q, nr);
    stpts<T, PTS, TV>(v_out + N, q, ni);
#pragma unroll
    for (int k = 0; k < PTS; ++k) {
      const T a = round_to<T, TV>(nr[k]) * vin, b = round_to<T, TV>(ni[k]) * vin;
      wr[k] = fmx(-a, cr, fmx(b, ci, wr[k])) * inv;
      wi[k] = fmx(-a, ci, fmx(-b, cr, wi[k])) * inv;
    }
    stpts<T, PTS, T>(u, q, wr);
    stpts<T, PTS, T>(u + N, q, wi);
  }
}

// ---- FP64 small algebra ----
// An FP64 instruction of one warp takes its scheduler 64 cycles on GB300 whether one lane works or
// 32 do, so the kernels below spread every product over lanes and warps and keep the serial part
// to a few dozen instructions.
struct zc {
  double re, im;
};
__device__ __forceinline__ zc ld(const double* p) { return zc{p[0], p[1]}; }
__device__ __forceinline__ void st(double* p, zc v) { p[0] = v.re; p[1] = v.im; }
__device__ __forceinline__ zc zmul(zc a, zc b) { return zc{a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ zc zfma(zc a, zc b, zc c) {
  return zc{fma(a.re, b.re, fma(-a.im, b.im, c.re)), fma(a.re, b.im, fma(a.im, b.re, c.im))};
}

constexpr int STEP_MAXJ = 64;  // largest restart length (helm6_opts.max_restart <= 64)
constexpr int STEP_W = RB / 32;

// One delayed Gram-Schmidt Arnoldi step j: column sums of the reduction's partials (block c sums
// column c), then, in the block that finishes last, the step's algebra.
// red: s_i = V_i^H u_j, t_i = V_i^H w (i < j), a = ||u_j||^2, b = u_j^H w.
// u_j = V s + alpha v_j with alpha^2 = a - ||s||^2.
//   * column j-1 of the raw Hessenberg Hr gets += s and subdiagonal alpha; its rotated form goes
//     to R.  The rotations so far are kept as their product Q (row r reaches columns 0..r+1), so
//     that the column is rotated by one matrix-vector product instead of j dependent rotations;
//     the new rotation zeroes the subdiagonal and gives the residual estimate *est = |g_j|
//     (j = 0: g_0 = alpha);
//   * with w = A M^{-1} u_j (has_w): v_j^H w = (b - s^H t)/alpha = c_j, column j of Hr is
//     ([t; c_j] - Hr[:, 0..j-1] s)/alpha, and T (z_l = sum_i T[i,l] z~_i) gets column
//     (e_j - T s)/alpha;
//   * coef = [s, t, c_j, 1/alpha] for the update pass v_j = (u - V s)/alpha,
//     u_{j+1} = (w - V t - v_j c_j)/alpha;
//   * gc (device-driven solves): iteration count, history, and whether step j + 1 runs.
// *brk = 1 when alpha^2 <= 1e-28 a (u_j in the span of the basis: breakdown).
// One launch in place of three (column sums, algebra on one thread's rotations, control): 37 -> 14 us
// per step at restart length 30, 22 -> 9 us on the small grids' first steps.
__global__ void __launch_bounds__(RB) dcgs_step_kernel(int j, int has_w, const double* __restrict__ partial, int nblocks,
                                                       double* red, StepMem a, GraphCtl* gc, int m,
                                                       cudaGraphConditionalHandle next) {
  __shared__ double sh[STEP_W];
  __shared__ bool last;
  const int ncols = 4 * j + 3, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  {
    const int c = blockIdx.x;
    double v = 0.0;
    for (int b = tid; b < nblocks; b += RB) v += partial[(int64_t)b * ncols + c];
    v = block_sum(v, sh);
    if (tid == 0) {
      red[c] = v;
      __threadfence();
      last = atomicAdd(a.count, 1u) == (unsigned)ncols - 1u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (tid == 0) *a.count = 0u;
  }
  // partial products of warp w: rows by lane, the columns w, w + 8, ...
  __shared__ zc sp[3][STEP_W][STEP_MAXJ + 1];
  __shared__ zc ss[STEP_MAXJ + 1], st_[STEP_MAXJ + 1], sh_[STEP_MAXJ + 1];  // s, t, corrected column j - 1
  __shared__ zc srot[STEP_MAXJ + 1];
  __shared__ double ssum[3], sal[3];  // ||s||^2, s^H t; alpha, 1 / alpha, breakdown
  volatile double* vr = red;
  const int ldh = a.ldh;
  if (tid < j) {
    const zc sv{vr[2 * tid], vr[2 * tid + 1]}, tv{vr[2 * j + 2 * tid], vr[2 * j + 2 * tid + 1]};
    ss[tid] = sv;
    st_[tid] = tv;
    a.coef[2 * tid] = sv.re;
    a.coef[2 * tid + 1] = sv.im;
    a.coef[2 * j + 2 * tid] = tv.re;
    a.coef[2 * j + 2 * tid + 1] = tv.im;
    const zc h = ld(a.Hr + 2 * ((int64_t)(j - 1) * ldh + tid));
    sh_[tid] = zc{h.re + sv.re, h.im + sv.im};
  }
  __syncthreads();
  // ||s||^2 (warp 0), s^H t (warps 1 and 2)
  if (warp < 3) {
    double v = 0.0;
    for (int i = lane; i < j; i += 32) {
      const zc q = ss[i], t = st_[i];
      v = warp == 0 ? fma(q.re, q.re, fma(q.im, q.im, v))
                    : warp == 1 ? fma(q.re, t.re, fma(q.im, t.im, v)) : fma(q.re, t.im, fma(-q.im, t.re, v));
    }
    v = warp_sum(v);
    if (lane == 0) ssum[warp] = v;
  }
  const zc z0{0.0, 0.0};
  for (int r = lane; r < j; r += 32) {
    zc q = z0, h = z0, t = z0;
    for (int i = warp; i < j; i += STEP_W) {
      // Q row r reaches column r + 1, Hr is Hessenberg (row r from column r - 1), T upper triangular
      if (i <= r + 1) q = zfma(ld(a.Q + 2 * ((int64_t)i * ldh + r)), sh_[i], q);
      if (has_w && i >= r - 1) h = zfma(i == j - 1 ? sh_[r] : ld(a.Hr + 2 * ((int64_t)i * ldh + r)), ss[i], h);
      if (has_w && a.T && i >= r) t = zfma(ld(a.T + 2 * ((int64_t)i * a.ldt + r)), ss[i], t);
    }
    sp[0][warp][r] = q;
    sp[1][warp][r] = h;
    sp[2][warp][r] = t;
  }
  __syncthreads();
  if (tid == RB - 1) {
    const double av = vr[4 * j], al2 = av - (j > 0 ? ssum[0] : 0.0);
    const bool bd = !(al2 > 1e-28 * fmax(av, 1e-300)) || !isfinite(al2);
    const double inv = bd ? 0.0 : rsqrt(al2);
    sal[0] = bd ? 0.0 : al2 * inv;
    sal[1] = inv;
    sal[2] = bd ? 1.0 : 0.0;
    *a.brk = bd ? 1 : 0;
  }
  // the eight warps' products of row r: threads 0..63 Q, 64..127 Hr, 128..191 T
  {
    const int k = tid >> 6;
    if (k < 3)
      for (int r = tid & 63; r < j; r += 64) {
        zc v = z0;
        for (int w = 0; w < STEP_W; ++w) {
          v.re += sp[k][w][r].re;
          v.im += sp[k][w][r].im;
        }
        if (k == 0) srot[r] = v;
        else sp[k][0][r] = v;
      }
  }
  __syncthreads();
  const double al = sal[0], inv = sal[1];
  const bool bd = sal[2] != 0.0;
  const bool run = has_w && !bd;
  // ([t; c_j] - Hr s) / alpha and (e_j - T s) / alpha; rows 0..j - 1 (row j of Hr s is alpha s_{j-1})
  if (run && tid >= 64) {
    const int k = tid >> 6;
    if (k == 1)
      for (int r = tid & 63; r < j; r += 64) {
        const zc t = st_[r], h = sp[1][0][r];
        st(a.Hr + 2 * ((int64_t)j * ldh + r), zc{(t.re - h.re) * inv, (t.im - h.im) * inv});
      }
    else if (k == 2 && a.T)
      for (int r = tid & 63; r < j; r += 64) {
        const zc t = sp[2][0][r];
        st(a.T + 2 * ((int64_t)j * a.ldt + r), zc{-t.re * inv, -t.im * inv});
      }
  }
  if (tid == RB - 1) {
    zc cj = z0;
    if (run) {
      cj = zc{(vr[4 * j + 1] - (j > 0 ? ssum[1] : 0.0)) * inv, (vr[4 * j + 2] - (j > 0 ? ssum[2] : 0.0)) * inv};
      zc h = cj;
      if (j > 0) {
        h.re = fma(-al, ss[j - 1].re, h.re);
        h.im = fma(-al, ss[j - 1].im, h.im);
      }
      st(a.Hr + 2 * ((int64_t)j * ldh + j), zc{h.re * inv, h.im * inv});
      if (a.T) st(a.T + 2 * ((int64_t)j * a.ldt + j), zc{inv, 0.0});
    }
    a.coef[4 * j] = cj.re;
    a.coef[4 * j + 1] = cj.im;
    a.coef[4 * j + 2] = inv;
  }
  if (j == 0) {
    if (tid == 0) {
      st(a.g, zc{al, 0.0});
      st(a.Q, zc{1.0, 0.0});
      *a.est = al;
    }
  } else if (warp == 0) {
    // the rotation [c s; -conj(s) c] that takes (x, alpha) to (., 0)
    const int jj = j - 1;
    const zc x = srot[jj];
    const double nx = fma(x.re, x.re, x.im * x.im), n2 = fma(al, al, nx);
    double c;
    zc s;
    if (nx > 1e-290 && n2 < 1e290) {
      const double rx = rsqrt(nx), r2 = rsqrt(n2), f = al * rx * r2;
      c = nx * rx * r2;
      s = zc{x.re * f, x.im * f};
    } else {
      const double ax = hypot(x.re, x.im), den = hypot(ax, al);
      if (den == 0.0) {
        c = 1.0;
        s = z0;
      } else if (ax == 0.0) {
        c = 0.0;
        s = zc{1.0, 0.0};
      } else {
        c = ax / den;
        s = zc{x.re / ax * (al / den), x.im / ax * (al / den)};
      }
    }
    double* rc = a.R + 2 * (int64_t)jj * ldh;
    if (lane == 0) {
      st(rc + 2 * jj, zc{fma(c, x.re, s.re * al), fma(c, x.im, s.im * al)});
      st(rc + 2 * j, z0);
      const zc gj = ld(a.g + 2 * jj), gn = zmul(zc{-s.re, s.im}, gj);
      st(a.g + 2 * j, gn);
      st(a.g + 2 * jj, zc{c * gj.re, c * gj.im});
      *a.est = sqrt(fma(gn.re, gn.re, gn.im * gn.im));
    }
    for (int i = lane; i < jj; i += 32) st(rc + 2 * i, srot[i]);
    // rows jj and j of Q: [c s; -conj(s) c] times (row jj, e_j)
    for (int i = lane; i <= j; i += 32) {
      double* q = a.Q + 2 * (int64_t)i * ldh;
      if (i < j) {
        const zc o = ld(q + 2 * jj);
        st(q + 2 * jj, zc{c * o.re, c * o.im});
        st(q + 2 * j, zmul(zc{-s.re, s.im}, o));
      } else {
        st(q + 2 * jj, s);
        st(q + 2 * j, zc{c, 0.0});
      }
    }
    // the corrected column of the raw matrix
    double* hc = a.Hr + 2 * (int64_t)jj * ldh;
    for (int i = lane; i <= j; i += 32) st(hc + 2 * i, i < j ? sh_[i] : zc{al, 0.0});
    __syncwarp();
  }
  if (gc && tid == 0) {
    const double e = *a.est;
    bool stop;
    if (j == 0) {
      stop = bd || !isfinite(e);
    } else {
      gc->iters++;
      if (gc->nhist < HELM6_MAX_HIST) gc->hist[gc->nhist++] = e * gc->beta / gc->normF;
      stop = !(e > gc->itol) || !isfinite(e) || bd || j >= m || gc->iters >= gc->maxit;
    }
    if (stop) gc->k = j;
    if (j < m) cudaGraphSetConditional(next, stop ? 0u : 1u);
  }
}

// y = R^-1 g (R upper triangular, column-major), one step per column: lane r keeps row r's
// right side, the lane of the column divides and broadcasts; then q = T y, rows by lane and columns
// by warp.  The next column is requested before the current one is used.
__global__ void __launch_bounds__(RB) ls_solve_kernel(const double* __restrict__ R, int ldh, int j,
                                                      const double* __restrict__ g, double* y,
                                                      const double* __restrict__ T, int ldt, double* q,
                                                      const int* j_dev) {
  __shared__ zc sy[STEP_MAXJ], sp[STEP_W][STEP_MAXJ];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (j_dev) j = *j_dev;
  const zc z0{0.0, 0.0};
  if (warp == 0) {
    constexpr int RR = STEP_MAXJ / 32;  // rows of a lane
    zc acc[RR], di[RR], cur[RR], nxt[RR];
    auto column = [&](int c, zc(&o)[RR]) {
#pragma unroll
      for (int k = 0; k < RR; ++k) o[k] = c >= 0 && lane + 32 * k < c ? ld(R + 2 * ((int64_t)c * ldh + lane + 32 * k)) : z0;
    };
#pragma unroll
    for (int k = 0; k < RR; ++k) {
      const int r = lane + 32 * k;
      acc[k] = di[k] = z0;
      if (r < j) {
        acc[k] = ld(g + 2 * r);
        const zc d = ld(R + 2 * ((int64_t)r * ldh + r));
        const double n2 = d.re * d.re + d.im * d.im;
        if (n2 > 0.0) di[k] = zc{d.re / n2, -d.im / n2};
      }
    }
    column(j - 1, cur);
    for (int c = j - 1; c >= 0; --c) {
      column(c - 1, nxt);
#pragma unroll
      for (int k = 0; k < RR; ++k)
        if (c >> 5 == k && lane == (c & 31)) {
          const zc v = zmul(acc[k], di[k]);
          sy[c] = v;
          st(y + 2 * c, v);
        }
      __syncwarp();
      const zc v{-sy[c].re, -sy[c].im};
#pragma unroll
      for (int k = 0; k < RR; ++k) {
        if (32 * k < c) acc[k] = zfma(cur[k], v, acc[k]);
        cur[k] = nxt[k];
      }
    }
  }
  __syncthreads();
  if (!T) return;
  for (int r = lane; r < j; r += 32) {
    zc v = z0;
    for (int i = warp; i < j; i += STEP_W)
      if (i >= r) v = zfma(ld(T + 2 * ((int64_t)i * ldt + r)), sy[i], v);
    sp[warp][r] = v;
  }
  __syncthreads();
  for (int r = threadIdx.x; r < j; r += RB) {
    zc v = z0;
    for (int w = 0; w < STEP_W; ++w) {
      v.re += sp[w][r].re;
      v.im += sp[w][r].im;
    }
    st(q + 2 * r, v);
  }
}

// y (+)= alpha * x over 2N reals (accumulate = 0: y = alpha * x)
template <typename TI, typename TO>
__global__ void axpy_kernel(const TI* __restrict__ x, TO* __restrict__ y, int64_t n2, double alpha) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n2; idx += stride)
    y[idx] += (TO)(alpha * (double)x[idx]);
}

int grid_for(int64_t n, int bs) {
  static int sms = 0;
  if (!sms) sms = device_sm_count();
  int64_t g = (n + bs - 1) / bs;
  const int64_t cap = (int64_t)sms * 8;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

static std::atomic<long long> g_launches{0};
void note_launch(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
long long launch_total() { return g_launches.load(std::memory_order_relaxed); }

int current_device() {
  int d = -1;
  return cudaGetDevice(&d) == cudaSuccess ? d : -1;
}

int device_sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}

template <typename T>
void launch_sumsq(const T* x, int64_t N, double* partial, int nblocks, cudaStream_t s) {
  note_launch();
  sumsq_kernel<T><<<nblocks, RB, 0, s>>>(x, N, partial);
}

template <typename T>
void launch_scale_copy(const T* x, T* y, int64_t N, const double* inv_dev, double host_scale,
                       cudaStream_t s) {
  note_launch();
  scale_copy_kernel<T><<<grid_for(2 * N, RB), RB, 0, s>>>(x, y, 2 * N, inv_dev, host_scale);
}

template <typename TI, typename TO>
void launch_lincomb(const TI* V, int64_t vstride, int count, const double* y, double scale, TO* out,
                    int64_t N, int accumulate, cudaStream_t s, const int* count_dev, const double* scale_dev) {
  note_launch();
  if ((N & 1) == 0 && (vstride & 1) == 0)
    lincomb_kernel<TI, TO, true><<<grid_for(N / 2, RB), RB, 0, s>>>(V, vstride, count, y, scale, out, N, accumulate,
                                                                      count_dev, scale_dev);
  else
    lincomb_kernel<TI, TO, false><<<grid_for(N, RB), RB, 0, s>>>(V, vstride, count, y, scale, out, N, accumulate,
                                                                   count_dev, scale_dev);
}

template <typename TI, typename TO>
void launch_convert(const TI* x, TO* y, int64_t N, double scale, cudaStream_t s, const double* scale_dev) {
  note_launch();
  convert_kernel<TI, TO><<<grid_for(2 * N, RB), RB, 0, s>>>(x, y, 2 * N, scale, scale_dev);
}

void launch_interleaved_to_planar(const double* zin, double* out, int64_t N, cudaStream_t s) {
  note_launch();
  inter_to_planar_kernel<<<grid_for(N, RB), RB, 0, s>>>((const double2*)zin, out, N);
}

void launch_planar_to_interleaved(const double* in, double* zout, int64_t N, cudaStream_t s) {
  note_launch();
  planar_to_inter_kernel<<<grid_for(N, RB), RB, 0, s>>>(in, (double2*)zout, N);
}

void launch_caller_to_planar(const Geom& g, int xaxis, const double* zin, double* out, cudaStream_t s) {
  if (xaxis < 0) {
    launch_interleaved_to_planar(zin, out, g.N, s);
    return;
  }
  note_launch();
  inter_to_planar_x_kernel<<<grid_for(g.N, RB), RB, 0, s>>>((const double2*)zin, out, g.mx, g.my, g.mz, xaxis);
}

void launch_planar_to_caller(const Geom& g, int xaxis, const double* in, double* zout, cudaStream_t s) {
  if (xaxis < 0) {
    launch_planar_to_interleaved(in, zout, g.N, s);
    return;
  }
  note_launch();
  planar_to_inter_x_kernel<<<grid_for(g.N, RB), RB, 0, s>>>(in, (double2*)zout, g.mx, g.my, g.mz, xaxis);
}

void launch_reduce_sum(const double* partial, int n, double* out, cudaStream_t s) {
  note_launch();
  reduce_sum_kernel<<<1, RB, 0, s>>>(partial, n, out);
}

void launch_dcgs_step(int j, int has_w, const double* partial, int nblocks, double* red, const StepMem& a, GraphCtl* gc,
                      int m, cudaGraphConditionalHandle next, cudaStream_t s) {
  note_launch();
  dcgs_step_kernel<<<4 * j + 3, RB, 0, s>>>(j, has_w, partial, nblocks, red, a, gc, m, next);
}

void launch_ls_solve(const double* R, int ldh, int j, const double* g, double* y, const double* T, int ldt, double* q,
                     cudaStream_t s, const int* j_dev) {
  note_launch();
  ls_solve_kernel<<<1, RB, 0, s>>>(R, ldh, j, g, y, T, ldt, q, j_dev);
}

__global__ void axpby_kernel(const double* __restrict__ x, double* __restrict__ y, int64_t n, double a, double b) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = fma(a, y[i], b * x[i]);
}

void launch_axpby(const double* x, double* y, int64_t N, double a, double b, cudaStream_t s) {
  note_launch();
  axpby_kernel<<<grid_for(2 * N, RB), RB, 0, s>>>(x, y, 2 * N, a, b);
}

template <typename TI, typename TO>
void launch_axpy(const TI* x, TO* y, int64_t N, double alpha, cudaStream_t s) {
  note_launch();
  axpy_kernel<TI, TO><<<grid_for(2 * N, RB), RB, 0, s>>>(x, y, 2 * N, alpha);
}

template void launch_axpy<float, double>(const float*, double*, int64_t, double, cudaStream_t);
template void launch_axpy<double, double>(const double*, double*, int64_t, double, cudaStream_t);

template <typename T>
int cgs_blocks(int64_t N) {
  static int sms = 0;
  if (!sms) sms = device_sm_count();
  int64_t g = (N + RB - 1) / RB;
  const int64_t cap = (int64_t)sms * 8;
  return (int)std::max<int64_t>(1, std::min(g, cap));
}

// Points per thread of the two Gram-Schmidt passes, as many as the planes' alignment allows
// up to 2 for an FP32 or FP64 basis (one 8- or 16-byte load per plane and vector) and 4 for
// an FP16 one (8-byte basis loads; fewer instructions per byte than 2 points).
template <typename TV>
int cgs_pts(int64_t N, int64_t vs) {
  if (std::is_same<TV, __half>::value && N % 4 == 0 && vs % 4 == 0) return 4;
  return (N % 2 == 0 && vs % 2 == 0) ? 2 : 1;
}

// Vectors per warp group of the 8-point FP16 reduction pass for `count` basis vectors: the
// fewest groups G (a power of two, at most 8) that leave at most 6 vectors to a group, and
// the kernel instance compiled for exactly that share (measured at 256 x 258 x 258: an
// instance sized for more vectors than it gets, or a split into more groups, is slower).
int dot_share(int count) {
  int G = 1;
  while (G < 8 && (count + G - 1) / G > 6) G *= 2;
  return std::max(1, std::min(6, (count + G - 1) / G));
}

template <typename T, typename TV>
void launch_dcgs_dot(const TV* V, int64_t vs, int count, const T* u, const T* w, int64_t N, double* partial,
                     int nblocks, double vscale, cudaStream_t s) {
  note_launch();
  const double vinv = 1.0 / vscale;
  if constexpr (std::is_same<TV, __half>::value) {
    if (N % 8 == 0 && vs % 8 == 0) {
      // 8 points per thread: 16-byte basis loads, twice the bytes in flight of 4 points
      switch (dot_share(count)) {
#define DOT8(CH)                                                                                   \
  case CH:                                                                                         \
    dcgs_dot_kernel<T, 8, TV, CH><<<nblocks, RB, 0, s>>>(V, vs, count, u, w, N, partial, vinv); \
    return;
        DOT8(1) DOT8(2) DOT8(3) DOT8(4) DOT8(5) DOT8(6)
#undef DOT8
      }
    }
    if (cgs_pts<TV>(N, vs) == 4) {
      dcgs_dot_kernel<T, 4, TV, CHD<T>><<<nblocks, RB, 0, s>>>(V, vs, count, u, w, N, partial, vinv);
      return;
    }
  }
  if (cgs_pts<TV>(N, vs) == 2)
    dcgs_dot_kernel<T, 2, TV, CHD<T>><<<nblocks, RB, 0, s>>>(V, vs, count, u, w, N, partial, vinv);
  else
    dcgs_dot_kernel<T, 1, TV, CHD<T>><<<nblocks, RB, 0, s>>>(V, vs, count, u, w, N, partial, vinv);
}

// Blocks of the reduction pass: two per SM (its per-block epilogue favours few blocks).
int dot_blocks() { return 2 * device_sm_count(); }

template <typename T, typename TV>
void launch_dcgs_update(const TV* V, int64_t vs, int count, T* u, const T* w, TV* v_out, int64_t N,
                        const double* coef, int nblocks, double vscale, cudaStream_t s) {
  note_launch();
  const int p = cgs_pts<TV>(N, vs);
  if constexpr (std::is_same<TV, __half>::value) {
    if (N % 8 == 0 && vs % 8 == 0) {
      // 8 points per thread, the basis read 4 vectors at a time (measured best at 256 x 258 x 258)
      dcgs_update_kernel<T, 8, TV, 4><<<nblocks, RB, 0, s>>>(V, vs, count, u, w, v_out, N, coef, vscale);
      return;
    }
    if (p == 4) {
      dcgs_update_kernel<T, 4, TV><<<nblocks, RB, 0, s>>>(V, vs, count, u, w, v_out, N, coef, vscale);
      return;
    }
  }
  if (p == 2)
    dcgs_update_kernel<T, 2, TV><<<nblocks, RB, 0, s>>>(V, vs, count, u, w, v_out, N, coef, vscale);
  else
    dcgs_update_kernel<T, 1, TV><<<nblocks, RB, 0, s>>>(V, vs, count, u, w, v_out, N, coef, vscale);
}

template int cgs_blocks<float>(int64_t);
template int cgs_blocks<double>(int64_t);
#define INST_CGS(T, TV)                                                                              \
  template void launch_dcgs_dot<T, TV>(const TV*, int64_t, int, const T*, const T*, int64_t, double*, int, double, \
                                       cudaStream_t);                                                          \
  template void launch_dcgs_update<T, TV>(const TV*, int64_t, int, T*, const T*, TV*, int64_t, const double*, int, \
                                          double, cudaStream_t);
INST_CGS(float, float)
INST_CGS(float, __half)
INST_CGS(double, double)

#define INST_T(T)                                                                              \
  template void launch_sumsq<T>(const T*, int64_t, double*, int, cudaStream_t);                  \
  template void launch_scale_copy<T>(const T*, T*, int64_t, const double*, double, cudaStream_t);
INST_T(float)
INST_T(double)
template void launch_lincomb<float, double>(const float*, int64_t, int, const double*, double, double*,
                                            int64_t, int, cudaStream_t, const int*, const double*);
template void launch_lincomb<double, double>(const double*, int64_t, int, const double*, double,
                                             double*, int64_t, int, cudaStream_t, const int*, const double*);
template void launch_lincomb<float, float>(const float*, int64_t, int, const double*, double, float*,
                                           int64_t, int, cudaStream_t, const int*, const double*);
template void launch_convert<double, float>(const double*, float*, int64_t, double, cudaStream_t, const double*);
template void launch_convert<float, double>(const float*, double*, int64_t, double, cudaStream_t, const double*);
template void launch_convert<double, double>(const double*, double*, int64_t, double, cudaStream_t, const double*);

// ---- control of device-driven solves (graph with conditional nodes) ----
namespace {

// After a true residual: its norm, the solve's status and whether another cycle follows.
__global__ void gctl_residual_kernel(GraphCtl* g, const double* sumsq, const int* zst, const int* tcerr, int first,
                                     cudaGraphConditionalHandle hw) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const double beta = sqrt(fmax(*sumsq, 0.0));
  if (first) {
    g->iters = 0;
    g->outer = 0;
    g->nhist = 0;
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    g->t0 = t;
    if (g->nhist < HELM6_MAX_HIST) g->hist[g->nhist++] = beta / g->normF;
  } else {
    g->outer++;
    if (g->nhist > 0) g->hist[g->nhist - 1] = beta / g->normF;  // the true residual replaces the estimate
  }
  g->beta = beta;
  int st = -1;
  if (!first && *tcerr) st = HELM6_ERR_CUDA;
  else if (!first && *zst == HELM6_BREAKDOWN) st = HELM6_BREAKDOWN;
  else if (!isfinite(beta)) st = HELM6_NONFINITE;
  else if (beta <= g->tol_abs) st = HELM6_OK;
  else if (g->iters >= g->maxit) st = HELM6_NOT_CONVERGED;
  if (st == -1) {
    g->inv_beta = 1.0 / beta;
    g->itol = fmax(g->inner, g->itol_num / beta);
  } else {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    g->t1 = t;
  }
  g->status = st;
  cudaGraphSetConditional(hw, st == -1 ? 1u : 0u);
}

// A cycle starts: step 0 runs, the later steps only when their predecessor enables them.
__global__ void gctl_cycle_kernel(GraphCtl* g, StepHandles ha, int m) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  g->k = 0;
  for (int j = 0; j <= m; ++j) cudaGraphSetConditional(ha.h[j], j == 0 ? 1u : 0u);
}

}  // namespace

void launch_gctl_residual(GraphCtl* g, const double* sumsq, const int* zst, const int* tcerr, int first,
                          cudaGraphConditionalHandle hw, cudaStream_t s) {
  note_launch();
  gctl_residual_kernel<<<1, 32, 0, s>>>(g, sumsq, zst, tcerr, first, hw);
}
void launch_gctl_cycle(GraphCtl* g, const StepHandles& ha, int m, cudaStream_t s) {
  note_launch();
  gctl_cycle_kernel<<<1, 32, 0, s>>>(g, ha, m);
}
}  // namespace helm6
