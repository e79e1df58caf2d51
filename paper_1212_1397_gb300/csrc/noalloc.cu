// helm6_residual_noalloc: r = F - A u and ||r||^2 without allocating device memory.
//
// For callers that cannot call cudaMalloc (see include/helm6.h): the FP64 stencil kernel works
// directly on the boundary's interleaved complex128 arrays, and its only scratch -- one FP64
// partial sum per thread block -- is the file-scope device array g_noalloc_partials instead of
// library-allocated workspace.
#include <cmath>
#include <mutex>

#include "helm6_internal.h"

namespace helm6 {

namespace {

constexpr int kMaxDevices = 64;

// Block partial sums of |r|^2.  Every GPU that loads the library holds this array until
// the process exits.  Each call writes slots [0, nblocks) before reading them.
static __device__ __align__(256) double g_noalloc_partials[HELM6_NOALLOC_MAX_BLOCKS];

// Device address of g_noalloc_partials per device ordinal, looked up once per device.
double* g_partials_ptr[kMaxDevices] = {};
std::mutex g_setup_mutex;

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__global__ void finish_kernel(const double* __restrict__ partials, int n, double* __restrict__ out) {
  __shared__ double sh[32];
  double v = 0.0;
  for (int b = threadIdx.x; b < n; b += blockDim.x) v += partials[b];
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = (threadIdx.x < blockDim.x / 32) ? sh[threadIdx.x] : 0.0;
    v = warp_sum(v);
    if (threadIdx.x == 0) *out = v;
  }
}

// Device address of the scratch array on the current device (looked up once per device).
int scratch_for_current_device(double** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return HELM6_ERR_CUDA;
  if (dev < 0 || dev >= kMaxDevices) return HELM6_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (!g_partials_ptr[dev]) {
    double* p = nullptr;
    if (cudaGetSymbolAddress((void**)&p, g_noalloc_partials) != cudaSuccess || !p) {
      cudaGetLastError();
      return HELM6_ERR_CUDA;
    }
    g_partials_ptr[dev] = p;
  }
  *out = g_partials_ptr[dev];
  return HELM6_OK;
}

}  // namespace

}  // namespace helm6

using namespace helm6;

extern "C" int helm6_residual_noalloc(int n, double h, helm6_c64 k, const int faces[6], const void* F,
                                      const void* u, void* r, double* sumsq, void* stream) {
  if (!faces || !F || !u || !r || !sumsq || n < 1 || n > 4094) return HELM6_ERR_INVALID;
  for (int a = 0; a < 6; ++a)
    if (faces[a] != HELM6_DIRICHLET && faces[a] != HELM6_NEUMANN && faces[a] != HELM6_SOMMERFELD)
      return HELM6_ERR_INVALID;
  for (int a = 0; a < 4; ++a)
    if (faces[a] == HELM6_SOMMERFELD) return HELM6_ERR_INVALID;
  if (!(std::isfinite(k.re) && std::isfinite(k.im))) return HELM6_ERR_INVALID;
  Geom g;
  for (int a = 0; a < 6; ++a) g.face[a] = faces[a];
  auto cnt = [&](int a) { return n + (faces[2 * a] != HELM6_DIRICHLET) + (faces[2 * a + 1] != HELM6_DIRICHLET); };
  g.mx = cnt(0);
  g.my = cnt(1);
  g.mz = cnt(2);
  g.N = (int64_t)g.mx * g.my * g.mz;
  // the grids this entry point takes: up to this many 32 x 8 x 16 bricks (stencil64's blocks are
  // larger, or a few hundred, so their partial sums fit the scratch; checked all the same)
  const int64_t nbricks = (int64_t)((g.mx + 31) / 32) * ((g.my + 7) / 8) * ((g.mz + 15) / 16);
  if (nbricks > HELM6_NOALLOC_MAX_BLOCKS || stencil_blocks(g) > HELM6_NOALLOC_MAX_BLOCKS) return HELM6_ERR_INVALID;
  double* scratch = nullptr;
  const int rc = scratch_for_current_device(&scratch);
  if (rc != HELM6_OK) return rc;
  StencilCoef coef;
  stencil_coefficients(cd(k.re, k.im), (h > 0) ? h : 1.0 / (n + 1), coef);
  cudaStream_t s = (cudaStream_t)stream;
  const int nblocks = launch_residual64_il(g, coef, (const double*)F, (const double*)u, (double*)r, scratch, s);
  note_launch();
  finish_kernel<<<1, 256, 0, s>>>(scratch, nblocks, sumsq);
  return cudaGetLastError() == cudaSuccess ? HELM6_OK : HELM6_ERR_CUDA;
}
