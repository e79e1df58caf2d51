// FP64 x/y eigen-transforms of the preconditioner (Eq. 3DAP) on the tensor cores, in exact
// integer slices.
//
// One transform contracts every row of a planar FP64 field along its contiguous axis with a
// real basis B (P modes x K points): out(row, p) = sum_k in(row, k) B(p, k).  GB300's FP64
// pipe issues two operations per clock and SM, so neither butterflies nor a dense product on
// that pipe comes near memory speed.  Here a row is taken as integers on its own scale,
//     in(row, k) = 2^(E_row - 1076) v_k,  |v_k| < 2^54   (E_row: the row's largest exponent),
// the basis as integers |b| <= 2^55 on the matrix' scale, both are written as seven signed
// base-256 digits (integers of magnitude <= 128: exact in FP16), and the product becomes
//     sum_l 2^(-8 l) S_l,   S_l = sum_{i + j = l} sum_k A_i(k) B_j(k),  l = 0..6,
// 28 FP16 tensor-core products with FP32 accumulation.  Every S_l is an integer below 2^24
// (checked on the host from the basis' digits), hence exact; the seven sums are combined in
// 64-bit integers and rounded to FP64 once.  The digit pairs left out (l >= 7) are 2^-53 of
// a result of the row's own size, below the rounding of an FP64 butterfly.
//
// Where both faces of the axis are alike (sine and cosine axes) the basis is symmetric or
// antisymmetric about the middle of the axis, B(p, K-1-k) = (-1)^p B(p, k), so even modes
// need v_k + v_{K-1-k} and odd ones v_k - v_{K-1-k} over half the points (the first step of
// an FFT, taken here exactly, on the integers): half the products.
//
// Persistent and warp-specialised, one CTA pair (cta_group::2) per two SMs: a unit of work is a
// 128-row tile, 64 rows in each CTA, with a range of column groups (a group: up to 128 modes of
// one parity; its seven accumulators take 7 x 64 tensor-memory columns of each CTA).  The pair
// halves what each SM's shared memory carries, which bounds the kernel: an SM reads 64 rows
// and 64 modes per product (one CTA alone: 128 rows and 64 modes for the same result), and every
// data point is turned into digits once per parity instead of twice.  K goes by in stages of 16:
//   * eight converter warps in two groups taking alternate stages copy a stage's row segments
//     (the mirrored ones too) into an FP64 ring with cp.async and turn them into the seven FP16
//     digit planes of the A operand;
//   * a producer thread streams its CTA's half of the basis' digit planes (cp.async.bulk) and passes
//     each landed copy on to the stage's barrier (the MMA warp's waiting on both took 4 % of A_p^-1);
//   * the MMA warp of the first CTA issues the 28 products of a stage for both; the second one's passes
//     its operands' barrier on to the first one's, so that each waits once per stage;
//   * eight epilogue warps take the finished sums out of tensor memory as 64-bit integers,
//     release it, then round and store them while the next group runs;
//   * two scanner warps find the row exponents of the next unit's rows (which also brings those
//     rows into L2).
// One or two modes beyond whole groups (258 points: 129 of each parity) are formed in FP64 by a
// kernel of their own.
// All arithmetic on data points and sums is 32-bit integer or FP32, most of it on the FMA pipe
// (multiply-adds, FP32 sums as integer conversions): an FP64 operation or conversion takes a
// scheduler 64 cycles, an FP32-to-integer conversion 8, a logic operation or a carry 2, an
// integer or FP32 multiply-add 1 (measured).
// Every wait is bounded; a timeout sets *err, and each CTA still waits (bounded, whatever the other
// roles do) for the MMAs and copies in flight before it frees tensor memory.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "helm6_internal.h"
#include "per_device.h"
#include "waits.h"

namespace helm6 {

namespace {

constexpr int DG = 7;                    // digits and accumulator levels
constexpr int X_M = 64;                  // rows of a CTA (a pair's tile: 128)
constexpr int X_KT = 16;                 // points of a stage (one MMA K step)
constexpr int X_NMAX = 128;              // columns of a group: 7 x 128 / 2 <= 512 tensor-memory columns
constexpr int X_NS = 4;                  // operand stages
constexpr int X_ND = 4;                  // FP64 ring stages
constexpr int X_EPI = 8, X_CONV = 8;     // warps 0-7 epilogue, 8-15 converters
constexpr int X_WPROD = 16, X_WMMA = 17;
constexpr int X_SCAN = 2;                // warps 18, 19 scanners
constexpr int X_THREADS = 640;
constexpr int A_PLANE = X_M * X_KT * 2;  // one digit plane of a stage: two core-matrix columns
constexpr int A_COL = (X_M / 8) * 128;   // K step of the plane
constexpr int A_BYTES = DG * A_PLANE;
constexpr int B_BYTES = DG * (X_NMAX / 2) * X_KT * 2;
constexpr int D_ROW = 2 * X_KT * 8;      // a row's segment and its mirror image
constexpr int D_BYTES = X_M * D_ROW;
constexpr int STG_LD = 9;                // staging row pitch of the row-major store (doubles)
constexpr int STG_BYTES = 32 * STG_LD * 8;
constexpr int O_A = 0;
constexpr int O_B = O_A + X_NS * A_BYTES;
constexpr int O_D = O_B + X_NS * B_BYTES;
constexpr int O_S = O_D + X_ND * D_BYTES;
constexpr int O_E = O_S + X_EPI * STG_BYTES;   // row exponents, two units
constexpr int O_BAR = O_E + 2 * X_M * 4;
constexpr int X_NBAR = 3 * X_NS + 7;
constexpr int O_MISC = O_BAR + X_NBAR * 8;
constexpr int X_SMEM = O_MISC + 16 + 1024;
static_assert(X_SMEM <= 232448, "shared memory per CTA");
static_assert(O_B % 128 == 0 && O_D % 128 == 0 && O_S % 16 == 0 && O_BAR % 8 == 0, "alignment");
static_assert(X_ND % 2 == 0 && X_NS % 2 == 0, "the converter groups take alternate stages");
constexpr int kPolls = 1 << 22;  // naps of a bounded wait

struct X64Args {
  const double* in;
  double* out;
  const uint8_t* W;  // [group][kt][half][digit][2 core-matrix columns][npad / 2 modes][16 B]
  int M_total, K, P, nk;
  int fold, eb;      // symmetric basis; |B| <= 2^eb
  int ngroups, gcols, nch, npad;  // groups, columns per group, groups per parity, padded columns
  int split, nunits;              // units per tile and in all
  int transposed, R, ldin, ldo;
  int tail;          // last modes, formed in FP64 from the rows Bt
  const double* Bt;  // [tail][K]
  int* err;
};

__device__ __forceinline__ uint32_t s_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor, no swizzle: start, K step, 8-row step.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

__device__ __forceinline__ bool try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred P1;\n mbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n"
      " selp.b32 %0, 1, 0, P1;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// One look at a phase, without the suspension of try_wait.
__device__ __forceinline__ bool test_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred P1;\n mbarrier.test_wait.parity.shared::cta.b64 P1, [%1], %2;\n"
      " selp.b32 %0, 1, 0, P1;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait by one thread; gives up when the flag is raised by another role.  It sleeps between
// polls: a spinning warp's issue slots are the converters' and the epilogue's (measured: half of
// all instructions were polls).
template <int NAP>
__device__ __forceinline__ bool poll1(uint32_t bar, uint32_t parity, volatile int* fail) {
  return wait_role([=] { return try_wait(bar, parity); }, [] { __nanosleep(NAP); }, fail, kPolls, 64);
}

// Bounded wait for products or copies under way, whatever the other roles do.  (In the second CTA the
// products' barrier also waits for the first one's MMA warp to end, after one bounded wait at most.)
__device__ __forceinline__ void poll_flight(uint32_t bar, uint32_t parity, volatile int* fail) {
  wait_flight([=] { return try_wait(bar, parity); }, [] { __nanosleep(100); }, fail, 4ll * kPolls);
}

// Warp-uniform bounded wait: every lane polls.  (Lane 0 alone and a shuffle of its answer: the warp
// diverges and meets again on each wait; 372/799/742/404 us for the four transforms of a 256^3
// preconditioner against 344/682/631/377.)
template <int NAP>
__device__ __forceinline__ bool pollw(uint32_t bar, uint32_t parity, volatile int* fail) {
  const bool ok = poll1<NAP>(bar, parity, fail);
  return __all_sync(0xffffffffu, ok) != 0;
}

// D (FP32) += A B^T, FP16 operands from shared memory; executed by the whole warp, issued by one
// elected lane (the operands stay in uniform registers).
__device__ __forceinline__ void mma_f16(uint32_t tmem, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p, e;\n setp.ne.b32 p, %4, 0;\n elect.sync _|e, 0xffffffff;\n"
      " @e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(id), "r"(acc));
}

// The pair's MMAs issued so far have completed: arrive on this barrier of both CTAs.
__device__ __forceinline__ void commit(uint32_t bar) {
  asm volatile(
      "{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
      " @e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n}\n" ::"r"(bar),
      "h"((uint16_t)3)
      : "memory");
}

// Arrive on the first CTA's barrier at the same place.
// What the arrival announces lies in this CTA's own shared memory (already passed to the async proxy)
// or tensor memory, so the default form is enough; .release.cluster waited for every load and store
// the CTA had in flight (388/812/765/414 us for the four transforms of a 256^3 preconditioner
// against 372/799/742/404).
__device__ __forceinline__ void arrive_lead(uint32_t bar) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"(bar));
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(a) : "memory");
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// 4 consecutive tensor-memory columns of the warp's 32 lanes.
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

template <int VEC>
__device__ __forceinline__ void cp_async(uint32_t dst, const void* src, int bytes) {
  if constexpr (VEC == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// A data point on its row's scale: |x| 2^(1084 - emax) as 62 bits, of which the upper 30 go (signed)
// into th and the next 24 into tl; `par` = -1 negates.  emax: the row's largest biased exponent.
// The implicit bit is set for zeros and denormals too: with emax >= 64 the shift removes it.
__device__ __forceinline__ void add_fixed(double x, int emax, int par, int& th, int& tl) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t s = ((((uint32_t)emax << 21) | 0x1fffffu) - 2u * hi) >> 21;  // emax - exponent
  const uint32_t h = (__funnelshift_l(lo, hi, 9) & 0x1fffffffu) | 0x20000000u;
  uint64_t w;
  asm("shr.u64 %0, %1, %2;" : "=l"(w) : "l"((uint64_t)h << 32 | (lo << 9)), "r"(s));  // 0 from 64 on
  const int sg = (((int)hi >> 31) | 1) * par;
  th += sg * (int)(uint32_t)(w >> 32);
  tl += sg * (int)((uint32_t)w >> 8);
}

// The same for rows whose largest exponent is below 64, where denormals count.
__device__ __noinline__ int2 add_fixed_tiny(double x, int emax, int par, int2 t) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7ffu);
  const uint64_t m = ((uint64_t)((hi & 0xfffffu) | (e ? 0x100000u : 0u)) << 32 | lo) << 9;
  const uint64_t w = m >> min(emax - max(e, 1), 63);
  const int sg = (((int)hi >> 31) | 1) * par;
  return make_int2(t.x + sg * (int)(uint32_t)(w >> 32), t.y + sg * (int)((uint32_t)w >> 8));
}

// The exponent of a row's scale from the largest |x| high word: one more where two such points could
// add up to all of 31 bits (the digits' balancing needs the room).
// (A row of zeros takes any scale.)
__device__ __forceinline__ int row_emax(int mx) {
  return mx == 0 ? 1023 : max((int)(((uint32_t)mx + 0x4000u) >> 20), 1);
}

// Sum of the seven levels, sum_l s_l 2^(40 - 8 l), as a 64-bit integer.  FAST: |s_l| <= 2^22, where adding
// 1.5 2^23 leaves the integer in the low bits of the FP32 pattern (on the FMA pipe; a conversion
// costs eight times as much).
template <bool FAST>
__device__ __forceinline__ int64_t level_sum(const float (&a)[DG]) {
  uint32_t v[DG];
#pragma unroll
  for (int l = 0; l < DG; ++l)
    v[l] = FAST ? __float_as_uint(a[l] + 12582912.f) : (uint32_t)__float2int_rn(a[l]) + 0x4B400000u;
  // modulo 2^64, the patterns' offsets taken off at the end
  uint64_t t = (uint64_t)(v[0] * 256u + v[1]) << 32;
  t += (uint64_t)v[2] * 16777216u;
  t += (uint64_t)v[3] * 65536u;
  t += (uint64_t)v[4] * 256u;
  constexpr uint64_t O = 0x4B400000ull;
  constexpr uint64_t off = (O << 40) + (O << 32) + (O << 24) + (O << 16) + (O << 8) + O + (O >> 8);
  return (int64_t)(t + (uint64_t)(v[5] + ((v[6] + 128u) >> 8)) - off);
}

// t 2^sc for an integer |t| < 2^63 and a scale that keeps every such result a normal number;
// ebase = 1085 + sc.  (Integers below 2^32 by a shift, not by conversions: in a solve the high modes of
// a smooth residual are that small against their row, and with FP64 conversions for them the x
// transform of a smooth 255^3 field took 507 us instead of 412.)
__device__ __forceinline__ double to_double(int64_t t, int ebase) {
  const int m = (int)(t >> 63);
  const uint64_t w = (uint64_t)(t ^ m) - (int64_t)m;
  const bool low = (uint32_t)(w >> 32) == 0;
  const uint64_t u = low ? w << 31 : w;
  const uint32_t uh = (uint32_t)(u >> 32), ul = (uint32_t)u;
  const int lz = __clz((int)uh), sh = lz - 1;  // leading bit to 62
  const uint64_t n = ((uint64_t)__funnelshift_l(ul, uh, sh) << 32 | (ul << (sh & 31))) + 0x200u;
  const uint32_t hi = (uint32_t)(n >> 42) + (uint32_t)((lz + (low ? 31 : 0)) * -(1 << 20)) + ((uint32_t)ebase << 20);
  return w ? __hiloint2double((int)(hi | ((uint32_t)m & 0x80000000u)), (int)(uint32_t)(n >> 10)) : 0.0;
}

// The unit's tile (this CTA's first row) and group range.
struct Unit {
  int m0, g0, g1;
};
__device__ __forceinline__ Unit unit(const X64Args& p, int u, int rank) {
  const int part = u % p.split;
  return Unit{(u / p.split) * 2 * X_M + rank * X_M, part * p.ngroups / p.split, (part + 1) * p.ngroups / p.split};
}

// The last p.tail modes in FP64, two modes of four rows at a time per warp, the lanes' shares of a row
// added pairwise.  Bound by the FP64 pipe: two products per data point at 258 points.
constexpr int TM_BLOCK = 256;
__global__ void __launch_bounds__(TM_BLOCK, 6) x64_tail_modes_kernel(X64Args p) {
  const int lane = threadIdx.x & 31;
  const int r0 = (int)((blockIdx.x * TM_BLOCK + threadIdx.x) >> 5) * 4, nr = min(4, p.M_total - r0);
  if (nr <= 0) return;
  const double* x = p.in + (int64_t)r0 * p.ldin;
  for (int t = 0; t < p.tail; t += 2) {
    const bool two = t + 1 < p.tail;
    const double *b0 = p.Bt + (int64_t)t * p.K, *b1 = two ? b0 + p.K : b0;
    double a[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) a[e] = 0.0;
#pragma unroll 1
    for (int k = lane; k < p.K; k += 32) {
      const double u = b0[k], v = b1[k];
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (e < nr) {
          const double w = x[(int64_t)e * p.ldin + k];
          a[2 * e] = fma(u, w, a[2 * e]);
          if (two) a[2 * e + 1] = fma(v, w, a[2 * e + 1]);
        }
    }
    // sum c of the eight to lane c: exchanges that halve what a lane is left with
#pragma unroll
    for (int h = 4; h > 0; h /= 2) {
      const bool up = lane & h;
#pragma unroll
      for (int c = 0; c < h; ++c) {
        const double give = up ? a[c] : a[c + h], keep = up ? a[c + h] : a[c];
        a[c] = keep + __shfl_xor_sync(0xffffffffu, give, h);
      }
    }
    double v = a[0];
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    const int row = r0 + lane / 2, m = p.P - p.tail + t + (lane & 1);
    if (lane < 2 * nr && m < p.P) {
      const int plane = row / p.R, rr = row - plane * p.R;
      p.out[p.transposed ? ((int64_t)plane * p.P + m) * p.ldo + rr : (int64_t)row * p.ldo + m] = v;
    }
  }
}

template <int VEC, bool FOLD>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(X_THREADS, 1) xform64_kernel(X64Args p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = (int)blockIdx.x & 1, pair = (int)blockIdx.x >> 1, npairs = (int)gridDim.x >> 1;
  uint32_t* tslot = (uint32_t*)(smem + O_MISC);
  volatile int* fail = (volatile int*)(tslot + 1);
  int* rowexp = (int*)(smem + O_E);
  const uint32_t bar0 = s_addr(smem + O_BAR);
  auto full = [&](int s) { return bar0 + 8u * s; };            // the stage's operands are there (first CTA: in both)
  auto sfree = [&](int s) { return bar0 + 8u * (X_NS + s); };  // the stage's MMAs completed
  auto bfull = [&](int s) { return bar0 + 8u * (2 * X_NS + s); };  // its basis digits are (its copy alone completes it)
  const uint32_t tfull = bar0 + 8u * (3 * X_NS);                   // the group's accumulators complete
  const uint32_t tempty = bar0 + 8u * (3 * X_NS + 1);              // first CTA: ... and drained in both
  auto efull = [&](int b) { return bar0 + 8u * (3 * X_NS + 2 + b); };  // row exponents of a unit known
  auto efree = [&](int b) { return bar0 + 8u * (3 * X_NS + 5 + b); };  // ... and read by everybody
  const uint32_t drain = bar0 + 8u * (3 * X_NS + 4);               // every MMA issued completed

  if (tid == 0) {
    auto init = [](uint32_t b, int n) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(b), "r"(n)); };
    for (int s = 0; s < X_NS; ++s) {
      init(full(s), 4 + (rank ? 1 : 2));  // a converter group, the producer; first CTA: the relay
      init(sfree(s), 1);
      init(bfull(s), 1);
    }
    init(tfull, 1);
    init(tempty, 2 * X_EPI);
    for (int b = 0; b < 2; ++b) {
      init(efull(b), X_SCAN);
      init(efree(b), X_EPI + X_CONV);
    }
    init(drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
    asm volatile("fence.proxy.async.shared::cta;");
    *fail = 0;
  }
  if (warp == X_WMMA) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_addr(tslot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  cluster_sync();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tslot;
  const int nun = pair < p.nunits ? (p.nunits - 1 - pair) / npairs + 1 : 0;
  auto unit_at = [&](int i) { return unit(p, pair + i * npairs, rank); };
  const uint32_t bplane = (uint32_t)p.npad * X_KT, bstage = DG * bplane;  // this CTA's half of the modes

  if (warp == X_WPROD) {
    // ---- basis producer: copies as slots come free, and each landed copy passed on to the stage's
    // barrier ----
    if (lane == 0) {
      // unit, group and K stage of copy q; copies before r have landed
      int i = 0, g = 0, kt = 0, q = 0, r = 0, idle = 0;
      Unit un = unit_at(0);
      while ((i < nun || r < q) && idle < kPolls) {
        bool step = false;
        if (i < nun && (q < X_NS || test_wait(sfree(q % X_NS), (q / X_NS - 1) & 1))) {
          const uint8_t* src = p.W + (((size_t)(un.g0 + g) * p.nk + kt) * 2 + rank) * bstage;
          const uint32_t bar = bfull(q % X_NS);
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bstage) : "memory");
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                  s_addr(smem + O_B + (q % X_NS) * B_BYTES)),
              "l"(src), "r"(bstage), "r"(bar)
              : "memory");
          ++q;
          if (++kt == p.nk) {
            kt = 0;
            if (un.g0 + ++g == un.g1) {
              g = 0;
              un = unit_at(++i);
            }
          }
          step = true;
        }
        if (r < q && test_wait(bfull(r % X_NS), (r / X_NS) & 1)) {
          arrive(full(r % X_NS));
          ++r;
          step = true;
        }
        if (step) {
          idle = 0;
        } else {
          if ((++idle & 63) == 0 && *fail) break;
          __nanosleep(50);
        }
      }
      if (idle == kPolls) *fail = 1;
      for (; r < q; ++r) poll_flight(bfull(r % X_NS), (r / X_NS) & 1, fail);  // every copy has landed before the CTA ends
    }
    __syncwarp();
  } else if (warp == X_WMMA) {
    // ---- MMA issuer (first CTA; the whole warp runs the loop, one elected lane issues) and, in the
    // second CTA, the relay of its operands' barriers to the first ----
    // kind::f16: D = FP32, A = B = FP16, both K-major, M = 128 (64 rows per CTA), N = npad
    const uint32_t id = (1u << 4) | ((uint32_t)(p.npad >> 3) << 17) | ((uint32_t)(2 * X_M >> 4) << 24);
    const uint64_t adesc = sdesc(s_addr(smem + O_A), A_COL, 128);
    const uint64_t bdesc = sdesc(s_addr(smem + O_B), (uint32_t)p.npad * 8, 128);
    int s = 0, ng = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int i = 0; i < nun && ok; ++i) {
      const Unit un = unit_at(i);
      for (int g = un.g0; g < un.g1 && ok; ++g, ++ng) {
        if (rank == 0) {
          if (ng >= 1 && !poll1<20>(tempty, (ng - 1) & 1, fail)) ok = false;
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;");
        }
        for (int kt = 0; kt < p.nk; ++kt) {
          ok = poll1<20>(full(s), ph, fail);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          if (rank) {
            if (lane == 0) arrive_lead(full(s));
          } else {
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint64_t a0 = adesc + (uint64_t)(s * (A_BYTES >> 4)), b0 = bdesc + (uint64_t)(s * (B_BYTES >> 4));
#pragma unroll
            for (int l = 0; l < DG; ++l)
#pragma unroll
              for (int d = 0; d <= l; ++d)
                mma_f16(tmem + (uint32_t)(l * (p.npad / 2)), a0 + (uint64_t)(d * (A_PLANE >> 4)),
                        b0 + (uint64_t)((l - d) * (bplane >> 4)), id, (kt > 0 || d > 0) ? 1u : 0u);
            commit(sfree(s));
          }
          if (++s == X_NS) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (ok && rank == 0) commit(tfull);
      }
    }
    // every MMA issued above has completed before either CTA frees its tensor memory
    if (rank == 0) commit(drain);
    poll_flight(drain, 0, fail);
    __syncwarp();
  } else if (warp > X_WMMA) {
    // ---- scanners: the largest |x| high word of each row, four rows at a time (the loads in flight,
    // not their number, set the time) ----
    const int w0 = (warp - X_WMMA - 1) * (X_M / X_SCAN);
    bool ok = true;
    for (int i = 0; i < nun && ok; ++i) {
      const int b = i & 1, m0 = unit_at(i).m0;
      if (i >= 2 && !pollw<100>(efree(b), ((i >> 1) - 1) & 1, fail)) break;
      for (int rr = w0; rr < w0 + X_M / X_SCAN; rr += 4) {
        uint32_t mx[4] = {0u, 0u, 0u, 0u};
        const uint32_t* src = (const uint32_t*)(p.in + (int64_t)(m0 + rr) * p.ldin) + 1;
        const int nr = min(4, p.M_total - (m0 + rr));
#pragma unroll 4
        for (int k = lane; k < p.K; k += 32)
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (e < nr) mx[e] = max(mx[e], src[2 * ((int64_t)e * p.ldin + k)] & 0x7fffffffu);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const uint32_t v = __reduce_max_sync(0xffffffffu, mx[e]);
          if (lane == 0) rowexp[b * X_M + rr + e] = (int)v;
        }
      }
      __syncwarp();
      if (lane == 0) arrive(efull(b));
    }
  } else if (warp >= X_EPI) {
    // ---- converters: warps of group grp take stages grp, grp + 2, ...; warp cw of a group owns
    // rows 16 cw .. 16 cw + 15; lane l converts row 16 cw + l % 16, points 8 (l / 16) .. + 7 ----
    const int grp = (warp - X_EPI) >> 2, cw = (warp - X_EPI) & 3;
    const int r = 16 * cw + (lane & 15), hk = lane >> 4, sw = r & 7;
    const uint32_t ring = s_addr(smem + O_D) + (uint32_t)(cw * 16 * D_ROW);
    int nst = 0;
    for (int i = 0; i < nun; ++i) {
      const Unit un = unit_at(i);
      nst += (un.g1 - un.g0) * p.nk;
    }
    // the next stage to copy: unit index, group within it, stage
    int ci = 0, cg = 0, ck = grp, cq = grp;
    Unit cu = unit_at(0);
    // one copy instruction covers RPC rows; a lane keeps its place within a row
    constexpr int SEG = FOLD ? D_ROW : D_ROW / 2, LPR = SEG / VEC, RPC = 32 / LPR;
    const int lr = lane / LPR, bb = (lane % LPR) * VEC, chunk = (bb & 127) >> 4, ce = (bb & 127) >> 3;
    auto issue = [&]() {
      if (cq < nst) {
        while (ck >= p.nk) {  // into the next group (a group can be a single stage)
          ck -= p.nk;
          if (++cg == cu.g1 - cu.g0) {
            cg = 0;
            cu = unit_at(++ci);
          }
        }
        // the segment starts at k0, its mirror image at K - 16 - k0
        const int k = (FOLD && bb >= 128 ? p.K - X_KT - ck * X_KT : ck * X_KT) + ce;
        const bool kok = k >= 0 && k < p.K;  // 16-byte copies: K and ldin even
        const int row = cu.m0 + 16 * cw + lr;
        const double* src = p.in + (int64_t)row * p.ldin + (kok ? k : 0);
        const uint32_t dst = ring + (uint32_t)((cq % X_ND) * D_BYTES + lr * D_ROW + (bb & 128) + (bb & 15));
#pragma unroll
        for (int c = 0; c < 16 / RPC; ++c) {
          const bool in = kok && row + c * RPC < p.M_total;
          cp_async<VEC>(dst + (uint32_t)(c * RPC * D_ROW + ((chunk ^ ((lr + c * RPC) & 7)) << 4)),
                        in ? src + (int64_t)(c * RPC) * p.ldin : p.in, in ? VEC : 0);
        }
      }
      cq += 2;
      ck += 2;
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int d = 0; d < X_ND / 2; ++d) issue();
    int q = 0;
    bool ok = true;
    for (int i = 0; i < nun && ok; ++i) {
      const Unit un = unit_at(i);
      if (!pollw<20>(efull(i & 1), (i >> 1) & 1, fail)) break;
      const int emax = row_emax(rowexp[(i & 1) * X_M + r]);
      __syncwarp();
      if (lane == 0) arrive(efree(i & 1));
      const bool tiny = __any_sync(0xffffffffu, emax < 64);
      for (int g = un.g0; g < un.g1 && ok; ++g) {
        const int par = (FOLD && g >= p.nch) ? -1 : 1;  // odd modes: differences
        for (int kt = 0; kt < p.nk; ++kt, ++q) {
          if ((q & 1) != grp) continue;
          const int s = q % X_NS, u = q / X_NS;
          asm volatile("cp.async.wait_group %0;" ::"n"(X_ND / 2 - 1) : "memory");
          __syncwarp();
          const uint8_t* d0 = smem + O_D + (size_t)(q % X_ND) * D_BYTES + (size_t)r * D_ROW;
          int th[8], tl[8];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const double2 a = *(const double2*)(d0 + (((4 * hk + c) ^ sw) << 4));
            // points 8 hk + 2 c, + 1 pair with positions 15 - (8 hk + 2 c), - 1 of the mirror image (the
            // middle point is its own)
            double2 b = make_double2(0.0, 0.0);
            if constexpr (FOLD) {
              b = *(const double2*)(d0 + 128 + (((7 - 4 * hk - c) ^ sw) << 4));
              const int k = kt * X_KT + 8 * hk + 2 * c;
              if (2 * k == p.K - 1) b.y = 0.0;
              if (2 * k + 2 == p.K - 1) b.x = 0.0;
            }
            int h0 = 0, l0 = 0, h1 = 0, l1 = 0;
            if (!tiny) {
              add_fixed(a.x, emax, 1, h0, l0);
              add_fixed(a.y, emax, 1, h1, l1);
              if constexpr (FOLD) {
                add_fixed(b.y, emax, par, h0, l0);
                add_fixed(b.x, emax, par, h1, l1);
              }
            } else {
              int2 t0 = add_fixed_tiny(a.x, emax, 1, make_int2(0, 0)), t1 = add_fixed_tiny(a.y, emax, 1, make_int2(0, 0));
              if constexpr (FOLD) {
                t0 = add_fixed_tiny(b.y, emax, par, t0);
                t1 = add_fixed_tiny(b.x, emax, par, t1);
              }
              h0 = t0.x, l0 = t0.y, h1 = t1.x, l1 = t1.y;
            }
            // balanced base-256 digits: 128 added to each byte, the lower word's carry into the upper
            // one; the lower word's free byte takes the FP16 exponent bits of its three digits
            l0 += 0x808080;
            l1 += 0x808080;
            th[2 * c] = (int)((uint32_t)(h0 + (l0 >> 24)) + 0x80808080u);
            th[2 * c + 1] = (int)((uint32_t)(h1 + (l1 >> 24)) + 0x80808080u);
            tl[2 * c] = (l0 & 0xffffff) | 0x64000000;
            tl[2 * c + 1] = (l1 & 0xffffff) | 0x64000000;
          }
          __syncwarp();
          issue();  // the ring slot just read is free again
          if (u >= 1 && !pollw<20>(sfree(s), (u - 1) & 1, fail)) {
            ok = false;
            break;
          }
          uint8_t* sA = smem + O_A + s * A_BYTES + hk * A_COL + (r >> 3) * 128 + (r & 7) * 16;
#pragma unroll
          for (int d = 0; d < DG; ++d) {
            uint32_t w[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              uint32_t f;  // two fields 1024 + 128 + digit as FP16
              if (d < 4) {
                const uint32_t b = 3u - d;
                f = (__byte_perm((uint32_t)th[2 * c], (uint32_t)th[2 * c + 1], b | ((b + 4u) << 8)) & 0x00ff00ffu) | 0x64006400u;
              } else {
                const uint32_t b = 6u - d;
                f = __byte_perm((uint32_t)tl[2 * c], (uint32_t)tl[2 * c + 1], b | 0x30u | ((b + 4u) << 8) | 0x7000u);
              }
              const uint32_t k1152 = 0x64806480u;
              const __half2 h = __hsub2(*(const __half2*)&f, *(const __half2*)&k1152);
              w[c] = *(const uint32_t*)&h;
            }
            *(uint4*)(sA + d * A_PLANE) = make_uint4(w[0], w[1], w[2], w[3]);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) arrive(full(s));
        }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else {
    // ---- epilogue: the accumulators of a CTA's 64 rows and N modes sit in 128 lanes and N / 2 columns:
    // lanes 0-63 hold modes 0 .. N/2 - 1 of the rows, lanes 64-127 modes N/2 .. N - 1.  Warp w takes
    // lane quarter w % 4 and half of its columns ----
    const int quarter = warp & 3, h = warp >> 2, npq = p.npad >> 2;  // columns of a warp (at most 32)
    double* stg = (double*)(smem + O_S + warp * STG_BYTES);
    int ng = 0;
    bool ok = true;
    for (int i = 0; i < nun && ok; ++i) {
      const Unit un = unit_at(i);
      if (!pollw<100>(efull(i & 1), (i >> 1) & 1, fail)) break;
      const int lrow = 32 * (quarter & 1) + lane, row0 = un.m0 + 32 * (quarter & 1), row = row0 + lane;
      const bool live = row < p.M_total;
      const int nrows = min(32, p.M_total - row0);
      const int mx = rowexp[(i & 1) * X_M + lrow];
      __syncwarp();
      if (lane == 0) arrive(efree(i & 1));
      const bool nonfinite = mx >= 0x7ff00000;
      // out = T 2^sc, |T| < 2^63: into the exponent field where that cannot leave its range
      const int sc = row_emax(mx) - 1075 + p.eb;
      const bool plain = __all_sync(0xffffffffu, !nonfinite && sc >= -1022 && sc <= 2046 - 1086);
      int64_t obase = 0;
      if (p.transposed) {
        const int plane = row / p.R, rr = row - plane * p.R;
        obase = (int64_t)plane * p.ldo * p.P + rr;
      }
      for (int g = un.g0; g < un.g1; ++g, ++ng) {
        if (!pollw<100>(tfull, ng & 1, fail)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        // this warp's columns: every second mode from its parity on, or consecutive modes
        const int odd = FOLD && g >= p.nch ? 1 : 0, step = FOLD ? 2 : 1;
        const int m0 = (g - odd * p.nch) * p.gcols + (quarter >> 1) * (p.npad >> 1) + h * npq;
        const int col0 = step * m0 + odd, ncol = min(npq, (p.P - col0 + step - 1) / step);
        const uint32_t taddr = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(h * npq);
        int64_t T[X_NMAX / 4];
#pragma unroll
        for (int c = 0; c < X_NMAX / 4; c += 4) {
          if (c < npq) {
            uint32_t a[DG][4];
#pragma unroll
            for (int l = 0; l < DG; ++l) tmem_ld4(taddr + (uint32_t)(l * (p.npad >> 1) + c), a[l]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            float f[4][DG], big = 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
#pragma unroll
              for (int l = 0; l < DG; ++l) {
                f[j][l] = __uint_as_float(a[l][j]);
                big = fmaxf(big, fabsf(f[j][l]));
              }
            }
            if (!__any_sync(0xffffffffu, big > 4194304.f)) {
#pragma unroll
              for (int j = 0; j < 4; ++j) T[c + j] = level_sum<true>(f[j]);
            } else {
#pragma unroll
              for (int j = 0; j < 4; ++j) T[c + j] = level_sum<false>(f[j]);
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncwarp();
        if (lane == 0) arrive_lead(tempty);
        // rounded and stored while the next group's products run
#pragma unroll
        for (int c = 0; c < X_NMAX / 4; c += 8) {
          if (c >= ncol) continue;
          double v[8];
          if (plain) {
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = to_double(T[c + j], 1085 + sc);
          } else {  // rows at the ends of the exponent range, NaN and Inf
#pragma unroll
            for (int j = 0; j < 8; ++j)
              v[j] = nonfinite ? __longlong_as_double(0x7ff8000000000000ll) : scalbn(__ll2double_rn(T[c + j]), sc);
          }
          const int nc = min(8, ncol - c);
          if (p.transposed) {
            if (live) {
              double* o = p.out + obase + (int64_t)(col0 + step * c) * p.ldo;
#pragma unroll
              for (int j = 0; j < 8; ++j)
                if (j < nc) o[(int64_t)(step * j) * p.ldo] = v[j];
            }
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) stg[lane * STG_LD + j] = v[j];
            __syncwarp();
            const int j = lane & 7;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const int rr = 4 * e + (lane >> 3);
              if (rr < nrows && j < nc) p.out[(int64_t)(row0 + rr) * p.ldo + col0 + step * (c + j)] = stg[rr * STG_LD + j];
            }
            __syncwarp();
          }
        }
      }
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  cluster_sync();  // the peer's copies, arrivals and MMAs into this CTA are done
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (tid == 0 && *fail) atomicExch(p.err, 1);
  if (warp == X_WMMA) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

int round32(int n) { return ((n + 31) / 32) * 32; }

// One axis' closed-form eigenbasis (the layouts and normalisation of the dense bases): entry
// (node l, mode j) is trig[l j mod 2 D], every angle exactly reduced.
struct X64Axis {
  int N, m, D;           // intervals, unknowns, half period of the table
  int nlo, nhi, inverse;
  double sc;             // 2 / N
};

__device__ __forceinline__ double basis_entry(const X64Axis& a, const double* trig, int p, int k) {
  // inverse: B(p, k) = V(node p, mode k); forward: B(p, k) = W(mode p, node k)
  const int node = a.inverse ? p : k, mode = a.inverse ? k : p;
  const bool quarter = a.nlo != a.nhi;
  const int64_t l = a.nlo ? node : node + 1;
  const int64_t j = quarter ? 2 * (mode + 1) - 1 : (a.nlo ? mode : mode + 1);
  const double v = trig[(l * j) % (2 * a.D)];
  if (a.inverse) return v;
  double w = 1.0;
  if (a.nlo && a.nhi && (j == 0 || j == a.N)) w *= 0.5;
  if ((a.nlo && l == 0) || (a.nhi && l == a.N)) w *= 0.5;
  return a.sc * w * v;
}

// FP64 rows of the last modes (or nodes) of an axis, first m - tail.
__global__ void x64_tail_kernel(X64Axis a, X64Basis h, const double* __restrict__ trig) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < h.tail * a.m) ((double*)(h.dev + h.planes))[i] = basis_entry(a, trig, a.m - h.tail + i / a.m, i % a.m);
}

// Digit planes of one column (mode or node p) per block, in the transform kernel's layout.  *over is
// set when an accumulator could leave the integers that FP32 holds exactly: level l sums the basis
// digits 0..l times data digits of at most 128.
__global__ void __launch_bounds__(128) x64_digits_kernel(X64Axis a, X64Basis h, const double* __restrict__ trig,
                                                         double scale, int* over) {
  __shared__ int ssum;
  const int g = blockIdx.x / h.gcols, c = blockIdx.x % h.gcols, half = h.gcols / 2;
  const int odd = h.fold && g >= h.nch ? 1 : 0, ch = g - odd * h.nch;
  const int p = h.fold ? 2 * (ch * h.gcols + c) + odd : ch * h.gcols + c;
  const int K = a.m, Kf = h.fold ? (K + 1) / 2 : K;
  const size_t plane = (size_t)h.gcols * X_KT, stage = DG * plane;
  if (threadIdx.x == 0) ssum = 0;
  __syncthreads();
  int sum = 0;
  for (int k = threadIdx.x; k < h.nk * X_KT; k += blockDim.x) {
    double b = 0.0;  // padding modes and points
    if (p < a.m && k < Kf && !(odd && 2 * k == K - 1)) b = basis_entry(a, trig, p, k);
    int64_t x = __double2ll_rn(b * scale);
    uint8_t* o = h.dev + (((size_t)g * h.nk + k / X_KT) * 2 + c / half) * stage +
                 (size_t)((k % X_KT) / 8) * half * 16 + (size_t)(c % half) * 16 + (size_t)(k % 8) * 2;
    for (int d = DG - 1; d >= 0; --d) {
      const int v = d > 0 ? (int)((x + 128) & 255) - 128 : (int)x;
      x = (x - v) >> 8;
      sum += abs(v);
      *(__half*)(o + (size_t)d * plane) = __int2half_rn(v);
    }
  }
  atomicAdd(&ssum, sum);
  __syncthreads();
  if (threadIdx.x == 0 && 128ll * ssum > 1ll << 24) atomicExch(over, 1);
}

}  // namespace

// Sizes of the basis planes of an axis with n interior nodes.
X64Basis x64_plan(int n, int lo, int hi) {
  const bool nlo = lo != HELM6_DIRICHLET, nhi = hi != HELM6_DIRICHLET;
  X64Basis h;
  h.m = n + (nlo ? 1 : 0) + (nhi ? 1 : 0);
  h.fold = nlo == nhi;
  const int Kf = h.fold ? (h.m + 1) / 2 : h.m, cnt = Kf;  // points of a product; modes of the larger parity
  h.nk = (Kf + X_KT - 1) / X_KT;
  // One or two modes more than the groups hold would split them into twice as many, and each group
  // turns its tile's points into digits again, the slowest role: they are formed apart (258
  // points, four groups of 96 columns: 682 and 631 us for the two transforms of a 256^3 field; two
  // groups of 128 and two modes apart: 565 and 534).  Each further pair of modes would cost 160.
  const int whole = (h.fold ? 2 : 1) * (cnt / X_NMAX) * X_NMAX;
  h.tail = whole > 0 && h.m > whole && h.m - whole <= 2 ? h.m - whole : 0;
  h.nch = h.tail ? cnt / X_NMAX : (cnt + X_NMAX - 1) / X_NMAX;
  h.gcols = h.tail ? X_NMAX : round32((cnt + h.nch - 1) / h.nch);
  h.ngroups = (h.fold && h.m > 1 ? 2 : 1) * h.nch;
  h.planes = (size_t)h.ngroups * h.nk * 2 * DG * h.gcols * X_KT;
  h.bytes = h.planes + (size_t)h.tail * h.m * sizeof(double);
  return h;
}

// Products of more points than this never pass the digits' check (which fails for single lengths from 250
// points of a quarter-wave axis on, from 232 point pairs of a cosine and 275 of a sine axis; the last lengths to
// pass have 279 points, 282 and 284 pairs).
bool x64_may_fit(const X64Basis& h) { return (h.fold ? (h.m + 1) / 2 : h.m) <= 288; }

// The trigonometric table of an axis: sin or cos of pi t / D, t < 2 D, from the first octant.
void x64_trig(int n, int lo, int hi, std::vector<double>& trig) {
  const bool nlo = lo != HELM6_DIRICHLET, nhi = hi != HELM6_DIRICHLET;
  const int N = n + 1, D = nlo != nhi ? 2 * N : N;
  trig.resize(2 * (size_t)D);
  for (int t = 0; t < 2 * D; ++t) {
    int q = t;
    double sg = 1.0;
    if (nlo) {
      if (q > D) q = 2 * D - q;                 // cos(2 pi - x) = cos x
      if (2 * q > D) { q = D - q; sg = -1.0; }  // cos(pi - x) = -cos x
      trig[t] = 2 * q == D ? 0.0 : sg * (4 * q <= D ? std::cos(M_PI * q / D) : std::sin(M_PI * (D - 2 * q) / (2.0 * D)));
    } else {
      if (q >= D) { q -= D; sg = -1.0; }        // sin(x + pi) = -sin x
      if (2 * q > D) q = D - q;                 // sin(pi - x) = sin x
      trig[t] = sg * (4 * q <= D ? std::sin(M_PI * q / D) : std::cos(M_PI * (D - 2 * q) / (2.0 * D)));
    }
  }
}

// Fill the planes at h.dev of the forward or inverse basis (stream-ordered); *over (device) is set when
// the axis is out of the kernel's range.
void launch_x64_digits(int n, int lo, int hi, int inverse, X64Basis& h, const double* trig, int* over, cudaStream_t s) {
  const bool nlo = lo != HELM6_DIRICHLET, nhi = hi != HELM6_DIRICHLET;
  X64Axis a;
  a.N = n + 1;
  a.m = h.m;
  a.nlo = nlo;
  a.nhi = nhi;
  a.D = nlo != nhi ? 2 * a.N : a.N;
  a.inverse = inverse;
  a.sc = 2.0 / a.N;
  // |B| <= 1 (inverse) or 2 / N
  h.eb = 0;
  if (!inverse)
    while (std::ldexp(1.0, h.eb - 1) >= a.sc) --h.eb;
  if (!inverse && a.sc > 1.0) h.eb = 1;
  note_launch();
  x64_digits_kernel<<<h.ngroups * h.gcols, 128, 0, s>>>(a, h, trig, std::ldexp(1.0, 55 - h.eb), over);
  if (h.tail) {
    note_launch();
    x64_tail_kernel<<<(h.tail * h.m + 127) / 128, 128, 0, s>>>(a, h, trig);
  }
}

int x64_configure() {
  static OncePerDevice once;
  auto set = [](auto* k) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, X_SMEM) == cudaSuccess;
  };
  return once(current_device(),
              [&] {
                return set(xform64_kernel<16, true>) && set(xform64_kernel<16, false>) && set(xform64_kernel<8, true>) &&
                       set(xform64_kernel<8, false>);
              })
             ? HELM6_OK
             : HELM6_ERR_CUDA;
}

void launch_xform64(const X64Basis& b, const double* in, double* out, int M_total, int transposed, int R, int* err,
                    cudaStream_t s, int ldin, int ldo) {
  if (M_total <= 0) return;
  X64Args a;
  a.in = in;
  a.out = out;
  a.W = b.dev;
  a.M_total = M_total;
  a.K = a.P = b.m;
  a.nk = b.nk;
  a.fold = b.fold;
  a.eb = b.eb;
  a.ngroups = b.ngroups;
  a.gcols = a.npad = b.gcols;
  a.nch = b.nch;
  a.transposed = transposed;
  a.R = R;
  a.ldin = ldin;
  a.ldo = ldo;
  a.tail = b.tail;
  a.Bt = (const double*)(b.dev + b.planes);
  a.err = err;
  static int sms = 0;
  if (!sms) sms = device_sm_count();
  // a tile's groups go to one CTA pair (its rows are scanned once) unless that leaves SMs idle
  const int tiles = (M_total + 2 * X_M - 1) / (2 * X_M), pairs = std::max(1, sms / 2);
  a.split = std::max(1, std::min(b.ngroups, pairs / tiles));
  a.nunits = tiles * a.split;
  const unsigned grid = 2u * (unsigned)std::min(a.nunits, pairs);
  // 16-byte copies: rows, segments and mirrored segments all start on an even point
  const bool v16 = ldin % 2 == 0 && b.m % 2 == 0 && (uintptr_t)in % 16 == 0;
  note_launch();
  if (b.fold) {
    if (v16)
      xform64_kernel<16, true><<<grid, X_THREADS, X_SMEM, s>>>(a);
    else
      xform64_kernel<8, true><<<grid, X_THREADS, X_SMEM, s>>>(a);
  } else {
    if (v16)
      xform64_kernel<16, false><<<grid, X_THREADS, X_SMEM, s>>>(a);
    else
      xform64_kernel<8, false><<<grid, X_THREADS, X_SMEM, s>>>(a);
  }
  if (a.tail) {
    note_launch();
    x64_tail_modes_kernel<<<(unsigned)(((int64_t)M_total + 4 * TM_BLOCK / 32 - 1) / (4 * TM_BLOCK / 32)), TM_BLOCK, 0, s>>>(a);
  }
}

}  // namespace helm6
