// Hot-path kernels: WENO reconstruction per cell (Section 2), gas-kinetic flux per face Gauss
// point (Section 3.2), per-cell gather of face fluxes with the two-stage fourth-order update
// (Section 3.3), the time-step bound, and caller-order permutations.
#include <cuda_runtime.h>

#include <cfloat>
#include <cmath>
#include <type_traits>

#include "gks_device.cuh"
#include "gks_ff.cuh"
#include "gks_kinetic.cuh"
#include "gks_flux_f32x2.cuh"

namespace gks {
namespace {

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// ------------------------------------------------------------------------------------------
// Gather copy of a state (48 bytes per cell, see Lay<R>) and the stencil differences taken
// from it. FP32 path: each value is kept as hi + lo floats, so Q_k - Q_0 is formed as
// (hi_k - hi_0) + (lo_k - lo_0) without FP64 arithmetic and is as accurate as rounding the
// FP64 difference to FP32. FP64 path: the FP64 values themselves.
// (double)x by integer arithmetic, for every x: the conversion instruction runs at the FP64 rate
// (1/64 of the FP32 rate) even where it is predicated off. Subnormal numbers are scaled by 2^64
// first (exact).
__device__ __forceinline__ double widen(float x) {
  const bool sub = (__float_as_uint(x) & 0x7fffffffu) < 0x00800000u;  // subnormal or zero
  const uint32_t u = __float_as_uint(sub ? x * 18446744073709551616.f : x);
  const uint32_t m = u & 0x7fffffffu;
  uint32_t hi = (m >> 3) + (sub ? 0x34000000u : 0x38000000u);
  if (m == 0) hi = 0;
  if (m >= 0x7f800000u) hi = 0x7ff00000u | ((m >> 3) & 0xfffffu);  // infinite or NaN
  return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
}
template <class R>
struct Gq;
template <>
struct Gq<float> {
  float hi[5], lo[5];
  __device__ __forceinline__ void load(const float* __restrict__ QA, int64_t c) {
    const float4* p = reinterpret_cast<const float4*>(QA + 12 * c);
    const float4 a = __ldg(p), b = __ldg(p + 1);
    const float2 d = __ldg(reinterpret_cast<const float2*>(p + 2));
    hi[0] = a.x; hi[1] = a.y; hi[2] = a.z; hi[3] = a.w; hi[4] = b.x;
    lo[0] = b.y; lo[1] = b.z; lo[2] = b.w; lo[3] = d.x; lo[4] = d.y;
  }
  __device__ __forceinline__ void flip(int v) { hi[v] = -hi[v]; lo[v] = -lo[v]; }
  __device__ __forceinline__ float minus(const Gq& c, int v) const {
    return (hi[v] - c.hi[v]) + (lo[v] - c.lo[v]);
  }
  __device__ __forceinline__ float value(int v) const { return hi[v] + lo[v]; }
  __device__ __forceinline__ float value_minus(int v, float x) const { return hi[v] + (lo[v] - x); }
  __device__ static void store(float* QA, int64_t c, const double q[5]) {
    float h[5], l[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      h[v] = (float)q[v];
      l[v] = (float)(q[v] - widen(h[v]));
    }
    float4* p = reinterpret_cast<float4*>(QA + 12 * c);
    p[0] = make_float4(h[0], h[1], h[2], h[3]);
    p[1] = make_float4(h[4], l[0], l[1], l[2]);
    p[2] = make_float4(l[3], l[4], 0.f, 0.f);
  }
  __device__ static void store_ff(float* QA, int64_t c, const ff q[5]) {
    float4* p = reinterpret_cast<float4*>(QA + 12 * c);
    p[0] = make_float4(q[0].h, q[1].h, q[2].h, q[3].h);
    p[1] = make_float4(q[4].h, q[0].l, q[1].l, q[2].l);
    p[2] = make_float4(q[3].l, q[4].l, 0.f, 0.f);
  }
};
template <>
struct Gq<double> {
  double q[5];
  __device__ __forceinline__ void load(const double* __restrict__ QA, int64_t c) {
    const double2* p = reinterpret_cast<const double2*>(QA + 6 * c);
    const double2 a = __ldg(p), b = __ldg(p + 1), d = __ldg(p + 2);
    q[0] = a.x; q[1] = a.y; q[2] = b.x; q[3] = b.y; q[4] = d.x;
  }
  __device__ __forceinline__ void flip(int v) { q[v] = -q[v]; }
  __device__ __forceinline__ double minus(const Gq& c, int v) const { return q[v] - c.q[v]; }
  __device__ __forceinline__ double value(int v) const { return q[v]; }
  __device__ __forceinline__ double value_minus(int v, double x) const { return q[v] - x; }
  __device__ static void store(double* QA, int64_t c, const double qq[5]) {
    double2* p = reinterpret_cast<double2*>(QA + 6 * c);
    p[0] = make_double2(qq[0], qq[1]);
    p[1] = make_double2(qq[2], qq[3]);
    p[2] = make_double2(qq[4], 0.0);
  }
};

// FP64 value of variable v of a gather copy.
__device__ __forceinline__ double unpack_value(const Gq<float>& g, int v) {
  return widen(g.hi[v]) + widen(g.lo[v]);
}
__device__ __forceinline__ double unpack_value(const Gq<double>& g, int v) { return g.q[v]; }

// ------------------------------------------------------------------------------------------
// Asynchronous bulk copies global -> shared completed on an mbarrier (transaction bytes), and a
// bounded wait on it.
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
// bytes: a multiple of 16; dst and src 16-byte aligned
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
// Bulk store shared -> global in a bulk group (src and dst 16-byte aligned, bytes a multiple of
// 16). The threads that wrote the source with ordinary stores fence them into the async proxy
// (fence_proxy_async_shared) and the block synchronises before one thread issues the store;
// that thread waits until the store has read its source before the block's shared memory may
// be reused.
__device__ __forceinline__ void fence_proxy_async_shared() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst),
               "r"(smem_u32(src)), "r"(bytes)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_store_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Each try_wait suspends the thread for at most a hardware time limit; the loop gives up after
// `tries` attempts (by default kWaitTries, far beyond the microseconds a tile's copies take).
constexpr int kWaitTries = 1 << 22;
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int tries) {
  for (int it = 0; it < tries; ++it)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// ------------------------------------------------------------------------------------------
// Reconstruction, one block of five warps per 32-cell tile (lane = cell). For each conserved
// variable v of each cell:
//   dq_k = Q_k - Q_0 over the big stencil                      (phase 1, all warps, to shared)
//   a    = A+ dq   (quadratic P0, 9 coefficients in centred scaled coordinates) and
//   b_m  = B_m dq|S_m (linear P_m) with beta_m (Eq. indicator); rows and sub-stencils are
//   spread over the warps                                                            (phase 2)
//   beta_0, tau, omega, omega-bar (Section 2), one variable per warp               (phase 3)
//   C = (wb_0/g_0) a + sum_m (wb_m - wb_0 g_m/g_0) b_m, i.e. Eq. weno as one polynomial (phase 4)
// Output: 10 coefficients per variable of the polynomial in physical offsets from the centroid.
// Bound by the chain of dependent latencies of a block (about 19,000 cycles at 5 blocks per SM
// before this form: gathers, row loads, the weights), with L1 two thirds busy and DRAM at half
// its rate; so the order of the block is built to start every load early and to keep late loads
// out of the chain:
//  - the stencil indices and the cell's own state are requested before anything else; a range
//    whose tiles all have the first one's stencil size takes their place from the tile index,
//    with no table load before them;
//  - with kPf one thread then starts the tile's other transfers: the pseudo-inverse rows (a
//    contiguous block of the interleaved layout) by a bulk prefetch into L2, the per-cell record
//    of phase 3 by a bulk copy into shared memory on an mbarrier, and the sub-stencil entries
//    either by such a copy too (kStB: where that costs the range no resident blocks) or by a
//    prefetch into L2;
//  - phase 2: warps 0-2 take three rows each in one member loop unrolled by six, so that 18
//    independent row loads are in flight and a stencil difference is read once for three rows;
//    the other warps take the sub-stencils; the mbarrier is awaited where its data are read.
// Measured per FP32 pass on the 64^3-cube mesh with the enlarged stencils (and the 32^3-cube
// mesh in FP64): two rows on each of the five warps, table loads and a barrier before the
// gathers, moments loaded in phase 3: 0.419 ms (0.676); three rows on three warps 0.411
// (0.663); the record in shared memory, fewer quotients 0.404 (0.627); indices first, two
// barriers instead of three 0.385 (0.614); six unstaged entries in flight and two of eight
// sub-stencils on row warps 0.362 (0.604); rows, entries and indices without L1 lines 0.356
// (0.599). Not adopted:
// six blocks per SM (64 registers, spills) 0.409; row loads started before the gathers' barrier
// 0.385-0.400 (the prefetch has not landed); no prefetch of the rows 0.396, of the entries
// 0.387; a bulk prefetch of a later block's tile 0.415-0.467 (indices only 0.367); batches of 2,
// 3 and 5 members 0.427, 0.393, 0.424; staging the rows in shared memory costs 2 resident
// blocks.
constexpr int kReconWarps = 5;
constexpr int kRowWarps = 3;  // warps 0-2 take three rows of A+ each, the others sub-stencils
constexpr int kRowShare = 6;  // sub-stencils from this one on go to row warps (unstaged entries)
constexpr int kBatch = 4;     // stencil members a thread gathers at a time
constexpr int kReconThreads = kReconWarps * kTile;
// resident blocks per SM of the register bound (launch bounds): five in FP32 (80 registers a
// thread), three in FP64, as many as its shared memory allows
template <class R>
constexpr int kReconBlocksPerSM = sizeof(R) == 4 ? 5 : 3;

// Shared-memory layout of one block for a range with largest stencil Kr, largest sum of
// sub-stencil member counts Sr and largest number of sub-stencil slots Mr, in units of one
// interleaved row (kTile values): [mbarrier, 16 B][per-cell records, kCellRec] (with kPf),
// [B entries 4 Sr] (with kPf and stb: the sub-stencil entries staged by a bulk copy), then
// a[9][5], b[Mr][3][5], beta[Mr][5], dq[Kr][5] (the last in the lane-major form of DqRow below).
// Every part starts on a 16-byte boundary.

template <class R>
struct ReconSmem {
  size_t c_off, b_off, ca_off, cb_off, cbet_off, dq_off, bytes;
  __host__ __device__ ReconSmem(int Kr, int Sr, int Mr, bool pf, bool stb) {
    const size_t row = (size_t)kTile * sizeof(R);
    c_off = pf ? 16 : 0;
    b_off = c_off + (pf ? kCellRec * row : 0);
    ca_off = b_off + (pf && stb ? 4 * (size_t)Sr * row : 0);
    cb_off = ca_off + 45 * row;
    cbet_off = cb_off + 15 * (size_t)Mr * row;
    dq_off = cbet_off + 5 * (size_t)Mr * row;
    // the dq region holds the tile's output records [lane][kPolyStride] once phase 2 is done
    bytes = dq_off + (5 * (size_t)Kr > (size_t)kPolyStride ? 5 * (size_t)Kr : kPolyStride) * row;
  }
};

// Stencil differences in shared memory: variables 0-3 of member k as 16-byte vectors with the
// lane fastest ([k][h][lane], h < 1 in FP32, h < 2 in FP64), variable 4 in a plain row [k][lane]
// after all of them, so that a thread reads or writes a member's five differences in two (FP32)
// or three (FP64) shared-memory accesses instead of five; consecutive lanes touch consecutive
// 16-byte words (no bank conflicts). Against five scalar rows: 0.599 -> 0.595 ms per FP32 pass
// on the 64^3-cube mesh.
template <class R>
struct DqRow;
template <>
struct DqRow<float> {
  __device__ __forceinline__ static void put(unsigned char* s, int k, int lane, const float d[4]) {
    reinterpret_cast<float4*>(s)[k * kTile + lane] = make_float4(d[0], d[1], d[2], d[3]);
  }
  __device__ __forceinline__ static void get(const unsigned char* s, int k, int lane, float d[4]) {
    const float4 x = reinterpret_cast<const float4*>(s)[k * kTile + lane];
    d[0] = x.x; d[1] = x.y; d[2] = x.z; d[3] = x.w;
  }
};
template <>
struct DqRow<double> {
  __device__ __forceinline__ static void put(unsigned char* s, int k, int lane, const double d[4]) {
    double2* p = reinterpret_cast<double2*>(s) + 2 * k * kTile + lane;
    p[0] = make_double2(d[0], d[1]);
    p[kTile] = make_double2(d[2], d[3]);
  }
  __device__ __forceinline__ static void get(const unsigned char* s, int k, int lane, double d[4]) {
    const double2* p = reinterpret_cast<const double2*>(s) + 2 * k * kTile + lane;
    const double2 x = p[0], y = p[kTile];
    d[0] = x.x; d[1] = x.y; d[2] = y.x; d[3] = y.y;
  }
};

// Loads of data that a block reads once (pseudo-inverse rows, sub-stencil entries, stencil
// indices): read-only path without an L1 line, so that the gathered states stay in L1 (0.362 ->
// 0.356 ms per FP32 pass on the 64^3-cube mesh).
__device__ __forceinline__ float ld_once(const float* p) {
  float v;
  asm volatile("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ double ld_once(const double* p) {
  double v;
  asm volatile("ld.global.nc.L1::no_allocate.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ int32_t ld_once(const int32_t* p) {
  int32_t v;
  asm volatile("ld.global.nc.L1::no_allocate.s32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 ld_once(const float4* p) {
  float4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ double2 ld_once(const double2* p) {
  double2 v;
  asm volatile("ld.global.nc.L1::no_allocate.v2.f64 {%0, %1}, [%2];"
               : "=d"(v.x), "=d"(v.y)
               : "l"(p));
  return v;
}

// One sub-stencil entry (three pseudo-inverse coefficients and the member index) of one lane:
// one 16-byte load in FP32, two in FP64, from shared memory (staged) or through the read-only
// path (global). Against four interleaved rows: 0.571 -> 0.569 ms per FP32 pass.
template <class R>
struct BRec;
template <>
struct BRec<float> {
  __device__ __forceinline__ static void get(const float* e, bool staged, float c[4]) {
    const float4* p = reinterpret_cast<const float4*>(e);
    const float4 x = staged ? *p : ld_once(p);
    c[0] = x.x; c[1] = x.y; c[2] = x.z; c[3] = x.w;
  }
};
template <>
struct BRec<double> {
  __device__ __forceinline__ static void get(const double* e, bool staged, double c[4]) {
    const double2* p = reinterpret_cast<const double2*>(e);
    const double2 x = staged ? p[0] : ld_once(p), y = staged ? p[1] : ld_once(p + 1);
    c[0] = x.x; c[1] = x.y; c[2] = y.x; c[3] = y.y;
  }
};

// A variable's ten output coefficients to shared memory in the widest stores its place allows (a
// record of kPolyStride values starts on a 16-byte boundary; variable v at 10 v values): in FP32
// two 16-byte and one 8-byte store, in FP64 five 16-byte ones.
template <class R>
struct PolyPair;
template <>
struct PolyPair<float> {
  __device__ __forceinline__ static void put(float* so, int v, const float o[10]) {
    if ((v & 1) == 0) {
      reinterpret_cast<float4*>(so)[0] = make_float4(o[0], o[1], o[2], o[3]);
      reinterpret_cast<float4*>(so)[1] = make_float4(o[4], o[5], o[6], o[7]);
      *reinterpret_cast<float2*>(so + 8) = make_float2(o[8], o[9]);
    } else {
      *reinterpret_cast<float2*>(so) = make_float2(o[0], o[1]);
      *reinterpret_cast<float4*>(so + 2) = make_float4(o[2], o[3], o[4], o[5]);
      *reinterpret_cast<float4*>(so + 6) = make_float4(o[6], o[7], o[8], o[9]);
    }
  }
};
template <>
struct PolyPair<double> {
  __device__ __forceinline__ static void put(double* so, int, const double o[10]) {
    double2* p = reinterpret_cast<double2*>(so);
#pragma unroll
    for (int j = 0; j < 5; ++j) p[j] = make_double2(o[2 * j], o[2 * j + 1]);
  }
};

// Quotients of the weights and the output scaling: the FP32 path uses the fast division
// intrinsic (x times an approximate reciprocal, within 2 ulp for divisors below 2^126: the
// indicators, weights and cell sizes here), the FP64 path the IEEE division. Against IEEE
// divisions in FP32: 0.436 -> 0.417 ms per pass on the 64^3-cube mesh (the weights of phase 3
// take about a dozen quotients per thread).
template <class R>
__device__ __forceinline__ R wdiv(R a, R b) {
  return a / b;
}
template <>
__device__ __forceinline__ float wdiv<float>(float a, float b) {
  return __fdividef(a, b);
}

// b[s] <- tau / b[s], s = 0..M (M <= 8; the entries beyond M are 1). FP32: one fast quotient
// each. FP64: a division is a chain of a dozen FP64 instructions on a pipe that bounds the
// kernel, so three quotients are taken from one division by the product of the three (each product
// rounds once more) where tau and the three lie in 2^-240..2^240 (tau may be zero: uniform data),
// so that nothing on the way leaves the FP64 range; else the three divisions.
template <class R>
__device__ __forceinline__ void quotients(R tau, int M, R b[kMaxSub + 1]) {
#pragma unroll
  for (int s = 0; s <= kMaxSub; ++s)
    if (s <= M) b[s] = wdiv(tau, b[s]);
}
template <>
__device__ __forceinline__ void quotients<double>(double tau, int M, double b[kMaxSub + 1]) {
  // positive and within 2^-240..2^240, by the exponent bits
  auto inner = [](double x) {
    return (uint32_t)__double2hiint(x) - 0x30f00000u < 0x1e000000u;
  };
  const bool tau_ok = inner(tau) || tau == 0.0;
#pragma unroll
  for (int g = 0; g < 3; ++g) {
    if (3 * g > M) continue;
    const double x = b[3 * g], y = b[3 * g + 1], z = b[3 * g + 2];
    if (tau_ok && inner(x) && inner(y) && inner(z)) {
      const double xy = x * y, r = tau / (xy * z), rz = r * z;
      b[3 * g] = rz * y;
      b[3 * g + 1] = rz * x;
      b[3 * g + 2] = r * xy;
    } else {
      b[3 * g] = tau / x;
      b[3 * g + 1] = tau / y;
      b[3 * g + 2] = tau / z;
    }
  }
}

// A uniform range (TileRanges::uni): with on >= 1 the tile's stencil arrays start at
// st0 + K (tile - tile0), with on == 2 its sub-stencil entries at sb0 + S (tile - tile0).
struct ReconUni {
  int on, K, S;
  uint64_t cnt;
  int64_t st0, sb0, tile0;
};
// The ranges of one launch: one range per launch on large meshes, every range in one launch on
// small ones (launch_recon), where a block finds its range by its tile.
struct ReconSet {
  int n;
  ReconUni r[kMaxTileRanges];
};

__device__ __forceinline__ ReconUni range_of(const ReconUni& u, int64_t) { return u; }
__device__ __forceinline__ ReconUni range_of(const ReconSet& set, int64_t tile) {
  ReconUni u = set.r[0];
#pragma unroll
  for (int r = 1; r < kMaxTileRanges; ++r)
    if (r < set.n && tile >= set.r[r].tile0) u = set.r[r];
  return u;
}

// kMany: one launch over several ranges (set), else one range.
template <class R, bool kPf, bool kStB, bool kMany>
__global__ void __launch_bounds__(kReconThreads, kReconBlocksPerSM<R>) k_recon(
    int64_t nc, int64_t tile0, int Kr, int Sr, int Mr,
    const __grid_constant__ std::conditional_t<kMany, ReconSet, ReconUni> set,
    const R* __restrict__ QA,
    const int32_t* __restrict__ t_K, const uint64_t* __restrict__ t_cnt,
    const int32_t* __restrict__ t_st, const int32_t* __restrict__ t_sb,
    const int32_t* __restrict__ t_idx, const R* __restrict__ Ap, const R* __restrict__ Bp,
    const R* __restrict__ cell, R wg, R weps, int wpow, R* __restrict__ poly, int* flag,
    int wait_tries, int withhold) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const ReconSmem<R> L(Kr, Sr, Mr, kPf, kStB);
  R* sa = reinterpret_cast<R*>(smem_raw + L.ca_off);      // [n][v][lane]
  R* sb = reinterpret_cast<R*>(smem_raw + L.cb_off);      // [m][t][v][lane]
  R* sbet = reinterpret_cast<R*>(smem_raw + L.cbet_off);  // [m][v][lane]
  unsigned char* sdqv = smem_raw + L.dq_off;              // variables 0-3, DqRow<R>
  R* sdq4 = reinterpret_cast<R*>(sdqv + 4 * (size_t)Kr * kTile * sizeof(R));  // [k][lane]
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);
  const int64_t tile = tile0 + blockIdx.x;
  const int lane = threadIdx.x & (kTile - 1);
  const int warp = threadIdx.x / kTile;
  const ReconUni u = range_of(set, tile);
  const int64_t tl = tile - (kMany ? u.tile0 : tile0);
  const int K = u.on ? u.K : __ldg(t_K + tile);
  const int64_t st = u.on ? u.st0 + tl * u.K : (int64_t)__ldg(t_st + tile);
  // phase 1, first half: the stencil indices of the first batch and the cell's own state are
  // requested before anything else
  const int64_t i = tile * kTile + lane;
  const bool valid = i < nc;
  const int64_t ic = valid ? i : tile * kTile;  // padded lanes mirror the tile's first cell
  const int32_t* sidx = t_idx + st * kTile + lane;
  int32_t e[kBatch];
#pragma unroll
  for (int j = 0; j < kBatch; ++j) {
    const int k = warp + j * kReconWarps;
    e[j] = k < K ? ld_once(sidx + k * kTile) : -1;
  }
  Gq<R> c0;
  c0.load(QA, ic);
  const uint64_t cnt = u.on == 2 ? u.cnt : __ldg(t_cnt + tile);
  const int64_t sbo = u.on == 2 ? u.sb0 + tl * u.S : (int64_t)__ldg(t_sb + tile);
  const R* Ag = Ap + st * 9 * kTile;
  const R* Bg = Bp + sbo * 4 * kTile;
  int S = 0, Mt = 0;  // entries and sub-stencil slots of this tile
#pragma unroll
  for (int q = 0; q < kMaxSub; ++q) {
    const int c = (int)((cnt >> (8 * q)) & 0xffu);
    S += c;
    if (c) Mt = q + 1;
  }
  if (kPf && threadIdx.x == kReconThreads - kTile) {  // the last warp: it has the fewest members
    mbar_init(bar);
    const uint32_t ab = 9u * K * kTile * sizeof(R), bb = 4u * S * kTile * sizeof(R);
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(Ag), "r"(ab) : "memory");
    if (!kStB && bb)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(Bg), "r"(bb) : "memory");
    // withhold != 0 (the timeout test of gks_debug_recon_wait): no copy is issued and 16
    // bytes more than the copies would bring are expected, so the barrier's phase never
    // completes and the bounded wait below runs out with nothing in flight
    constexpr uint32_t cb = kCellRec * kTile * sizeof(R);
    mbar_expect_tx(bar, cb + (kStB ? bb : 0u) + (withhold ? 16u : 0u));
    if (!withhold) {
      bulk_load(smem_raw + L.c_off, cell + tile * kCellRec * kTile, cb, bar);
      if (kStB && bb) bulk_load(smem_raw + L.b_off, Bg, bb, bar);
    }
  }

  // phase 1: stencil differences, members split over the warps, kBatch per batch: all index
  // loads, then all state loads, then the differences
  for (int k0 = warp; k0 < K; k0 += kBatch * kReconWarps) {
    if (k0 != warp) {
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int k = k0 + j * kReconWarps;
        e[j] = k < K ? ld_once(sidx + k * kTile) : -1;
      }
    }
    Gq<R> g[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j)
      if (e[j] >= 0) g[j].load(QA, e[j] & kCellMask);
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      if (e[j] < 0) continue;
      const int fl = e[j] >> kFlipShift;
      if (fl & 1) g[j].flip(1);
      if (fl & 2) g[j].flip(2);
      if (fl & 4) g[j].flip(3);
      const int k = k0 + j * kReconWarps;
      R d[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) d[v] = g[j].minus(c0, v);
      DqRow<R>::put(sdqv, k, lane, d);
      sdq4[k * kTile + lane] = g[j].minus(c0, 4);
    }
  }
  __syncthreads();
  const R* Bt = (kPf && kStB ? reinterpret_cast<const R*>(smem_raw + L.b_off) : Bg) + 4 * lane;
  // the copies (per-cell records, staged entries) are awaited where they are read: by the
  // sub-stencil warps before their entries, by the row warps after their rows. A block whose
  // wait ran out reports it and stops at the barrier before phase 3.
  bool ok = true;
  auto wait_copies = [&]() {
    if (!kPf) return;
    const int tries = wait_tries > 0 ? wait_tries : kWaitTries;
    ok = mbar_wait(bar, 0, tries);
    if (!ok) ok = mbar_wait(bar, 0, tries);  // let copies still in flight land before leaving
  };

  // phase 2: rows n = 3 warp .. 3 warp + 2 of a = A+ dq on the row warps (in one member loop:
  // each stencil difference is read once for the three rows), and the sub-stencil fits b_m with
  // their indicators beta_m = |b_m|^2 (scaled coordinates) on the others meanwhile
  if (warp < kRowWarps) {
    R acc[3][5];
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int v = 0; v < 5; ++v) acc[j][v] = R(0);
    const R* q = Ag + 3 * warp * kTile + lane;
#pragma unroll 6
    for (int k = 0; k < K; ++k, q += 9 * kTile) {
      const R r0 = ld_once(q), r1 = ld_once(q + kTile), r2 = ld_once(q + 2 * kTile);
      R d[5];
      DqRow<R>::get(sdqv, k, lane, d);
      d[4] = sdq4[k * kTile + lane];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        acc[0][v] += r0 * d[v];
        acc[1][v] += r1 * d[v];
        acc[2][v] += r2 * d[v];
      }
    }
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int v = 0; v < 5; ++v) sa[(5 * (3 * warp + j) + v) * kTile + lane] = acc[j][v];
  }
  wait_copies();
  // sub-stencils: the two sub warps alternate; where the entries come through L2 (kStB = false:
  // the kinds with many sub-stencils) the seventh and eighth go to row warps 0 and 1, and six
  // entries are in flight instead of two
  constexpr int kSubU = kStB ? 2 : 6;
  const bool sub_warp = warp >= kRowWarps;
  const int s_first = sub_warp ? warp - kRowWarps : (kStB ? kMaxSub : kRowShare + warp);
  const int s_end = !kStB && sub_warp && Mt > kRowShare ? kRowShare : Mt;
  // (a wait that ran out left no entries to index with)
  for (int s = s_first; ok && s < s_end; s += sub_warp ? kReconWarps - kRowWarps : kMaxSub) {
    int slot = 0;
    for (int q = 0; q < s; ++q) slot += (int)((cnt >> (8 * q)) & 0xffu);
    const int cs = (int)((cnt >> (8 * s)) & 0xffu);
    const R* e = Bt + (int64_t)4 * kTile * slot;
    R b[3][5];
#pragma unroll
    for (int t = 0; t < 3; ++t)
#pragma unroll
      for (int v = 0; v < 5; ++v) b[t][v] = R(0);
#pragma unroll kSubU
    for (int j = 0; j < cs; ++j, e += 4 * kTile) {
      R c[4];
      BRec<R>::get(e, kPf && kStB, c);
      const int k = (int)c[3];
      R dq[5];
      DqRow<R>::get(sdqv, k, lane, dq);
      dq[4] = sdq4[k * kTile + lane];
#pragma unroll
      for (int v = 0; v < 5; ++v)
#pragma unroll
        for (int t = 0; t < 3; ++t) b[t][v] += c[t] * dq[v];
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      sbet[(5 * s + v) * kTile + lane] = b[0][v] * b[0][v] + b[1][v] * b[1][v] + b[2][v] * b[2][v];
#pragma unroll
      for (int t = 0; t < 3; ++t) sb[((3 * s + t) * 5 + v) * kTile + lane] = b[t][v];
    }
  }
  if (__syncthreads_or(!ok)) {
    if (threadIdx.x == 0) atomicOr(flag, kErrTimeout);
    return;
  }

  // phase 3: nonlinear weights, variable v = warp
  const R* rec = (kPf ? reinterpret_cast<const R*>(smem_raw + L.c_off)
                      : cell + tile * kCellRec * kTile) + lane;
  R m2[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) m2[q] = rec[q * kTile];
  const int M = (int)rec[7 * kTile];
  const R g0 = R(1) - wg * rec[7 * kTile];
  const R ig0 = rec[9 * kTile];
  const int v = warp;
  {
    R a[9];
#pragma unroll
    for (int n = 0; n < 9; ++n) a[n] = sa[(5 * n + v) * kTile + lane];
    // |l| = 1 terms: cell means of the squared first derivatives, linear in the scaled
    // coordinates with second moments m2: a_lin^2 + m2 : H^2, H the matrix of second
    // derivatives; |l| = 2 terms: squared second derivatives
    const R h0 = R(2) * a[3], h1 = R(2) * a[4], h2 = R(2) * a[5];
    const R t0 = h0 * h0, t1 = h1 * h1, t2 = h2 * h2;
    const R s6 = a[6] * a[6], s7 = a[7] * a[7], s8 = a[8] * a[8];
    const R beta0 = a[0] * a[0] + a[1] * a[1] + a[2] * a[2] + (t0 + t1 + t2) + (s6 + s7 + s8) +
                    m2[0] * (t0 + s6 + s7) + m2[1] * (t1 + s6 + s8) + m2[2] * (t2 + s7 + s8) +
                    R(2) * (m2[3] * (a[6] * (h0 + h1) + a[7] * a[8]) +
                            m2[4] * (a[7] * (h0 + h2) + a[6] * a[8]) +
                            m2[5] * (a[8] * (h1 + h2) + a[6] * a[7]));
    R tau = R(0);
    for (int s = 0; s < M; ++s) tau += fabs(beta0 - sbet[(5 * s + v) * kTile + lane]);
    tau *= rec[8 * kTile];
    // bt[0] = beta_0 + eps, bt[1 + s] = beta_s + eps, then tau over each
    R wm[kMaxSub + 1];
    wm[0] = beta0 + weps;
#pragma unroll
    for (int s = 0; s < kMaxSub; ++s)
      wm[1 + s] = s < M ? sbet[(5 * s + v) * kTile + lane] + weps : R(1);
    quotients(tau, M, wm);
    R sum = R(0);
#pragma unroll
    for (int s = 0; s <= kMaxSub; ++s) {
      if (s > M) {
        wm[s] = R(0);
        continue;
      }
      const R r = wm[s];
      R pw = r;
      for (int q = 1; q < wpow; ++q) pw *= r;
      wm[s] = (s == 0 ? g0 : wg) * (R(1) + pw);
      sum += wm[s];
    }
    const R is = wdiv(R(1), sum);
    const R wb0 = wm[0] * is;
    const R corr = wb0 * wg * ig0;
    // phase 4 (same warp, same variable): linear part of the combination and the output
    R cl[3] = {R(0), R(0), R(0)};
#pragma unroll
    for (int s = 0; s < kMaxSub; ++s) {
      if (s < M) {
        const R f = wm[1 + s] * is - corr;
#pragma unroll
        for (int t = 0; t < 3; ++t) cl[t] += f * sb[((3 * s + t) * 5 + v) * kTile + lane];
      }
    }
    const R ca = wb0 * ig0;
    R C[9];
#pragma unroll
    for (int n = 0; n < 9; ++n) C[n] = ca * a[n];
    C[0] += cl[0];
    C[1] += cl[1];
    C[2] += cl[2];
    {
      const R ih = rec[6 * kTile], ih2 = ih * ih;
      // Q = c0 + c1 dx + c2 dy + c3 dz + c4 dx^2 + c5 dy^2 + c6 dz^2 + c7 dxdy + c8 dxdz + c9 dydz
      const R shift = C[3] * m2[0] + C[4] * m2[1] + C[5] * m2[2] + C[6] * m2[3] +
                      C[7] * m2[4] + C[8] * m2[5];
      R o[10];
      o[0] = R(0);  // c0's component v, selected without a dynamic register index
#pragma unroll
      for (int q = 0; q < 5; ++q)
        if (q == v) o[0] = c0.value_minus(q, shift);
      o[1] = C[0] * ih;
      o[2] = C[1] * ih;
      o[3] = C[2] * ih;
#pragma unroll
      for (int n = 3; n < 9; ++n) o[n + 1] = C[n] * ih2;
      // the tile's output records go to shared memory (the stencil differences are dead after
      // phase 2) and leave in one contiguous bulk store: written directly, every store of a
      // warp touched 32 sectors for 4 bytes each (0.569 -> 0.457 ms per FP32 pass on the
      // 64^3-cube mesh, 5.36 -> 5.34 ms in FP64)
      R* so = reinterpret_cast<R*>(smem_raw + L.dq_off) + lane * kPolyStride + 10 * v;
      PolyPair<R>::put(so, v, o);
    }
  }
  fence_proxy_async_shared();
  __syncthreads();
  if (threadIdx.x == 0) {
    const int64_t nv = nc - tile * kTile < kTile ? nc - tile * kTile : kTile;
    bulk_store(poly + (int64_t)kPolyStride * tile * kTile, smem_raw + L.dq_off,
               (uint32_t)(nv * kPolyStride * sizeof(R)));
    bulk_store_wait_read();
  }
}

// Coefficient accessor of one cell's polynomial (kPolyStride values per cell).
template <class R>
struct PolyRef {
  const R* __restrict__ p;
  __device__ __forceinline__ R operator()(int v, int j) const { return __ldg(p + 10 * v + j); }
};
// A variable's ten coefficients as five pair loads (a cell's record starts on a 16-byte
// boundary: kPolyStride values of 4 or 8 bytes; variable v at 10 v values).
// In FP32 a variable's ten coefficients start on a 16-byte boundary for even v and on an 8-byte
// one for odd v: three loads (16 + 16 + 8 or 8 + 16 + 16 bytes) instead of five.
__device__ __forceinline__ void load_coefs(const PolyRef<float>& c, int v, float k[10]) {
  const float* p = c.p + 10 * v;
  if ((v & 1) == 0) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p));
    const float4 b = __ldg(reinterpret_cast<const float4*>(p + 4));
    const float2 d = __ldg(reinterpret_cast<const float2*>(p + 8));
    k[0] = a.x; k[1] = a.y; k[2] = a.z; k[3] = a.w;
    k[4] = b.x; k[5] = b.y; k[6] = b.z; k[7] = b.w;
    k[8] = d.x; k[9] = d.y;
  } else {
    const float2 a = __ldg(reinterpret_cast<const float2*>(p));
    const float4 b = __ldg(reinterpret_cast<const float4*>(p + 2));
    const float4 d = __ldg(reinterpret_cast<const float4*>(p + 6));
    k[0] = a.x; k[1] = a.y;
    k[2] = b.x; k[3] = b.y; k[4] = b.z; k[5] = b.w;
    k[6] = d.x; k[7] = d.y; k[8] = d.z; k[9] = d.w;
  }
}
__device__ __forceinline__ void load_coefs(const PolyRef<double>& c, int v, double k[10]) {
  const double2* q = reinterpret_cast<const double2*>(c.p + 10 * v);
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const double2 t = __ldg(q + i);
    k[2 * i] = t.x;
    k[2 * i + 1] = t.y;
  }
}

// Positivity fallback at a Gauss point (off unless the solver asks for it; the paper prints no
// positivity treatment): a side whose reconstructed state has rho <= 0 or p <= 0 (or NaN) takes
// the cell average of its cell, read from the gather copy the reconstruction used, with a zero
// gradient. p > 0 is tested as rho E > |m|^2 / 2, which needs no division.
template <class R>
__device__ __forceinline__ void first_order_if_nonphysical(const R* __restrict__ QA, int64_t c,
                                                           R v[5], R g[5][3]) {
  const R m2 = v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
  if (v[0] > R(0) && v[0] * v[4] > R(0.5) * m2) return;
  Gq<R> q;
  q.load(QA, c);
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    v[k] = q.value(k);
#pragma unroll
    for (int a = 0; a < 3; ++a) g[k][a] = R(0);
  }
}

// The same for a pair of points, each on its own.
__device__ __forceinline__ void first_order_if_nonphysical2(const float* __restrict__ QA,
                                                            int64_t c, P2 v[5], P2 g[5][3]) {
  const P2 m2 = v[1] * v[1] + v[2] * v[2] + v[3] * v[3], e = v[0] * v[4];
  const bool b0 = !(v[0].lo() > 0.f && e.lo() > 0.5f * m2.lo());
  const bool b1 = !(v[0].hi() > 0.f && e.hi() > 0.5f * m2.hi());
  if (!b0 && !b1) return;
  Gq<float> q;
  q.load(QA, c);
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    v[k] = P2(b0 ? q.value(k) : v[k].lo(), b1 ? q.value(k) : v[k].hi());
#pragma unroll
    for (int a = 0; a < 3; ++a)
      g[k][a] = P2(b0 ? 0.f : g[k][a].lo(), b1 ? 0.f : g[k][a].hi());
  }
}
// The wall's ghost of a pair of points in place of the owner's values, one point at a time (the
// far-field state branches on the point's state).
__device__ __forceinline__ void wall_ghost2(const FluxParams<float>& P, int wall,
                                         const WallData<float>& wd, P2 v[5], P2 g[5][3]) {
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    float vo[5], go[5][3], vg[5], gg[5][3];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      vo[k] = h ? v[k].hi() : v[k].lo();
#pragma unroll
      for (int a = 0; a < 3; ++a) go[k][a] = h ? g[k][a].hi() : g[k][a].lo();
    }
    wall_ghost(P, wall, wd, vo, go, vg, gg);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      v[k] = h ? P2(v[k].lo(), vg[k]) : P2(vg[k], v[k].hi());
#pragma unroll
      for (int a = 0; a < 3; ++a)
        g[k][a] = h ? P2(g[k][a].lo(), gg[k][a]) : P2(gg[k][a], g[k][a].hi());
    }
  }
}

// ------------------------------------------------------------------------------------------
// Flux: per Gauss point both sides' reconstructions and gradients, F^n and dF/dt in the global
// frame (gks_flux.cuh), weighted by the quadrature weight; the four points of a face are summed
// with shuffles and written once. k_flux_pair (FP32, smooth form): two threads per face, two
// points per thread on packed arithmetic; k_flux: four threads per face, one point per thread, in
// FP64, and in FP32 for the full form with the two sides packed. kTau0 fixes a zero collision
// time and kFull the full form at compile time, so that an instance carries only its own form.
// Bound by issue slots and the FMA pipe (FP64: the FP64 pipe, 1/64 of the FP32 rate), so the form
// with the fewest operations wins. Per launch, against the flux in the face frame (values and
// gradients rotated to the normal and two tangents, one moment derivative per axis):
//   FP32 smooth, 64^3-cube mesh (2.39 M faces): 0.418 -> 0.326 ms, two points per thread 0.302;
//   FP32 full, 48^3-cube explosion (1.02 M faces): 326 -> 231 us;
//   FP64 smooth, 32^3 cubes (299 k faces): 2.53 -> 1.77 ms, with erfc and exp from one table and
//     one division per state (half_erfc, to_prim) 1.49, sums started from the other side's 1.44,
//     shorter slopes (side_der) and exchanges that halve the four-point sums 1.39;
//   FP64 full, 124 k faces of tetrahedra: 2.05 -> 1.31, 1.20, 1.16, 1.14 ms.
// Resident threads per SM, measured: FP32 smooth 8 blocks of 64 (0.302 ms; of 128 threads 4
// blocks 0.307, 3 blocks without spills 0.322, 5 blocks 0.407); FP32 full 4 blocks of 128 (231
// us; 3 and 5 blocks 254 and 254); FP64 unbounded (two blocks).
constexpr int kPairThreads = 64, kPairBlocks = 8;  // k_flux_pair
constexpr int kFullBlocks = 4, kSidesBlocks = 6;   // k_flux, FP32 full and smooth form, 128 threads
// Fewest faces of k_flux_pair, about one and a half waves of its threads: below it the GPU is not
// full, and four threads per face are done sooner (ten steps of the 8^3-cube mesh, 4,672 faces,
// 474 -> 468 us; 37,000 faces 659 -> 655 us; equal at 126,000; at 299,000 2.252 against 2.286 ms).
constexpr int64_t kPairFaces = 60000;
// One 16-byte (FP32) or 32-byte (FP64) part of a face record of kFaceStride values: part j holds
// values 4j .. 4j + 3 of acc (values 10 and 11 are padding, written as zeros).
template <class R>
struct FaceRec;
template <>
struct FaceRec<float> {
  __device__ __forceinline__ static void put(float* rec, int j, const float acc[10]) {
    float4 x;
    if (j == 0) x = make_float4(acc[0], acc[1], acc[2], acc[3]);
    else if (j == 1) x = make_float4(acc[4], acc[5], acc[6], acc[7]);
    else x = make_float4(acc[8], acc[9], 0.f, 0.f);
    reinterpret_cast<float4*>(rec)[j] = x;
  }
};
template <>
struct FaceRec<double> {
  __device__ __forceinline__ static void put(double* rec, int j, const double acc[10]) {
    double2 x, y;
    if (j == 0) { x = make_double2(acc[0], acc[1]); y = make_double2(acc[2], acc[3]); }
    else if (j == 1) { x = make_double2(acc[4], acc[5]); y = make_double2(acc[6], acc[7]); }
    else { x = make_double2(acc[8], acc[9]); y = make_double2(0.0, 0.0); }
    double2* p = reinterpret_cast<double2*>(rec) + 2 * j;
    p[0] = x;
    p[1] = y;
  }
};

template <bool kTau0>
__global__ void __launch_bounds__(kPairThreads, kPairBlocks)
    k_flux_pair(int64_t nf, const int32_t* __restrict__ f_owner, const int32_t* __restrict__ f_nb,
                const int8_t* __restrict__ f_wall, const float* __restrict__ fgp,
                const float* __restrict__ poly, const float* __restrict__ QA, int fallback,
                FluxParams<float> P, const float* __restrict__ wall_tab, float dt,
                float* __restrict__ fface, int* flag) {
  P.full = 0;
  if (kTau0) P.tau_model = 0;
  const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t f = gid >> 1;  // two threads per face, Gauss points 2 (gid & 1) and the next
  const bool active = f < nf;
  float acc[10];
#pragma unroll
  for (int q = 0; q < 10; ++q) acc[q] = 0.f;
  int wall = -1;
  if (active) {
    const int64_t stride = 4 * nf;
    const int32_t o = f_owner[f], nb = f_nb[f];
    wall = f_wall[f];
    auto pair_at = [&](int a) {
      return P2(__ldcs(reinterpret_cast<const float2*>(fgp + a * stride) + gid));
    };
    P2 d[3], n[3], v[5], g[5][3], acc2[10];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      d[a] = pair_at(a);
      n[a] = pair_at(6 + a);
    }
    eval_poly2(PolyRef<float>{poly + (int64_t)kPolyStride * o}, d, v, g);
    if (fallback) first_order_if_nonphysical2(QA, o, v, g);
    auto right = [&](P2* v, P2 (*g)[3]) {
      if (nb >= 0) {
        P2 e[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) e[a] = pair_at(3 + a);
        eval_poly2(PolyRef<float>{poly + (int64_t)kPolyStride * nb}, e, v, g);
        if (fallback) first_order_if_nonphysical2(QA, nb, v, g);
      } else {
        wall_ghost2(P, wall, wall_data(wall_tab, wall), v, g);  // the wall's ghost
      }
    };
    const unsigned ok = gp_flux_pair(P, v, g, right, n, pair_at(9), dt, acc2);
    if (ok != 3u) atomicOr(flag, kErrNonphysical);
#pragma unroll
    for (int q = 0; q < 10; ++q) acc[q] = hsum(acc2[q]);
  }
#pragma unroll
  for (int q = 0; q < 10; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], 1);
  // both lanes of the face hold the sums; lane j writes the record's 16-byte part j, lane 0 part 2
  if (active) {
    if (wall >= 0) wall_flux_fix(wall, wall_data(wall_tab, wall), acc);
    float* rec = fface + (int64_t)kFaceStride * f;
    FaceRec<float>::put(rec, (int)(gid & 1), acc);
    if ((gid & 1) == 0) FaceRec<float>::put(rec, 2, acc);
  }
}

// One Gauss point per thread, four consecutive threads per face: FP64, and the FP32 full form.
template <class R, bool kFull, bool kTau0>
__global__ void __launch_bounds__(128, sizeof(R) == 4 ? (kFull ? kFullBlocks : kSidesBlocks) : 1) k_flux(
    int64_t nf, const int32_t* __restrict__ f_owner, const int32_t* __restrict__ f_nb,
    const int8_t* __restrict__ f_wall, const R* __restrict__ fgp, const R* __restrict__ poly,
    const R* __restrict__ QA, int fallback, FluxParams<R> P, const R* __restrict__ wall_tab, R dt,
    R* __restrict__ fface, int* flag) {
  P.full = kFull;
  if (kTau0) P.tau_model = 0;
  const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t f = gid >> 2;
  const bool active = f < nf;
  R acc[10];
#pragma unroll
  for (int q = 0; q < 10; ++q) acc[q] = R(0);
  int wall = -1;
  if (active) {
    const int64_t stride = 4 * nf;
    const int32_t o = f_owner[f], nb = f_nb[f];
    wall = f_wall[f];
    R dl[3], dr[3], n1[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      dl[a] = __ldcs(fgp + a * stride + gid);
      dr[a] = __ldcs(fgp + (3 + a) * stride + gid);
      n1[a] = __ldcs(fgp + (6 + a) * stride + gid);
    }
    const R w = __ldcs(fgp + 9 * stride + gid);
    R vl[5], gl[5][3], vr[5], gr[5][3];
    eval_poly(PolyRef<R>{poly + (int64_t)kPolyStride * o}, dl, vl, gl);
    if (fallback) first_order_if_nonphysical(QA, o, vl, gl);
    if (nb >= 0) {
      eval_poly(PolyRef<R>{poly + (int64_t)kPolyStride * nb}, dr, vr, gr);
      if (fallback) first_order_if_nonphysical(QA, nb, vr, gr);
    } else {
      wall_ghost(P, wall, wall_data(wall_tab, wall), vl, gl, vr, gr);  // the wall's ghost
    }
    bool ok;
    if constexpr (sizeof(R) == 4)
      ok = gp_flux_sides(P, vl, gl, vr, gr, n1, w, dt, acc);  // both sides on packed f32x2
    else
      ok = gp_flux_global(P, vl, gl, vr, gr, n1, w, dt, acc);
    if (!ok) atomicOr(flag, kErrNonphysical);
  }
  // sum the four Gauss points of the face (lanes 4f .. 4f+3 of one warp). Away from walls each
  // exchange halves what a lane carries: lane bit 0 keeps F^n or dF/dt, bit 1 the first three or
  // the last two of it (8 additions a lane instead of 20, the same sums), and writes those.
  if (!__any_sync(0xffffffffu, wall >= 0)) {
    const int b0 = threadIdx.x & 1, b1 = (threadIdx.x >> 1) & 1;
    R y[6];
#pragma unroll
    for (int q = 0; q < 5; ++q)
      y[q] = (b0 ? acc[5 + q] : acc[q]) + __shfl_xor_sync(0xffffffffu, b0 ? acc[q] : acc[5 + q], 1);
    y[5] = R(0);
    R* rec = fface + (int64_t)kFaceStride * f + 5 * b0 + 3 * b1;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const R z = (b1 ? y[3 + q] : y[q]) + __shfl_xor_sync(0xffffffffu, b1 ? y[q] : y[3 + q], 2);
      if (active && (q < 2 || !b1)) rec[q] = z;
    }
    return;
  }
#pragma unroll
  for (int q = 0; q < 10; ++q) {
    acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], 1);
    acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], 2);
  }
  // every lane of the face now holds the sums; lanes 4f + j, j < 3, write the record's part j
  if (active && (gid & 3) < 3) {
    if (wall >= 0) wall_flux_fix(wall, wall_data(wall_tab, wall), acc);
    FaceRec<R>::put(fface + (int64_t)kFaceStride * f, (int)(gid & 3), acc);
  }
}

// rho > 0 and p > 0, the latter as rho E > |m|^2 / 2 (gamma > 1; no division; false for NaN).
__device__ __forceinline__ bool physical(const double q[5]) {
  const double m2 = q[1] * q[1] + q[2] * q[2] + q[3] * q[3];
  return q[0] > 0.0 && q[0] * q[4] > 0.5 * m2;
}

// Sum of the signed face fluxes of one cell (the owner loses the outward flux), in the cell's
// fixed face order: add(q, x) for the components q = kQ0..9 of each face. A cell's chain is a
// CSR entry, then a face record: kB of each are requested together before any is summed. On small
// meshes the stage kernels wait on that chain (8.5 us for 2,048 cells, one face at a time), so
// they take all faces of a cell at once (kFaceBatch; ten stage-pairs of the 8^3-cube mesh 582 ->
// 465 us together with the merged reconstruction launch, 495 with two or five at a time); on
// large ones occupancy is worth more (64^3 cubes, FP32: 66.5 us per stage one at a time, 70.0
// with three; FP64 update of 419,328 cells 46.2 us against 57.4 with six, of 1,048,576 cells 95.5
// against 123, of 55,296 cells 15.2 either way), so kB = 1.
constexpr int kFaceBatch = 6;
template <int kQ0, int kB, class F>
__device__ __forceinline__ void face_loop(int k0, int k1, const int32_t* __restrict__ cf_idx,
                                          const float* __restrict__ fface, F add) {
  for (int k = k0; k < k1; k += kB) {
    int32_t e[kB];
    float4 a[kB], b[kB];
    float2 c[kB];
#pragma unroll
    for (int j = 0; j < kB; ++j) e[j] = k + j < k1 ? __ldg(cf_idx + k + j) : -1;
#pragma unroll
    for (int j = 0; j < kB; ++j) {
      if (e[j] < 0) continue;
      const float* fp = fface + (int64_t)kFaceStride * (e[j] >> 1);
      if (kQ0 < 4) a[j] = __ldg(reinterpret_cast<const float4*>(fp));
      b[j] = __ldg(reinterpret_cast<const float4*>(fp) + 1);
      c[j] = __ldg(reinterpret_cast<const float2*>(fp) + 4);
    }
#pragma unroll
    for (int j = 0; j < kB; ++j) {
      if (e[j] < 0) continue;
      const float x[10] = {a[j].x, a[j].y, a[j].z, a[j].w, b[j].x,
                           b[j].y, b[j].z, b[j].w, c[j].x, c[j].y};
      const bool neg = !(e[j] & 1);
#pragma unroll
      for (int q = kQ0; q < 10; ++q) add(q, neg ? -x[q] : x[q]);
    }
  }
}
template <int kQ0, int kB, class F>
__device__ __forceinline__ void face_loop(int k0, int k1, const int32_t* __restrict__ cf_idx,
                                          const double* __restrict__ fface, F add) {
  for (int k = k0; k < k1; k += kB) {
    int32_t e[kB];
    double2 x[kB][5];
#pragma unroll
    for (int j = 0; j < kB; ++j) e[j] = k + j < k1 ? __ldg(cf_idx + k + j) : -1;
#pragma unroll
    for (int j = 0; j < kB; ++j) {
      if (e[j] < 0) continue;
      const double2* fp =
          reinterpret_cast<const double2*>(fface + (int64_t)kFaceStride * (e[j] >> 1));
#pragma unroll
      for (int q = kQ0 / 2; q < 5; ++q) x[j][q] = __ldg(fp + q);
    }
#pragma unroll
    for (int j = 0; j < kB; ++j) {
      if (e[j] < 0) continue;
      const bool neg = !(e[j] & 1);
#pragma unroll
      for (int q = kQ0; q < 10; ++q) {
        const double v = (q & 1) ? x[j][q / 2].y : x[j][q / 2].x;
        add(q, neg ? -v : v);
      }
    }
  }
}
// FP64 sums of FP64 face fluxes.
template <int kQ0, int kB>
__device__ __forceinline__ void face_sums(int k0, int k1, const int32_t* __restrict__ cf_idx,
                                          const double* __restrict__ fface, double s[10]) {
#pragma unroll
  for (int q = kQ0; q < 10; ++q) s[q] = 0.0;
  face_loop<kQ0, kB>(k0, k1, cf_idx, fface, [&](int q, double x) { s[q] += x; });
}
// FP64 sums of FP32 face fluxes without FP64 arithmetic in the loop (GB300 runs FP64 at 1/64 of
// the FP32 rate): each component is an unevaluated sum h + l + r of floats, TwoSum (Knuth)
// carrying the rounding errors of h into l and those of l into r. As long as r is zero (the
// partial sums fit 48 bits), h + l is the exact sum and the value handed on is rounded once, where
// a double accumulation rounds at every face; otherwise the roundings of r lose about 2^-72 of the
// largest partial sum and the value is rounded twice. A partial sum beyond the FP32 range, or a
// flux that is not finite, leaves NaN in r: such a cell is summed in FP64.
template <int kQ0, int kB>
__device__ __forceinline__ void face_sums(int k0, int k1, const int32_t* __restrict__ cf_idx,
                                          const float* __restrict__ fface, double s[10]) {
  float h[10], l[10], r[10];
#pragma unroll
  for (int q = kQ0; q < 10; ++q) h[q] = l[q] = r[q] = 0.f;
  face_loop<kQ0, kB>(k0, k1, cf_idx, fface, [&](int q, float x) {
    const ff t = two_sum(h[q], x), u = two_sum(l[q], t.l);
    h[q] = t.h;
    l[q] = u.h;
    r[q] = __fadd_rn(r[q], u.l);
  });
  bool rest = false, range = true;
#pragma unroll
  for (int q = kQ0; q < 10; ++q) {
    rest = rest || r[q] != 0.f;
    range = range && fabsf(r[q]) <= FLT_MAX;
    s[q] = widen(l[q]);
  }
  if (!range) {
#pragma unroll
    for (int q = kQ0; q < 10; ++q) s[q] = 0.0;
    face_loop<kQ0, 1>(k0, k1, cf_idx, fface, [&](int q, float x) { s[q] += widen(x); });
    return;
  }
  if (rest) {
#pragma unroll 1
    for (int q = kQ0; q < 10; ++q) {
      // (selected without a dynamic register index)
#pragma unroll
      for (int p = kQ0; p < 10; ++p)
        if (p == q) s[p] += widen(r[p]);
    }
  }
#pragma unroll
  for (int q = kQ0; q < 10; ++q) s[q] += widen(h[q]);
}

// Per cell: L = -(1/|Omega|) sum_f s_f F_f in the cell's fixed face order, and Lt from dF/dt
// (the residual of gks_residual), in FP64, written at the caller's cell index.
template <class R, int kB>
__global__ void __launch_bounds__(256) k_gather(
    int64_t nc, const int32_t* __restrict__ cf_ptr, const int32_t* __restrict__ cf_idx,
    const R* __restrict__ fface, const double* __restrict__ ivol,
    const int32_t* __restrict__ perm, double* __restrict__ L, double* __restrict__ Lt) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nc) return;
  const double iv = ivol[i];
  const int64_t c = perm[i];
  double s[10];
  face_sums<0, kB>(cf_ptr[i], cf_ptr[i + 1], cf_idx, fface, s);
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    L[v * nc + c] = s[v] * iv;
    Lt[v * nc + c] = s[5 + v] * iv;
  }
}

// ------------------------------------------------------------------------------------------
// The two stages of the fourth-order update (Section 3.3) on the gather copy of the state,
// which is the solver state itself: FP64 path [q0..q4, 0] per cell; FP32 path the float-float
// pairs (hi, lo) of each variable. With the cell's face sums s (F^n part) and st (dF/dt part),
// L = s / |Omega|, Lt = st / |Omega|:
//   stage 1: keep L, Lt;           Q*      = Q^n + dt/2 L + dt^2/8 Lt
//   stage 2 (Lt* of Q*):           Q^{n+1} = Q^n + dt L + dt^2/6 (Lt + 2 Lt*)
// FP32 path: every operation in float-float arithmetic, so the update is conservative to about
// 2^-46 relative and issues no FP64 instruction.

// Face sums as float-float pairs, components kQ0..9 (FP32 path).
template <int kQ0, int kB>
__device__ __forceinline__ void face_sums_ff(int k0, int k1, const int32_t* __restrict__ cf_idx,
                                             const float* __restrict__ fface, ff s[10]) {
#pragma unroll
  for (int q = kQ0; q < 10; ++q) s[q] = ff{0.f, 0.f};
  face_loop<kQ0, kB>(k0, k1, cf_idx, fface, [&](int q, float x) {
    const ff t = two_sum(s[q].h, x);
    s[q] = ff{t.h, __fadd_rn(s[q].l, t.l)};
  });
#pragma unroll
  for (int q = kQ0; q < 10; ++q) s[q] = two_sum(s[q].h, s[q].l);
}

template <bool kSecond, int kB>
__global__ void __launch_bounds__(256) k_stage_f(
    int64_t nc, const int32_t* __restrict__ cf_ptr, const int32_t* __restrict__ cf_idx,
    const float* __restrict__ fface, const ff* __restrict__ ivol, ff c1, ff c2,
    ff* __restrict__ L, ff* __restrict__ Lt, float* __restrict__ QA, float* __restrict__ QsA,
    int* flag) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nc) return;
  Gq<float> g;
  ff iv, s[10];
  if (kB > 1) {  // requested before the chain of the face sums
    iv = ivol[i];
    g.load(QA, i);
  }
  face_sums_ff<kSecond ? 5 : 0, kB>(cf_ptr[i], cf_ptr[i + 1], cf_idx, fface, s);
  if (kB == 1) {
    iv = ivol[i];
    g.load(QA, i);
  }
  ff q[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const ff qn{g.hi[v], g.lo[v]};
    const ff lt = ff_mul(s[5 + v], iv);
    if (!kSecond) {  // c1 = dt/2, c2 = dt^2/8
      const ff l = ff_mul(s[v], iv);
      L[v * nc + i] = l;
      Lt[v * nc + i] = lt;
      q[v] = ff_add(qn, ff_add(ff_mul(c1, l), ff_mul(c2, lt)));
    } else {  // c1 = dt, c2 = dt^2/6
      const ff lt2 = ff_add(Lt[v * nc + i], ff_twice(lt));
      q[v] = ff_add(qn, ff_add(ff_mul(c1, L[v * nc + i]), ff_mul(c2, lt2)));
    }
  }
  Gq<float>::store_ff(kSecond ? QA : QsA, i, q);
  // rho > 0 and rho E > |m|^2 / 2 on the leading parts (false for NaN)
  const float m2 = q[1].h * q[1].h + q[2].h * q[2].h + q[3].h * q[3].h;
  if (!(q[0].h > 0.f && q[0].h * q[4].h > 0.5f * m2)) atomicOr(flag, kErrNonphysical);
}

// FP32 reconstruction and flux with the FP64 update (GKS_PREC_MIXED_FP64UPD): the face sums
// accumulate the FP32 face fluxes in FP64, and the update reads and writes the FP64 state
// [5][nc], which is the master copy in this mode; the gather copies the reconstruction reads
// (float pairs) are written from it: Q* by stage 1, Q^{n+1} by stage 2.
template <bool kSecond, int kB>
__global__ void __launch_bounds__(256) k_stage_fd(
    int64_t nc, const int32_t* __restrict__ cf_ptr, const int32_t* __restrict__ cf_idx,
    const float* __restrict__ fface, const double* __restrict__ ivol, double c1, double c2,
    double* __restrict__ L, double* __restrict__ Lt, double* __restrict__ Q,
    float* __restrict__ QA, float* __restrict__ QsA, int* flag) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nc) return;
  double s[10];
  face_sums<kSecond ? 5 : 0, kB>(cf_ptr[i], cf_ptr[i + 1], cf_idx, fface, s);
  const double iv = ivol[i];
  double q[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const double qn = Q[v * nc + i];
    const double lt = s[5 + v] * iv;
    if (!kSecond) {
      const double l = s[v] * iv;
      L[v * nc + i] = l;
      Lt[v * nc + i] = lt;
      q[v] = qn + c1 * l + c2 * lt;
    } else {
      q[v] = qn + c1 * L[v * nc + i] + c2 * (Lt[v * nc + i] + 2.0 * lt);
      Q[v * nc + i] = q[v];
    }
  }
  Gq<float>::store(kSecond ? QA : QsA, i, q);
  // the check in FP32 where that is beyond doubt, else in FP64
  float f[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) f[v] = (float)q[v];
  const float e = f[0] * f[4], m2 = f[1] * f[1] + f[2] * f[2] + f[3] * f[3];
  if (!(f[0] > 1e-15f && e < 1e30f && e - 0.5f * m2 > 1e-5f * e + 1e-30f) && !physical(q))
    atomicOr(flag, kErrNonphysical);
}

template <bool kSecond, int kB>
__global__ void __launch_bounds__(256) k_stage_d(
    int64_t nc, const int32_t* __restrict__ cf_ptr, const int32_t* __restrict__ cf_idx,
    const double* __restrict__ fface, const double* __restrict__ ivol, double c1, double c2,
    double* __restrict__ L, double* __restrict__ Lt, double* __restrict__ QA,
    double* __restrict__ QsA, int* flag) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nc) return;
  const double iv = ivol[i];
  Gq<double> g;
  g.load(QA, i);
  double s[10];
  face_sums<kSecond ? 5 : 0, kB>(cf_ptr[i], cf_ptr[i + 1], cf_idx, fface, s);
  double q[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const double lt = s[5 + v] * iv;
    if (!kSecond) {
      const double l = s[v] * iv;
      L[v * nc + i] = l;
      Lt[v * nc + i] = lt;
      q[v] = g.q[v] + c1 * l + c2 * lt;
    } else {
      q[v] = g.q[v] + c1 * L[v * nc + i] + c2 * (Lt[v * nc + i] + 2.0 * lt);
    }
  }
  Gq<double>::store(kSecond ? QA : QsA, i, q);
  if (!physical(q)) atomicOr(flag, kErrNonphysical);
}

// ------------------------------------------------------------------------------------------
// The two-stage combinations of Section 3.3 on caller arrays of n values, for a differentiable
// rollout built from residual calls: stage 1 out = Q + c1 L + c2 Lt (c1 = dt/2, c2 = dt^2/8),
// stage 2 out = Q + c1 L + c2 (Lt + 2 Lts) (c1 = dt, c2 = dt^2/6); and their transposes.
__global__ void __launch_bounds__(256) k_s2o4_stage(int64_t n, int stage, double c1, double c2,
                                                    const double* __restrict__ Q,
                                                    const double* __restrict__ L,
                                                    const double* __restrict__ Lt,
                                                    const double* __restrict__ Lts,
                                                    double* __restrict__ out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double lt = stage == 1 ? Lt[i] : Lt[i] + 2.0 * Lts[i];
  out[i] = Q[i] + c1 * L[i] + c2 * lt;
}
__global__ void __launch_bounds__(256) k_s2o4_stage_vjp(int64_t n, int stage, double c1,
                                                        double c2, const double* __restrict__ g,
                                                        double* __restrict__ gQ,
                                                        double* __restrict__ gL,
                                                        double* __restrict__ gLt,
                                                        double* __restrict__ gLts) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double gi = g[i];
  gQ[i] = gi;
  gL[i] = c1 * gi;
  gLt[i] = c2 * gi;
  if (stage == 2) gLts[i] = 2.0 * c2 * gi;
}

// ------------------------------------------------------------------------------------------
// Implicit step (Section 4): backward Euler with the residual's change linearised by the flux
// splitting (T(Q_i) + T(Q_p) - r (Q_p - Q_i))/2 . n S, solved by Jacobi iterations:
//   (|Omega_i|/dt + 1/2 sum_f r_f S_f) dQ_i^(k)
//     = |Omega_i| Res_i - 1/2 sum_f [T_n(Q_p + dQ_p^(k-1)) - T_n(Q_p) - r_f dQ_p^(k-1)] S_f,
// |Omega_i| Res_i = s + dt/2 st (the face sums of F^n and dF/dt: the step-averaged GKS flux),
// r_f = max over the two sides of |U . n| + c at Q^n, n out of cell i; a wall face couples the
// cell to its mirror image. The Euler-flux change is formed from the increments themselves
// (du = (dm - u drho)/rho', dp = (gamma - 1)(dE - (m . du + dm . u')/2)), so no two nearly equal
// fluxes are subtracted.

// Per-cell values of the implicit step at Q^n: 1/rho, p, sound speed.
template <class R>
struct JPrim {
  R ir, p, c, pad;
};
// Four values of R (normal and area of a cell's face, JPrim) in one or two 16-byte loads.
template <class R>
struct __align__(16) R4 {
  R x, y, z, w;
};
__device__ __forceinline__ R4<float> ld4(const float* p) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(p));
  return {a.x, a.y, a.z, a.w};
}
__device__ __forceinline__ R4<double> ld4(const double* p) {
  const double2 a = __ldg(reinterpret_cast<const double2*>(p));
  const double2 b = __ldg(reinterpret_cast<const double2*>(p) + 1);
  return {a.x, a.y, b.x, b.y};
}
template <class R>
__device__ __forceinline__ JPrim<R> load_prim(const R* __restrict__ prim, int64_t c) {
  const R4<R> a = ld4(prim + 4 * c);
  return {a.x, a.y, a.z, R(0)};
}
// Iterates: one record of kJdq values per cell.
template <class R>
constexpr int kJdq = sizeof(R) == 4 ? 8 : 6;
__device__ __forceinline__ void load_dq(const float* __restrict__ dQ, int64_t c, float d[5]) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(dQ + 8 * c));
  d[0] = a.x; d[1] = a.y; d[2] = a.z; d[3] = a.w;
  d[4] = __ldg(dQ + 8 * c + 4);
}
__device__ __forceinline__ void load_dq(const double* __restrict__ dQ, int64_t c, double d[5]) {
  const double2* p = reinterpret_cast<const double2*>(dQ + 6 * c);
  const double2 a = __ldg(p), b = __ldg(p + 1);
  d[0] = a.x; d[1] = a.y; d[2] = b.x; d[3] = b.y;
  d[4] = __ldg(dQ + 6 * c + 4);
}
__device__ __forceinline__ void store_dq(float* __restrict__ dQ, int64_t c, const float d[5]) {
  *reinterpret_cast<float4*>(dQ + 8 * c) = make_float4(d[0], d[1], d[2], d[3]);
  dQ[8 * c + 4] = d[4];
}
__device__ __forceinline__ void store_dq(double* __restrict__ dQ, int64_t c, const double d[5]) {
  double2* p = reinterpret_cast<double2*>(dQ + 6 * c);
  p[0] = make_double2(d[0], d[1]);
  p[1] = make_double2(d[2], d[3]);
  dQ[6 * c + 4] = d[4];
}
// State of a cell from its gather copy in precision R (the leading parts of float-float pairs).
__device__ __forceinline__ void state_of(const float* __restrict__ QA, int64_t c, float q[5]) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(QA + 12 * c));
  q[0] = a.x; q[1] = a.y; q[2] = a.z; q[3] = a.w;
  q[4] = __ldg(QA + 12 * c + 4);
}
__device__ __forceinline__ void state_of(const double* __restrict__ QA, int64_t c, double q[5]) {
  const double2* p = reinterpret_cast<const double2*>(QA + 6 * c);
  const double2 a = __ldg(p), b = __ldg(p + 1);
  q[0] = a.x; q[1] = a.y; q[2] = b.x; q[3] = b.y;
  q[4] = __ldg(QA + 6 * c + 4);
}
template <class R>
__device__ __forceinline__ JPrim<R> prim_of(const R q[5], R gm1) {
  JPrim<R> w;
  w.ir = R(1) / q[0];
  w.p = gm1 * (q[4] - R(0.5) * (q[1] * (q[1] * w.ir) + q[2] * (q[2] * w.ir) +
                                q[3] * (q[3] * w.ir)));
  const R c2 = (gm1 + R(1)) * w.p * w.ir;
  w.c = sqrt(c2 > R(0) ? c2 : R(0));
  w.pad = R(0);
  return w;
}
template <class R>
__device__ __forceinline__ R wave_speed(const R q[5], const JPrim<R>& w, const R n[3]) {
  return fabs(q[1] * w.ir * n[0] + q[2] * w.ir * n[1] + q[3] * w.ir * n[2]) + w.c;
}
template <class R>
__device__ __forceinline__ void euler_flux_change(const R q[5], R ir, R p, const R d[5],
                                                  const R n[3], R gm1, R out[5]) {
  const R ir1 = R(1) / (q[0] + d[0]);
  R u[3], du[3], u1[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    u[a] = q[1 + a] * ir;
    du[a] = (d[1 + a] - u[a] * d[0]) * ir1;
    u1[a] = u[a] + du[a];
  }
  const R un = u[0] * n[0] + u[1] * n[1] + u[2] * n[2];
  const R dun = du[0] * n[0] + du[1] * n[1] + du[2] * n[2], un1 = un + dun;
  const R dp = gm1 * (d[4] - R(0.5) * (q[1] * du[0] + q[2] * du[1] + q[3] * du[2] +
                                       d[1] * u1[0] + d[2] * u1[1] + d[3] * u1[2]));
  out[0] = d[1] * n[0] + d[2] * n[1] + d[3] * n[2];
#pragma unroll
  for (int a = 0; a < 3; ++a) out[1 + a] = d[1 + a] * un1 + q[1 + a] * dun + dp * n[a];
  out[4] = (d[4] + dp) * un1 + (q[4] + p) * dun;
}

// The wall's ghost of a cell state q and of an increment d of it: q_g = G(q), d_g = G(q + d) -
// G(q), with G the value part of wall_ghost. The slip and adiabatic maps are linear, so
// d_g = G(d); the isothermal map's energy row holds |m|^2 / rho, whose change is formed as
// (2 m . dm + |dm|^2 - |m|^2 drho / rho) / (rho + drho) without cancellation.
template <class R>
__device__ __forceinline__ void wall_cell_ghost(const FluxParams<R>& P, int code,
                                                const WallData<R>& wd, const R q[5], R qg[5]) {
  const R zg[5][3] = {};
  R gg[5][3];
  wall_ghost(P, code, wd, q, zg, qg, gg);
}
template <class R>
__device__ __forceinline__ void wall_cell_ghost_inc(const FluxParams<R>& P, int code,
                                                    const WallData<R>& wd, const R q[5],
                                                    const R d[5], R dg[5]) {
  const R zg[5][3] = {};
  R gg[5][3];
  if (code >= 12) {  // far field: the change of the characteristic state
    R q1[5], g0[5], g1[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) q1[v] = q[v] + d[v];
    wall_ghost(P, code, wd, q, zg, g0, gg);
    wall_ghost(P, code, wd, q1, zg, g1, gg);
#pragma unroll
    for (int v = 0; v < 5; ++v) dg[v] = g1[v] - g0[v];
    return;
  }
  if (code < 6 || wd.Tw <= R(0)) {
    wall_ghost(P, code, wd, d, zg, dg, gg);
    return;
  }
  const R u0 = wd.uw[0], u1 = wd.uw[1], u2 = wd.uw[2];
  const R uw2 = u0 * u0 + u1 * u1 + u2 * u2;
  dg[0] = d[0];
  dg[1] = R(2) * u0 * d[0] - d[1];
  dg[2] = R(2) * u1 * d[0] - d[2];
  dg[3] = R(2) * u2 * d[0] - d[3];
  const R mdm = q[1] * d[1] + q[2] * d[2] + q[3] * d[3];
  const R dm2 = d[1] * d[1] + d[2] * d[2] + d[3] * d[3];
  const R m2 = q[1] * q[1] + q[2] * q[2] + q[3] * q[3];
  dg[4] = (R(2) * wd.Tw / (P.gamma - R(1)) + R(2) * uw2) * d[0] - d[4] +
          (R(2) * mdm + dm2 - m2 * d[0] / q[0]) / (q[0] + d[0]) -
          R(2) * (u0 * d[1] + u1 * d[2] + u2 * d[3]);
}

// Plan of the implicit step, tile-interleaved [tile][kCellFaces][32] in the order of a cell's
// faces: the cell across each (nb >= 0, -1 - wall code at a boundary face, kNoFace beyond the
// cell's faces) and the unit normal out of the cell with the face area. One coalesced read in
// place of the chain CSR entry -> face -> owner, neighbour, wall and normal of every sweep.
constexpr int32_t kNoFace = INT32_MIN;
template <class R>
__global__ void k_jacobi_plan(int64_t nc, int64_t n_tiles, const int32_t* __restrict__ cf_ptr,
                              const int32_t* __restrict__ cf_idx,
                              const int32_t* __restrict__ f_owner,
                              const int32_t* __restrict__ f_nb, const int8_t* __restrict__ f_wall,
                              const R* __restrict__ fn, int32_t* __restrict__ jnb,
                              R* __restrict__ jn) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n_tiles * kTile) return;
  const int64_t at = i / kTile * kCellFaces * kTile + i % kTile;
  const int k0 = i < nc ? cf_ptr[i] : 0, nk = i < nc ? cf_ptr[i + 1] - k0 : 0;
  for (int j = 0; j < kCellFaces; ++j) {
    const int64_t o = at + (int64_t)j * kTile;
    if (j >= nk) {
      jnb[o] = kNoFace;
      for (int a = 0; a < 4; ++a) jn[4 * o + a] = R(0);
      continue;
    }
    const int32_t e = cf_idx[k0 + j];
    const int64_t f = e >> 1;
    const bool nbside = e & 1;
    const int32_t p = nbside ? f_owner[f] : f_nb[f];
    jnb[o] = p >= 0 ? p : -1 - f_wall[f];
    for (int a = 0; a < 3; ++a) jn[4 * o + a] = nbside ? -fn[4 * f + a] : fn[4 * f + a];
    jn[4 * o + 3] = fn[4 * f + 3];
  }
}
template <class R>
__global__ void __launch_bounds__(256) k_jacobi_prim(int64_t nc, const R* __restrict__ QA, R gm1,
                                                     R* __restrict__ prim) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nc) return;
  R q[5];
  state_of(QA, i, q);
  const JPrim<R> w = prim_of(q, gm1);
  *reinterpret_cast<R4<R>*>(prim + 4 * i) = {w.ir, w.p, w.c, R(0)};
}

// Both kernels below wait on the gathers of a cell's neighbours in FP32, and on the FP64 pipe in
// FP64. The plan's coalesced entries, one record per cell for the iterate, and 1/rho, p and c per
// cell in place of per face took an FP32 step's init and three sweeps from 80 to 65 us (131,072
// cells, median launches), the FP64 one with its primitives from 548 to 415 us (131,072 cells) and
// from 258 to 163 us (48,000 cells, where blocks of 256 threads, 188 of them, left every second SM
// with twice the work of the others: 234 us). Requesting two, three or six faces of a cell together
// took 8, 10 and 31 us more (FP32).
template <class R>
__global__ void __launch_bounds__(256) k_jacobi_init(
    int64_t nc, const int32_t* __restrict__ cf_ptr, const int32_t* __restrict__ cf_idx,
    const int32_t* __restrict__ jnb, const R* __restrict__ jn, const R* __restrict__ fface,
    const double* __restrict__ vol, double dt, const R* __restrict__ QA,
    R* __restrict__ prim, FluxParams<R> P, const R* __restrict__ wall_tab, R* __restrict__ Rv,
    R* __restrict__ D, R* __restrict__ hrs, R* __restrict__ dQ0) {
  constexpr bool kPrimed = sizeof(R) == 8;  // prim filled by k_jacobi_prim
  const R gm1 = P.gamma - R(1);
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nc) return;
  R qi[5];
  state_of(QA, i, qi);
  const JPrim<R> wi = kPrimed ? load_prim(prim, i) : prim_of(qi, gm1);
  if (!kPrimed) *reinterpret_cast<R4<R>*>(prim + 4 * i) = {wi.ir, wi.p, wi.c, R(0)};
  R dsum = R(0);
  const int64_t at = i / kTile * kCellFaces * kTile + i % kTile;
  int32_t nba[kCellFaces];
#pragma unroll
  for (int j = 0; j < kCellFaces; ++j) nba[j] = __ldg(jnb + at + j * kTile);
#pragma unroll
  for (int j = 0; j < kCellFaces; ++j) {
    const int32_t nb = nba[j];
    if (nb == kNoFace) break;
    const R4<R> n4 = ld4(jn + 4 * (at + j * kTile));
    const R n[3] = {n4.x, n4.y, n4.z};
    R q[5];
    JPrim<R> w;
    if (nb >= 0) {
      state_of(QA, nb, q);
      w = kPrimed ? load_prim(prim, nb) : prim_of(q, gm1);
    } else {
      const int wall = -1 - nb;
      wall_cell_ghost(P, wall, wall_data(wall_tab, wall), qi, q);
      w = prim_of(q, gm1);
    }
    const R h = R(0.5) * fmax(wave_speed(qi, wi, n), wave_speed(q, w, n)) * n4.w;
    hrs[at + j * kTile] = h;
    dsum += h;
  }
  R res[5];
  if constexpr (std::is_same<R, float>::value) {
    ff s[10];
    face_sums_ff<0, 1>(cf_ptr[i], cf_ptr[i + 1], cf_idx, fface, s);
    const ff h = ff_from(0.5 * dt);
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const ff x = ff_add(s[v], ff_mul(h, s[5 + v]));
      res[v] = x.h + x.l;
    }
  } else {
    double s[10];
    face_sums<0, 1>(cf_ptr[i], cf_ptr[i + 1], cf_idx, fface, s);
#pragma unroll
    for (int v = 0; v < 5; ++v) res[v] = s[v] + 0.5 * dt * s[5 + v];
  }
  const R d = (R)(vol[i] / dt) + dsum;
  D[i] = d;
  const R id = R(1) / d;
  R d0[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    Rv[v * nc + i] = res[v];
    d0[v] = res[v] * id;
  }
  store_dq(dQ0, i, d0);
}

template <class R, bool kLast>
__global__ void __launch_bounds__(256) k_jacobi_sweep(
    int64_t nc, const int32_t* __restrict__ jnb, const R* __restrict__ jn,
    const R* __restrict__ QA, const R* __restrict__ prim,
    const R* __restrict__ Rv, const R* __restrict__ D, const R* __restrict__ hrs,
    const R* __restrict__ dQin, R* __restrict__ dQout, R* __restrict__ QAout, FluxParams<R> P,
    const R* __restrict__ wall_tab, int* flag) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nc) return;
  const R gm1 = P.gamma - R(1);
  R acc[5] = {R(0), R(0), R(0), R(0), R(0)};
  const int64_t at = i / kTile * kCellFaces * kTile + i % kTile;
  int32_t nba[kCellFaces];
#pragma unroll
  for (int j = 0; j < kCellFaces; ++j) nba[j] = __ldg(jnb + at + j * kTile);
#pragma unroll
  for (int j = 0; j < kCellFaces; ++j) {
    const int32_t nb = nba[j];
    if (nb == kNoFace) break;
    const int64_t c = nb >= 0 ? nb : i;
    R q[5], dp[5];
    state_of(QA, c, q);
    JPrim<R> w = load_prim(prim, c);
    load_dq(dQin, c, dp);
    const R4<R> n4 = ld4(jn + 4 * (at + j * kTile));
    const R h = __ldg(hrs + at + j * kTile);
    if (nb < 0) {  // the wall's ghost of the cell and of its increment
      const int wall = -1 - nb;
      R qg[5], dg[5];
      const WallData<R> wd = wall_data(wall_tab, wall);
      wall_cell_ghost(P, wall, wd, q, qg);
      wall_cell_ghost_inc(P, wall, wd, q, dp, dg);
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        q[v] = qg[v];
        dp[v] = dg[v];
      }
      w = prim_of(q, gm1);
    }
    const R n[3] = {n4.x, n4.y, n4.z}, hS = R(0.5) * n4.w;
    R dT[5];
    euler_flux_change(q, w.ir, w.p, dp, n, gm1, dT);
#pragma unroll
    for (int v = 0; v < 5; ++v) acc[v] += hS * dT[v] - h * dp[v];
  }
  const R id = R(1) / D[i];
  R d[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) d[v] = (Rv[v * nc + i] - acc[v]) * id;
  if (!kLast) {
    store_dq(dQout, i, d);
    return;
  }
  // Q^{n+1} = Q^n + dQ, written to the other gather copy (neighbours still read Q^n)
  if constexpr (std::is_same<R, float>::value) {
    Gq<float> g;
    g.load(QA, i);
    ff q[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) q[v] = ff_add(ff{g.hi[v], g.lo[v]}, ff{d[v], 0.f});
    Gq<float>::store_ff(QAout, i, q);
    const float m2 = q[1].h * q[1].h + q[2].h * q[2].h + q[3].h * q[3].h;
    if (!(q[0].h > 0.f && q[0].h * q[4].h > 0.5f * m2)) atomicOr(flag, kErrNonphysical);
  } else {
    Gq<double> g;
    g.load(QA, i);
    double q[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) q[v] = g.q[v] + d[v];
    Gq<double>::store(QAout, i, q);
    if (!physical(q)) atomicOr(flag, kErrNonphysical);
  }
}

__global__ void k_unpack(int64_t nc, const float* __restrict__ QA, double* __restrict__ Q) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nc) return;
  Gq<float> g;
  g.load(QA, i);
#pragma unroll
  for (int v = 0; v < 5; ++v) Q[v * nc + i] = unpack_value(g, v);
}

// The FP64 state in caller order from its gather copy.
template <class R>
__global__ void k_unpack_out(int64_t nc, const int32_t* __restrict__ perm,
                             const R* __restrict__ QA, double* __restrict__ dst) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nc) return;
  const int64_t c = perm[i];
  Gq<R> g;
  g.load(QA, i);
#pragma unroll
  for (int v = 0; v < 5; ++v) dst[v * nc + c] = unpack_value(g, v);
}

// Caller order -> internal order: the values (dst, may be null) and the gather copy (gq, may be
// null); flag != null also checks the state.
template <class R>
__global__ void k_permute_in(int64_t nc, const int32_t* __restrict__ perm,
                             const double* __restrict__ src, double* __restrict__ dst, R* gq,
                             int* flag) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nc) return;
  const int64_t c = perm[i];
  double q[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) q[v] = src[v * nc + c];
  if (dst) {
#pragma unroll
    for (int v = 0; v < 5; ++v) dst[v * nc + i] = q[v];
  }
  if (gq) Gq<R>::store(gq, i, q);
  if (flag && !physical(q)) atomicOr(flag, kErrNonphysical);
}
__global__ void k_permute_out(int64_t nc, const int32_t* __restrict__ perm,
                              const double* __restrict__ src, double* __restrict__ dst) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nc) return;
  const int64_t c = perm[i];
#pragma unroll
  for (int v = 0; v < 5; ++v) dst[v * nc + c] = src[v * nc + i];
}
// Time-step bound h / (|U| + c + 2 mu / (rho h)) of a cell and its state check, in FP64.
struct DtParams {
  double gamma, mu, T_ref, mu_pow;
  int power;
  float gm1;  // gamma - 1 of the FP64 gamma, for the FP32 estimate
  float cut;  // smallest share of the internal energy in rho E that the estimate takes
};
// FP32 rounds rho E and |m|^2 / 2 to about 5e-7 of rho E. In the sum of the speeds that is at most
// 1e-4 down to an internal share of 1e-5, as the speed of sound is small beside |U| there; the
// viscosity of the power law has it in full, times the exponent over the share.
inline float dt_cut(int power, double mu_pow) {
  return power ? std::max(1e-5f, 4e-3f * (float)fabs(mu_pow)) : 1e-5f;
}
__device__ __forceinline__ double dt_bound(const double q[5], double h, const DtParams& P) {
  const double u2 = (q[1] * q[1] + q[2] * q[2] + q[3] * q[3]) / (q[0] * q[0]);
  const double p = (P.gamma - 1.0) * (q[4] - 0.5 * q[0] * u2);
  const double c = sqrt(P.gamma * p / q[0]);
  // viscosity at the cell's temperature p / rho (the power law of Section 5.4, else constant)
  const double mue = P.power ? P.mu * pow(p / (q[0] * P.T_ref), P.mu_pow) : P.mu;
  return h / (sqrt(u2) + c + 2.0 * mue / (q[0] * h));
}
// The same in FP32, to better than 6e-4 (1e-4 without the power law; the margin of k_dt_partial is
// 2^-9 = 2e-3 for two such errors) for states and sizes whose products stay inside the FP32 range;
// 0 for any other, which every caller takes as "evaluate in FP64". ok: rho > 0 and p > 0 beyond
// doubt. With w = rho p the three speeds have 1 / rho in common (c = sqrt(gamma w) / rho), so that
// the lower limits of w, E and h keep every quantity that matters normal: what may still be
// subnormal beside them (a kinetic energy, a viscous term) is below 1e-7 of the sum.
__device__ __forceinline__ float dt_bound_f32(const float q[5], float h, const DtParams& P,
                                              bool& ok) {
  const float m2 = q[1] * q[1] + q[2] * q[2] + q[3] * q[3];
  const float e = q[0] * q[4], d = e - 0.5f * m2, w = P.gm1 * d;
  ok = q[0] > 1e-15f && q[0] < 1e15f && h > 1e-15f && h < 1e15f && q[4] > 1e-25f &&
       q[4] < 1e15f && d > P.cut * e && w > 1e-30f;
  if (!ok) return 0.f;
  const float ir = 1.f / q[0];
  float mue = (float)P.mu;
  if (P.power) {
    const float T = w * ir * ir, t = T / (float)P.T_ref;
    if (!(T > 1e-30f && t > 1e-10f && t < 1e10f)) return 0.f;
    mue *= powf(t, (float)P.mu_pow);
  }
  const float b = h / ((sqrtf(m2) + sqrtf((float)P.gamma * w) + 2.f * mue / h) * ir);
  return b > 1e-30f && b < 1e30f ? b : 0.f;
}

// The smallest bound of all cells, bit for bit the FP64 one: a block takes kCells cells per
// thread at a time, bounds them in FP32, and evaluates in FP64 only those within 2^-9 of the
// block's smallest (or outside the estimate's range), which contain its FP64 minimum as two errors
// of the estimate are below that. The FP64 evaluation of every cell (two divisions, two square roots and a
// third division on a pipe of 1/64 of the FP32 rate, 44 us for 442,368 cells) and the passes that
// unpacked and checked the state before it (25 us) are gone: 69 -> 16 us together. Each block
// evaluates at least one warp in FP64, so large meshes take four cells per thread (a call on
// 442,368 cells 31.6 us, 43.2 with one; on 1,048,576 cells 43 and 76 us); below a block per SM
// that way, one cell per thread spreads the FP64 work where many cells are alike (60,000 cells of
// the Riemann tube 35 us, 45 with four).
constexpr int kDtThreads = 256;
constexpr int kDtMaxBlocks = 8192;

// FP64 state of cell i: Q64 (the FP64-update mode's master copy) or the gather copy.
template <class R>
__device__ __forceinline__ void state64(const Gq<R>& g, const double* Q64, int64_t nc, int64_t i,
                                        double q[5]) {
#pragma unroll
  for (int v = 0; v < 5; ++v) q[v] = Q64 ? Q64[v * nc + i] : unpack_value(g, v);
}

template <class R, int kCells>
__global__ void __launch_bounds__(kDtThreads) k_dt_partial(
    int64_t nc, const R* __restrict__ QA, const double* __restrict__ Q64,
    const double* __restrict__ hdt, DtParams P, double* partial, int* flag) {
  __shared__ double red[kDtThreads / 32];
  __shared__ float redf[kDtThreads / 32];
  double best = DBL_MAX;
  constexpr int64_t kChunk = (int64_t)kDtThreads * kCells;
  for (int64_t base = blockIdx.x * kChunk; base < nc; base += gridDim.x * kChunk) {
    float b[kCells], lo = FLT_MAX;
#pragma unroll
    for (int j = 0; j < kCells; ++j) {
      const int64_t i = base + j * kDtThreads + threadIdx.x;
      b[j] = FLT_MAX;
      if (i >= nc) continue;
      Gq<R> g;
      g.load(QA, i);
      float q[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) q[v] = (float)g.value(v);
      bool ok;
      b[j] = dt_bound_f32(q, (float)hdt[i], P, ok);
      if (!ok) {
        double qd[5];
        state64(g, Q64, nc, i, qd);
        if (!physical(qd)) atomicOr(flag, kErrNonphysical);
      }
      if (b[j] > 0.f) lo = fminf(lo, b[j]);
    }
    for (int o = 16; o > 0; o >>= 1) lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    if ((threadIdx.x & 31) == 0) redf[threadIdx.x >> 5] = lo;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kDtThreads / 32; ++k) lo = fminf(lo, redf[k]);
    __syncthreads();
    lo *= 1.f + 1.f / 512.f;
#pragma unroll
    for (int j = 0; j < kCells; ++j) {
      const int64_t i = base + j * kDtThreads + threadIdx.x;
      if (i >= nc || !(b[j] <= lo)) continue;
      Gq<R> g;
      g.load(QA, i);
      double q[5];
      state64(g, Q64, nc, i, q);
      best = fmin(best, dt_bound(q, hdt[i], P));  // NaN states are caught by the state check
    }
  }
  for (int o = 16; o > 0; o >>= 1) best = fmin(best, __shfl_xor_sync(0xffffffffu, best, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = best;
  __syncthreads();
  if (threadIdx.x < 32) {
    best = threadIdx.x < kDtThreads / 32 ? red[threadIdx.x] : DBL_MAX;
    for (int o = 16; o > 0; o >>= 1) best = fmin(best, __shfl_xor_sync(0xffffffffu, best, o));
    if (threadIdx.x == 0) partial[blockIdx.x] = best;
  }
}
__global__ void k_dt_final(const double* partial, int n, double* out) {
  __shared__ double red[32];
  double best = DBL_MAX;
  for (int k = threadIdx.x; k < n; k += blockDim.x) best = fmin(best, partial[k]);
  for (int o = 16; o > 0; o >>= 1) best = fmin(best, __shfl_xor_sync(0xffffffffu, best, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = best;
  __syncthreads();
  if (threadIdx.x < 32) {
    best = threadIdx.x < (int)(blockDim.x / 32) ? red[threadIdx.x] : DBL_MAX;
    for (int o = 16; o > 0; o >>= 1) best = fmin(best, __shfl_xor_sync(0xffffffffu, best, o));
    if (threadIdx.x == 0) *out = best;
  }
}

}  // namespace

// Largest dynamic shared memory of one block (227 KB on this architecture).
constexpr size_t kMaxBlockSmem = 227 * 1024;

// Shared memory of one SM and the part the hardware keeps for each resident block.
constexpr size_t kSmemPerSM = 228 * 1024, kSmemPerBlockReserved = 1024;

inline int recon_blocks_per_sm(size_t smem) {
  return (int)(kSmemPerSM / (smem + kSmemPerBlockReserved));
}

// One launch over the tiles of ranges r0 .. r1 - 1 with stencil, entry and slot bounds K, S, M.
template <class R, bool kPf, bool kStB>
void launch_recon_ranges(const DevMesh& m, const GeoR<R>& g, const KParams<R>& p, const R* QA,
                         R* poly, int* flag, int r0, int r1, int K, int S, int M, size_t smem,
                         cudaStream_t st) {
  ReconSet set;
  set.n = r1 - r0;
  for (int r = r0; r < r1; ++r)
    set.r[r - r0] = ReconUni{m.rr.uni[r], m.rr.K[r],  m.rr.S[r], m.rr.cnt[r],
                             m.rr.st0[r], m.rr.sb0[r], m.rr.t0[r]};
  auto run = [&](auto kern, const auto& arg) {
    // the limit belongs to the kernel, not to this mesh: always the same value, so that solvers of
    // other sizes in other threads cannot lower it before the launch (a failure is left to the
    // caller's check)
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kMaxBlockSmem) != cudaSuccess)
      return;
    kern<<<(unsigned)(m.rr.t1[r1 - 1] - m.rr.t0[r0]), kReconThreads, smem, st>>>(
        m.nc, m.rr.t0[r0], K, S, M, arg, QA, m.t_K, m.t_cnt, m.t_st, m.t_sb, m.t_idx, g.Ap, g.Bp,
        g.cell, p.weno_gamma, p.weno_eps, p.weno_pow, poly, flag, p.wait_tries, p.withhold);
  };
  if (r1 - r0 > 1)
    run(k_recon<R, kPf, kStB, true>, set);
  else
    run(k_recon<R, kPf, kStB, false>, set.r[0]);
}

// Ghost slots of moving no-slip walls and far-field planes: QA[nc + g] = the image's flow
// variables from QA[g_src[g]]. Linear slots apply their composed map; the others apply the
// maps of their planes in order (slip: normal momentum negated; no-slip: rho kept,
// m -> 2 U_w rho - m, E -> E + 2 |U_w|^2 rho - 2 U_w . m; far field: the characteristic
// state), in precision R.
template <class R>
__global__ void __launch_bounds__(128) k_ghost_fill(int64_t nc, int64_t ng,
                                                    const int32_t* __restrict__ src,
                                                    const double* __restrict__ map,
                                                    const float* __restrict__ mapf,
                                                    const uint8_t* __restrict__ chain, int bcs,
                                                    FluxParams<R> P, const R* __restrict__ wall_tab,
                                                    R* QA) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= ng) return;
  Gq<R> g;
  g.load(QA, src[k]);
  if (const int code = chain[k]) {
    R q[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) q[v] = (R)g.value(v);
    for (int s = 0; s < 2; ++s) {
      const int w = ((code >> (3 * s)) & 7) - 1;
      if (w < 0) break;
      const int ax = w % 3, kind = (bcs >> (2 * ax)) & 3;
      if (kind == 1) {
        q[1 + ax] = -q[1 + ax];
      } else if (kind == 2) {
        const R* t = wall_tab + kPlaneStride * w;
        const R um = t[0] * q[1] + t[1] * q[2] + t[2] * q[3];
        q[4] = q[4] + R(2) * (t[0] * t[0] + t[1] * t[1] + t[2] * t[2]) * q[0] - R(2) * um;
#pragma unroll
        for (int a = 0; a < 3; ++a) q[1 + a] = R(2) * t[a] * q[0] - q[1 + a];
      } else {
        R o[5];
        farfield_state(P, wall_tab + kPlaneStride * w + 4, ax, w >= 3 ? R(1) : R(-1), q, o);
#pragma unroll
        for (int v = 0; v < 5; ++v) q[v] = o[v];
      }
    }
    if constexpr (std::is_same<R, float>::value) {
      ff o[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) o[v] = ff{q[v], 0.f};
      Gq<float>::store_ff(QA, nc + k, o);
    } else {
      Gq<double>::store(QA, nc + k, q);
    }
    return;
  }
  if constexpr (std::is_same<R, float>::value) {
    const float* c = mapf + 20 * k;
    auto co = [&](int j) { return ff{c[2 * j], c[2 * j + 1]}; };
    ff q[5], o[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) q[v] = ff{g.hi[v], g.lo[v]};
    o[0] = q[0];
    o[4] = ff_add(q[4], ff_mul(co(6), q[0]));
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float sj = c[2 * j];  // +-1, exact
      o[1 + j] = ff_add(ff{sj * q[1 + j].h, sj * q[1 + j].l}, ff_mul(co(3 + j), q[0]));
      o[4] = ff_add(o[4], ff_mul(co(7 + j), q[1 + j]));
    }
    Gq<float>::store_ff(QA, nc + k, o);
  } else {
    const double* c = map + 10 * k;
    double o[5];
    o[0] = g.q[0];
    o[4] = g.q[4] + c[6] * g.q[0];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      o[1 + j] = c[j] * g.q[1 + j] + c[3 + j] * g.q[0];
      o[4] += c[7 + j] * g.q[1 + j];
    }
    Gq<double>::store(QA, nc + k, o);
  }
}

// Threads per block of the per-cell kernels: 256, or 64 where 256 would leave SMs without a block.
inline int cell_threads(int64_t nc) { return nc < 256 * 152 ? 64 : 256; }
// Largest number of tiles reconstructed by one launch over all ranges: one wave of the FP32
// kernel (5 blocks on each of 152 SMs). Below it the launches and the streams' events cost more
// than the ranges gain from shared memory of their own size: ten steps of the 8^3-cube mesh 564
// (four launches) -> 485 us, of the 16^3-cube mesh (512 tiles) 700 -> 663 us; at 24^3 cubes
// (1,728 tiles) 1.299 against 1.278 ms, at 64^3 cubes a pass takes 0.381 ms in one launch against
// 0.356.
constexpr int64_t kReconMergeTiles = 760;
inline bool recon_merged(const TileRanges& rr) {
  return rr.n > 1 && rr.t1[rr.n - 1] - rr.t0[0] <= kReconMergeTiles;
}
int recon_launches(const DevMesh& m) {
  int n = m.ng > 0 ? 1 : 0;  // the ghost refresh of moving no-slip walls and far-field planes
  if (recon_merged(m.rr)) return n + 1;
  for (int r = 0; r < m.rr.n; ++r) n += m.rr.t1[r] > m.rr.t0[r] ? 1 : 0;
  return n;
}
// One launch per tile range (one over all of them on small meshes), the bulk-copy variant
// whenever its shared memory fits a block. The ranges are independent: with fj, range r > 0 runs on auxiliary stream r - 1, forked from and
// joined back into st, so that the ranges' blocks share the GPU.
template <class R>
void launch_recon(const DevMesh& m, const GeoR<R>& g, const KParams<R>& p, const R* QA,
                  R* poly, int* flag, cudaStream_t st, const ForkJoin* fj) {
  // the ghost slots beyond nc belong to the reconstruction: refresh them from the state first
  if (m.ng > 0)
    k_ghost_fill<R><<<blocks_for(m.ng, 128), 128, 0, st>>>(
        m.nc, m.ng, m.g_src, m.g_map, m.g_mapf, m.g_chain, m.bcs, flux_params(p),
        wall_table<R>(m), const_cast<R*>(QA));
  const TileRanges& rr = m.rr;
  auto launch = [&](int r0, int r1, cudaStream_t s) {
    int K = 0, S = 0, M = 0;
    for (int r = r0; r < r1; ++r) {
      K = std::max(K, rr.K[r]);
      S = std::max(S, rr.S[r]);
      M = std::max(M, rr.M[r]);
    }
    // the sub-stencil entries are staged in shared memory only where that costs the range no
    // resident blocks below the register bound; otherwise they are prefetched into L2 like the
    // rows (the pyramids and hexahedra of the hybrid meshes, which have eight sub-stencils)
    const ReconSmem<R> pb(K, S, M, true, true), pl(K, S, M, true, false);
    const int nb_l = std::min(kReconBlocksPerSM<R>, recon_blocks_per_sm(pl.bytes));
    if (pb.bytes <= kMaxBlockSmem && recon_blocks_per_sm(pb.bytes) >= nb_l) {
      launch_recon_ranges<R, true, true>(m, g, p, QA, poly, flag, r0, r1, K, S, M, pb.bytes, s);
    } else if (pl.bytes <= kMaxBlockSmem) {
      launch_recon_ranges<R, true, false>(m, g, p, QA, poly, flag, r0, r1, K, S, M, pl.bytes, s);
    } else {
      const ReconSmem<R> np(K, S, M, false, false);
      launch_recon_ranges<R, false, false>(m, g, p, QA, poly, flag, r0, r1, K, S, M, np.bytes, s);
    }
  };
  if (recon_merged(rr)) {  // the ranges are consecutive and cover all tiles
    launch(0, rr.n, st);
    return;
  }
  int used = 0;
  const bool fork = fj && fj->n > 0 && rr.n > 1;
  if (fork) cudaEventRecord(fj->fork, st);
  for (int r = 0; r < rr.n; ++r) {
    if (rr.t1[r] <= rr.t0[r]) continue;
    cudaStream_t s = st;
    if (fork && r > 0 && used < fj->n) {
      s = fj->aux[used];
      cudaStreamWaitEvent(s, fj->fork, 0);
    }
    launch(r, r + 1, s);
    if (s != st) {
      cudaEventRecord(fj->join[used], s);
      cudaStreamWaitEvent(st, fj->join[used], 0);
      ++used;
    }
  }
}
template <class R>
void launch_flux(const DevMesh& m, const GeoR<R>& g, const KParams<R>& p, const R* poly,
                 const R* QA, double dt, R* fface, int* flag, cudaStream_t st) {
  FluxParams<R> fp = flux_params(p);
  fp.erfc_tab = m.erfc_tab;
  fp.idt = (R)(1.0 / dt);
  // without a collision time the full form is the smooth one (its non-equilibrium terms carry
  // the weight tau = 0)
  auto run = [&](auto kern, int per_face, int nt) {
    kern<<<blocks_for(per_face * m.nf, nt), nt, 0, st>>>(
        m.nf, m.f_owner, m.f_nb, m.f_wall, g.fgp, poly, QA, p.gp_fallback, fp, wall_table<R>(m),
        (R)dt, fface, flag);
  };
  if constexpr (std::is_same<R, float>::value) {
    const bool pair = m.nf >= kPairFaces;
    if (fp.tau_model != 0 && fp.full)
      run(k_flux<R, true, false>, 4, 128);
    else if (pair)
      run(fp.tau_model == 0 ? k_flux_pair<true> : k_flux_pair<false>, 2, kPairThreads);
    else
      run(fp.tau_model == 0 ? k_flux<R, false, true> : k_flux<R, false, false>, 4, 128);
  } else {
    run(fp.tau_model == 0 ? k_flux<R, false, true>
                          : (fp.full ? k_flux<R, true, false> : k_flux<R, false, false>), 4, 128);
  }
}
template <class R>
void launch_gather(const DevMesh& m, const Geo64& g, const R* fface, double* L, double* Lt,
                   cudaStream_t st) {
  const int nt = cell_threads(m.nc);
  auto kern = nt < 256 ? k_gather<R, kFaceBatch> : k_gather<R, 1>;
  kern<<<blocks_for(m.nc, nt), nt, 0, st>>>(m.nc, m.cf_ptr, m.cf_idx, fface, g.ivol, m.perm, L,
                                            Lt);
}
template <class R>
void launch_stage(const DevMesh& m, const GeoR<R>& g, const R* fface, int stage, double dt,
                  void* L, void* Lt, R* QA, R* QsA, int* flag, cudaStream_t st, double* Q64,
                  const double* ivol64) {
  const int nt = cell_threads(m.nc);
  const bool small = nt < 256;
  const unsigned nb = blocks_for(m.nc, nt);
  // stage 1: c1 = dt/2, c2 = dt^2/8; stage 2: c1 = dt, c2 = dt^2/6
  const double c1 = stage == 1 ? 0.5 * dt : dt, c2 = stage == 1 ? dt * dt / 8.0 : dt * dt / 6.0;
  constexpr int kB = kFaceBatch;
  if constexpr (std::is_same<R, float>::value) {
    if (Q64) {  // FP64 update of the FP64 master state
      auto kern = stage == 1 ? (small ? k_stage_fd<false, kB> : k_stage_fd<false, 1>)
                             : (small ? k_stage_fd<true, kB> : k_stage_fd<true, 1>);
      kern<<<nb, nt, 0, st>>>(m.nc, m.cf_ptr, m.cf_idx, fface, ivol64, c1, c2,
                              static_cast<double*>(L), static_cast<double*>(Lt), Q64, QA, QsA,
                              flag);
      return;
    }
    auto kern = stage == 1 ? (small ? k_stage_f<false, kB> : k_stage_f<false, 1>)
                           : (small ? k_stage_f<true, kB> : k_stage_f<true, 1>);
    kern<<<nb, nt, 0, st>>>(m.nc, m.cf_ptr, m.cf_idx, fface,
                            reinterpret_cast<const ff*>(g.ivol), ff_from(c1), ff_from(c2),
                            static_cast<ff*>(L), static_cast<ff*>(Lt), QA, QsA, flag);
  } else {
    auto kern = stage == 1 ? (small ? k_stage_d<false, kB> : k_stage_d<false, 1>)
                           : (small ? k_stage_d<true, kB> : k_stage_d<true, 1>);
    kern<<<nb, nt, 0, st>>>(m.nc, m.cf_ptr, m.cf_idx, fface, g.ivol, c1, c2,
                            static_cast<double*>(L), static_cast<double*>(Lt), QA, QsA, flag);
  }
}
void launch_s2o4_stage(int64_t n, int stage, double dt, const double* Q, const double* L,
                       const double* Lt, const double* Lts, double* out, cudaStream_t st) {
  const double c1 = stage == 1 ? 0.5 * dt : dt, c2 = stage == 1 ? dt * dt / 8.0 : dt * dt / 6.0;
  k_s2o4_stage<<<blocks_for(n, 256), 256, 0, st>>>(n, stage, c1, c2, Q, L, Lt, Lts, out);
}
void launch_s2o4_stage_vjp(int64_t n, int stage, double dt, const double* g, double* gQ,
                           double* gL, double* gLt, double* gLts, cudaStream_t st) {
  const double c1 = stage == 1 ? 0.5 * dt : dt, c2 = stage == 1 ? dt * dt / 8.0 : dt * dt / 6.0;
  k_s2o4_stage_vjp<<<blocks_for(n, 256), 256, 0, st>>>(n, stage, c1, c2, g, gQ, gL, gLt, gLts);
}

constexpr int kJacobiThreads = 64;
template <class R>
void launch_jacobi_plan(const DevMesh& m, const R* fn, int32_t* jnb, R* jn, cudaStream_t st) {
  k_jacobi_plan<R><<<blocks_for(m.n_tiles * kTile, 256), 256, 0, st>>>(
      m.nc, m.n_tiles, m.cf_ptr, m.cf_idx, m.f_owner, m.f_nb, m.f_wall, fn, jnb, jn);
}
template <class R>
void launch_jacobi_init(const DevMesh& m, const R* fface, const JacobiBuf<R>& b, const double* vol,
                        double dt, const R* QA, const KParams<R>& kp, cudaStream_t st) {
  const FluxParams<R> fp = flux_params(kp);
  if constexpr (sizeof(R) == 8)
    k_jacobi_prim<R><<<blocks_for(m.nc, 64), 64, 0, st>>>(m.nc, QA, fp.gamma - R(1), b.prim);
  k_jacobi_init<R><<<blocks_for(m.nc, kJacobiThreads), kJacobiThreads, 0, st>>>(
      m.nc, m.cf_ptr, m.cf_idx, b.nb, b.n, fface, vol, dt, QA, b.prim, fp, wall_table<R>(m), b.Rv,
      b.D, b.hrs, b.dQ[0]);
}
template <class R>
void launch_jacobi_sweep(const DevMesh& m, const JacobiBuf<R>& b, const R* QA, int it, int last,
                         R* QAout, const KParams<R>& kp, int* flag, cudaStream_t st) {
  auto kern = last ? k_jacobi_sweep<R, true> : k_jacobi_sweep<R, false>;
  kern<<<blocks_for(m.nc, kJacobiThreads), kJacobiThreads, 0, st>>>(m.nc, b.nb, b.n, QA, b.prim, b.Rv, b.D,
                                              b.hrs, b.dQ[(it - 1) & 1], b.dQ[it & 1], QAout,
                                              flux_params(kp), wall_table<R>(m), flag);
}
void launch_unpack(int64_t nc, const float* QA, double* Q, cudaStream_t st) {
  k_unpack<<<blocks_for(nc, 256), 256, 0, st>>>(nc, QA, Q);
}
template <class R>
void launch_unpack_out(int64_t nc, const int32_t* perm, const R* QA, double* dst,
                       cudaStream_t st) {
  k_unpack_out<R><<<blocks_for(nc, 256), 256, 0, st>>>(nc, perm, QA, dst);
}
template <class R>
void launch_permute_in(int64_t nc, const int32_t* perm, const double* src, double* dst, R* gq,
                       int* flag, cudaStream_t st) {
  k_permute_in<R><<<blocks_for(nc, 256), 256, 0, st>>>(nc, perm, src, dst, gq, flag);
}
void launch_permute_out(int64_t nc, const int32_t* perm, const double* src, double* dst,
                        cudaStream_t st) {
  k_permute_out<<<blocks_for(nc, 256), 256, 0, st>>>(nc, perm, src, dst);
}
constexpr int64_t kDtLargeCells = 152 * 4 * kDtThreads;  // from here on four cells per thread
int dt_blocks(int64_t nc) {
  const int64_t chunk = (nc >= kDtLargeCells ? 4 : 1) * kDtThreads;
  const int64_t b = (nc + chunk - 1) / chunk;
  return (int)(b < kDtMaxBlocks ? b : kDtMaxBlocks);
}
template <class R>
void launch_dt(int64_t nc, const R* QA, const double* Q64, const double* hdt, double gamma,
               double mu, int power, double T_ref, double mu_pow, double* partial, int nblocks,
               double* out, int* flag, cudaStream_t st) {
  auto kern = nc >= kDtLargeCells ? k_dt_partial<R, 4> : k_dt_partial<R, 1>;
  const DtParams P{gamma, mu, T_ref, mu_pow, power, (float)(gamma - 1.0), dt_cut(power, mu_pow)};
  kern<<<nblocks, kDtThreads, 0, st>>>(nc, QA, Q64, hdt, P, partial, flag);
  k_dt_final<<<1, 256, 0, st>>>(partial, nblocks, out);
}

template void launch_dt<float>(int64_t, const float*, const double*, const double*, double, double,
                               int, double, double, double*, int, double*, int*, cudaStream_t);
template void launch_dt<double>(int64_t, const double*, const double*, const double*, double,
                                double, int, double, double, double*, int, double*, int*,
                                cudaStream_t);
template void launch_unpack_out<float>(int64_t, const int32_t*, const float*, double*,
                                       cudaStream_t);
template void launch_unpack_out<double>(int64_t, const int32_t*, const double*, double*,
                                        cudaStream_t);
template void launch_recon<double>(const DevMesh&, const GeoR<double>&, const KParams<double>&,
                                   const double*, double*, int*, cudaStream_t, const ForkJoin*);
template void launch_permute_in<double>(int64_t, const int32_t*, const double*, double*, double*,
                                        int*, cudaStream_t);
template void launch_permute_in<float>(int64_t, const int32_t*, const double*, double*, float*,
                                       int*, cudaStream_t);
template void launch_recon<float>(const DevMesh&, const GeoR<float>&, const KParams<float>&,
                                  const float*, float*, int*, cudaStream_t, const ForkJoin*);
template void launch_flux<double>(const DevMesh&, const GeoR<double>&, const KParams<double>&,
                                  const double*, const double*, double, double*, int*,
                                  cudaStream_t);
template void launch_flux<float>(const DevMesh&, const GeoR<float>&, const KParams<float>&,
                                 const float*, const float*, double, float*, int*, cudaStream_t);
template void launch_gather<double>(const DevMesh&, const Geo64&, const double*, double*, double*,
                                    cudaStream_t);
template void launch_gather<float>(const DevMesh&, const Geo64&, const float*, double*, double*,
                                   cudaStream_t);
template void launch_stage<double>(const DevMesh&, const GeoR<double>&, const double*, int, double,
                                   void*, void*, double*, double*, int*, cudaStream_t, double*,
                                   const double*);
template void launch_stage<float>(const DevMesh&, const GeoR<float>&, const float*, int, double,
                                  void*, void*, float*, float*, int*, cudaStream_t, double*,
                                  const double*);
template void launch_jacobi_plan<double>(const DevMesh&, const double*, int32_t*, double*,
                                         cudaStream_t);
template void launch_jacobi_plan<float>(const DevMesh&, const float*, int32_t*, float*,
                                        cudaStream_t);
template void launch_jacobi_init<double>(const DevMesh&, const double*, const JacobiBuf<double>&,
                                         const double*, double, const double*,
                                         const KParams<double>&, cudaStream_t);
template void launch_jacobi_init<float>(const DevMesh&, const float*, const JacobiBuf<float>&,
                                        const double*, double, const float*,
                                        const KParams<float>&, cudaStream_t);
template void launch_jacobi_sweep<double>(const DevMesh&, const JacobiBuf<double>&, const double*,
                                          int, int, double*, const KParams<double>&, int*,
                                          cudaStream_t);
template void launch_jacobi_sweep<float>(const DevMesh&, const JacobiBuf<float>&, const float*,
                                         int, int, float*, const KParams<float>&, int*,
                                         cudaStream_t);

}  // namespace gks
