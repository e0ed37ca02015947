// VGICP factor linearization kernels (arXiv 2202.00242 Sec. III-A, Eqs. 2-3 and
// the Hessian factor built from their derivatives at every optimizer iteration).
//
// One persistent launch processes a list of work items (pair, [begin, end)) over
// the source clouds.  Per source point k of pair (map, source, T = (R, t)):
//   q    = R mu_k + t                                   (float32)
//   key  = floor(q / r) exactly as in binary64 (float32 fast path, binary64
//          recomputation for the rare points whose float32 q lies within its
//          error bound of a voxel face)
//   vid  = hash lookup (open addressing, bounded linear probe)
//   in the SOURCE frame (J = R K with K = [[mu]x, -I], so J^T W J = K^T W' K):
//   d'   = R^T (mu'_v - q)
//   M'   = R^T C'_v R + C_k = B B^T + C_k with B = R^T L (C'_v = L L^T, the
//          Cholesky factor kept in the lookup slot), W' = M'^-1 (= R^T W R,
//          symmetric adjugate / det)
//   u    = W' d'
//   err += d'^T u
//   b   += [ u x mu ; -u ]
//   H   += [[ [mu]x^T W' [mu]x , [mu]x W' ], [ ., W' ]]
// The 28 unique terms and the inlier count are accumulated per thread in
// float32 over a work item (up to 16K points of one pair), reduced across the
// warp in float32, across warps in binary64, and written as one binary64
// partial per work item; a second kernel sums each pair's partials in item
// order.  The result is deterministic.
//
// Work items are claimed dynamically from an atomic counter, so uneven items
// (ragged tails of the clouds, pairs with few inliers) do not leave CTAs idle.
//
// Kernels (the autotuner picks among the 1-neighbour ones per factor set):
//   1  per-point: one point per thread, item constants in uniform registers so that
//      4 CTAs of 256 threads fit per SM; the default and usually the fastest;
//   2  staged: a producer warp streams tiles of points and covariances into
//      shared memory with bulk asynchronous copies (cp.async.bulk + mbarrier);
//      consumer warps look up, compact the hits and evaluate from shared memory;
//   3  compacting: the per-point lookup, with the hits queued per warp in shared
//      memory and evaluated 32 at a time (no idle lanes on misses);
//   27 neighbours: the per-point kernel with the 27 lookups in a loop, or, for large
//      batches, the neighbours taken from occupancy blocks (namespace blocks).
// Chosen by size, with the same results bit for bit:
//   few items: a cluster of 8 CTAs per item (namespace split);
//   a small single factor: items and their sum in one launch (namespace factor).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "vgicp_device.cuh"
#include "vgicp_internal.h"

namespace vgicp {
namespace {

constexpr int kSimpleThreads = 256;

struct Pose32 {
  float R[9];
  float t[3];
  float tmax;
};

// floor(q_a / r) with q = R64 mu + t64 in binary64 (the rare near-face path).
__device__ __forceinline__ int axis_key_f64(const PairDesc* pd, const MapDesc& md, int a, float x,
                                         float y, float z) {
  double s = __dmul_rn(pd->R64[3 * a + 0], (double)x);
  s = __dadd_rn(s, __dmul_rn(pd->R64[3 * a + 1], (double)y));
  s = __dadd_rn(s, __dmul_rn(pd->R64[3 * a + 2], (double)z));
  s = __dadd_rn(s, pd->t64[a]);
  double k = floor(__ddiv_rn(s, md.r));
  k = fmin(fmax(k, -2147483648.0), 2147483647.0);
  return (int)k;
}

// Key of the transformed source point, exact w.r.t. the binary64 definition
// floor((R64 mu + t64) / r).  Float32 bound: |q32 - q64| <= 2^-22 S with
// S = |x| + |y| + |z| + max|t| (rounding of R and t to float32 and three FMA
// roundings), and y = q32 * float(1/r) adds 2^-23 |y|; the margin
// 2^-21 S / r + 2^-23 covers both and the rounding of the fractional part.
__device__ __forceinline__ void source_key(const Pose32& P, const PairDesc* pd, const MapDesc& md,
                                           float x, float y, float z, float qx, float qy,
                                           float qz, int& kx, int& ky, int& kz) {
  const float S = fabsf(x) + fabsf(y) + fabsf(z) + P.tmax;
  const float m = fmaf(S, md.margin_scale, 1.1920928955078125e-7f);
  const float yx = qx * md.inv_r, yy = qy * md.inv_r, yz = qz * md.inv_r;
  const float fx = floorf(yx), fy = floorf(yy), fz = floorf(yz);
  const float rx = yx - fx, ry = yy - fy, rz = yz - fz;
  const bool ax = (rx < m) | (rx > 1.0f - m);
  const bool ay = (ry < m) | (ry > 1.0f - m);
  const bool az = (rz < m) | (rz > 1.0f - m);
  kx = clamp_to_int(fx);
  ky = clamp_to_int(fy);
  kz = clamp_to_int(fz);
  if (ax | ay | az) {
    // binary64, evaluated as ((R0 x + R1 y) + R2 z) + t without contraction
    if (ax) kx = axis_key_f64(pd, md, 0, x, y, z);
    if (ay) ky = axis_key_f64(pd, md, 1, x, y, z);
    if (az) kz = axis_key_f64(pd, md, 2, x, y, z);
  }
}

__device__ __forceinline__ void ld_v8(const void* p, uint64_t policy, uint32_t (&w)[8]) {
  asm("ld.global.nc.L2::cache_hint.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8], %9;"
      : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]),
        "=r"(w[7])
      : "l"(p), "l"(policy));
}
__device__ __forceinline__ unsigned long long slot_key(const uint32_t (&a)[8]) {
  return (unsigned long long)a[0] | ((unsigned long long)a[1] << 32);
}
__device__ __forceinline__ void ld_v4(const void* p, uint64_t policy, uint32_t (&w)[4]) {
  asm("ld.global.nc.L2::cache_hint.v4.b32 {%0, %1, %2, %3}, [%4], %5;"
      : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
      : "l"(p), "l"(policy));
}
// One probe of a lookup slot: two independent loads (a: key, spill, mu', l00, l10; b:
// l20, l11, l21, l22).
__device__ __forceinline__ void ld_slot(const VSlot* t, uint64_t policy, uint32_t (&a)[8],
                                        uint32_t (&b)[4]) {
  ld_v8(t, policy, a);
  ld_v4(reinterpret_cast<const char*>(t) + 32, policy, b);
}
// The slot's Gaussian: r0 = (mu', -), r1 = (l00, l10, l20, l11), r2 = (l21, l22, -, -).
__device__ __forceinline__ void slot_gaussian(const uint32_t (&a)[8], const uint32_t (&b)[4],
                                              float4& r0, float4& r1, float4& r2) {
  r0 = make_float4(__uint_as_float(a[kSlotMu]), __uint_as_float(a[kSlotMu + 1]),
                   __uint_as_float(a[kSlotMu + 2]), 0.f);
  r1 = make_float4(__uint_as_float(a[kSlotL]), __uint_as_float(a[kSlotL + 1]),
                   __uint_as_float(b[0]), __uint_as_float(b[1]));
  r2 = make_float4(__uint_as_float(b[2]), __uint_as_float(b[3]), 0.f, 0.f);
}
__device__ __forceinline__ uint64_t policy_evict_last_l() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// Lookup of key (kx, ky, kz) in a map's inline table: whether the voxel exists; on a
// hit also its slot and Gaussian.
__device__ __forceinline__ bool lookup(const MapDesc& md, uint32_t mask, int kx, int ky, int kz,
                                       uint64_t pol, uint32_t& h, float4& r0, float4& r1,
                                       float4& r2) {
  if (!key_in_range(kx) || !key_in_range(ky) || !key_in_range(kz)) return false;
  const unsigned long long key = pack_key(kx, ky, kz);
  h = hash_key(kx, ky, kz) & mask;
  for (int p = 0; p < md.max_probe; ++p) {
    uint32_t a[8], b[4];
    ld_slot(md.vslots + h, pol, a, b);
    const unsigned long long k = slot_key(a);
    if (k == key) {
      slot_gaussian(a, b, r0, r1, r2);
      return true;
    }
    if (k == kEmptyKey || (p == 0 && a[kSlotSpill] == 0u)) return false;  // empty, or nothing spilled
    h = (h + 1) & mask;
  }
  return false;
}

// Accumulator layout (float):
//   0..5   H_ww (00 01 02 11 12 22)      6..14 H_wv (row-major, w rows, v cols)
//   15..20 H_vv (00 01 02 11 12 22)      21..23 b_w   24..26 b_v   27 err
//   28     inlier count
// 1 / x to about 1 ulp (rcp.approx: one instruction; H, b and err are held to
// 1e-4 relative, many orders above this).  Deterministic.
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// M' = R^T C' R + C (upper triangle m00 m01 m02 m11 m12 m22) from the voxel
// covariance's Cholesky factor L (C' = L L^T, stored in the lookup slot as
// l00 l10 l20 l11 l21 l22): with B = R^T L, R^T C' R = B B^T (36 operations
// instead of 45 for R^T (C' R)).
__device__ __forceinline__ void fused_cov(const float* R, const float4 r1, const float4 r2,
                                          const float* c, float& m00, float& m01, float& m02,
                                          float& m11, float& m12, float& m22) {
  const float l00 = r1.x, l10 = r1.y, l20 = r1.z, l11 = r1.w, l21 = r2.x, l22 = r2.y;
  // B_i0 = sum_k R_ki L_k0, B_i1 = R_1i l11 + R_2i l21, B_i2 = R_2i l22
  const float b00 = fmaf(R[0], l00, fmaf(R[3], l10, R[6] * l20));
  const float b10 = fmaf(R[1], l00, fmaf(R[4], l10, R[7] * l20));
  const float b20 = fmaf(R[2], l00, fmaf(R[5], l10, R[8] * l20));
  const float b01 = fmaf(R[3], l11, R[6] * l21);
  const float b11 = fmaf(R[4], l11, R[7] * l21);
  const float b21 = fmaf(R[5], l11, R[8] * l21);
  const float b02 = R[6] * l22, b12 = R[7] * l22, b22 = R[8] * l22;
  m00 = fmaf(b00, b00, fmaf(b01, b01, fmaf(b02, b02, c[0])));
  m01 = fmaf(b00, b10, fmaf(b01, b11, fmaf(b02, b12, c[1])));
  m02 = fmaf(b00, b20, fmaf(b01, b21, fmaf(b02, b22, c[2])));
  m11 = fmaf(b10, b10, fmaf(b11, b11, fmaf(b12, b12, c[3])));
  m12 = fmaf(b10, b20, fmaf(b11, b21, fmaf(b12, b22, c[4])));
  m22 = fmaf(b20, b20, fmaf(b21, b21, fmaf(b22, b22, c[5])));
}

__device__ __forceinline__ void add_term_t(float* acc, const float* R, float x, float y, float z,
                                           const float* c, float tx, float ty, float tz,
                                           const float4 r1, const float4 r2) {
  // residual (tx, ty, tz) = mu' - q in the target frame, rotated into the source frame
  const float d0 = fmaf(R[0], tx, fmaf(R[3], ty, R[6] * tz));
  const float d1 = fmaf(R[1], tx, fmaf(R[4], ty, R[7] * tz));
  const float d2 = fmaf(R[2], tx, fmaf(R[5], ty, R[8] * tz));
  // M' = R^T C' R + C_k (upper triangle)
  float m00, m01, m02, m11, m12, m22;
  fused_cov(R, r1, r2, c, m00, m01, m02, m11, m12, m22);
  // W' = adj(M') / det(M')
  const float i00 = fmaf(m11, m22, -m12 * m12);
  const float i01 = fmaf(m02, m12, -m01 * m22);
  const float i02 = fmaf(m01, m12, -m02 * m11);
  const float i11 = fmaf(m00, m22, -m02 * m02);
  const float i12 = fmaf(m01, m02, -m00 * m12);
  const float i22 = fmaf(m00, m11, -m01 * m01);
  const float det = fmaf(m00, i00, fmaf(m01, i01, m02 * i02));
  const float s = rcp_approx(det);
  // (rounded before they are added below, so that every kernel forms the same sums)
  const float w00 = __fmul_rn(i00, s), w01 = __fmul_rn(i01, s), w02 = __fmul_rn(i02, s);
  const float w11 = __fmul_rn(i11, s), w12 = __fmul_rn(i12, s), w22 = __fmul_rn(i22, s);
  // u = W' d'
  const float u0 = fmaf(w00, d0, fmaf(w01, d1, w02 * d2));
  const float u1 = fmaf(w01, d0, fmaf(w11, d1, w12 * d2));
  const float u2 = fmaf(w02, d0, fmaf(w12, d1, w22 * d2));
  // err
  acc[27] = fmaf(d0, u0, fmaf(d1, u1, fmaf(d2, u2, acc[27])));
  // b = [u x mu ; -u]
  acc[21] = fmaf(u1, z, fmaf(-u2, y, acc[21]));
  acc[22] = fmaf(u2, x, fmaf(-u0, z, acc[22]));
  acc[23] = fmaf(u0, y, fmaf(-u1, x, acc[23]));
  acc[24] -= u0;
  acc[25] -= u1;
  acc[26] -= u2;
  // H_vv = W'
  acc[15] += w00; acc[16] += w01; acc[17] += w02;
  acc[18] += w11; acc[19] += w12; acc[20] += w22;
  // P = [mu]x W'  (rows: (-z W1 + y W2), (z W0 - x W2), (-y W0 + x W1))
  const float p00 = fmaf(y, w02, -z * w01), p01 = fmaf(y, w12, -z * w11), p02 = fmaf(y, w22, -z * w12);
  const float p10 = fmaf(z, w00, -x * w02), p11 = fmaf(z, w01, -x * w12), p12 = fmaf(z, w02, -x * w22);
  const float p20 = fmaf(x, w01, -y * w00), p21 = fmaf(x, w11, -y * w01), p22 = fmaf(x, w12, -y * w02);
  acc[6] += p00; acc[7] += p01; acc[8] += p02;
  acc[9] += p10; acc[10] += p11; acc[11] += p12;
  acc[12] += p20; acc[13] += p21; acc[14] += p22;
  // H_ww = -P [mu]x
  acc[0] = fmaf(p02, y, fmaf(-p01, z, acc[0]));
  acc[1] = fmaf(p00, z, fmaf(-p02, x, acc[1]));
  acc[2] = fmaf(p01, x, fmaf(-p00, y, acc[2]));
  acc[3] = fmaf(p10, z, fmaf(-p12, x, acc[3]));
  acc[4] = fmaf(p11, x, fmaf(-p10, y, acc[4]));
  acc[5] = fmaf(p21, x, fmaf(-p20, y, acc[5]));
}

__device__ __forceinline__ void add_term(float* acc, const Pose32& P, float x, float y, float z,
                                         const float* c, float qx, float qy, float qz,
                                         const float4 r0, const float4 r1, const float4 r2) {
  add_term_t(acc, P.R, x, y, z, c, r0.x - qx, r0.y - qy, r0.z - qz, r1, r2);
  acc[28] += 1.0f;
}


// Launch-shape constants (compile-time; overridable for tuning builds).
#ifndef VGICP_NCW
#define VGICP_NCW 4
#endif
#ifndef VGICP_PTS_PER_LANE
#define VGICP_PTS_PER_LANE 2
#endif
#ifndef VGICP_STAGES
#define VGICP_STAGES 4
#endif
#ifndef VGICP_MIN_BLOCKS
#define VGICP_MIN_BLOCKS 3
#endif

// ---------------------------------------------------------------------------
// PTX helpers: mbarrier and bulk asynchronous copy (global -> shared)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
               : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
// try_wait with a suspend-time hint: the thread sleeps until the phase completes
// (or the hint expires) instead of spinning on the issue slots.
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity), "r"(20000u)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait: gives up after limit_ns (2 s by default: a bug, never a normal
// state; a test launch may set a shorter limit).
constexpr uint64_t kWaitLimitNs = 2000000000ull;
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity,
                                          uint64_t limit_ns = kWaitLimitNs) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  while (!mbar_try_wait(bar, parity))
    if (global_ns() - t0 > limit_ns) return false;
  return true;
}
// L2 policies: the source stream is read once per factor (evict first), while
// the lookup tables are re-read by every source point of the factors that
// target them (evict last).
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1], %2, [%3], %4;" ::"r"(smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar)), "l"(policy)
      : "memory");
}
// 4-byte asynchronous copy global -> shared, completion tracked by an mbarrier
// through cp_async_arrive_noinc.
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_arrive_noinc(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ void consumer_bar() {
  asm volatile("bar.sync 1, %0;" ::"n"(VGICP_NCW * 32) : "memory");
}

// ---------------------------------------------------------------------------
// 1-neighbour kernel with shared-memory staging
// ---------------------------------------------------------------------------
namespace tma {
constexpr int kNCW = VGICP_NCW;               // consumer warps
constexpr int kThreads = (kNCW + 1) * 32;     // + one producer warp
constexpr int kPtsPerLane = VGICP_PTS_PER_LANE;
constexpr int kWarpPts = 32 * kPtsPerLane;    // 64 points per consumer warp
constexpr int kTile = kNCW * kWarpPts;        // 256 points per tile
constexpr int kStages = VGICP_STAGES;
constexpr int kXyzBytes = kTile * 12 + 32;    // + room for a 16-B alignment shift
constexpr int kCovBytes = kTile * 24 + 32;
constexpr int kFirst = 1, kLast = 2;

struct TileDesc {
  int32_t pair, begin, n, item, flags, xyz_off, cov_off, pad;
};

struct __align__(16) Smem {
  float4 hits[kNCW][kWarpPts * 3];            // staged voxel records of hits
  unsigned char xyz[kStages][kXyzBytes];
  unsigned char cov[kStages][kCovBytes];
  TileDesc desc[kStages];
  uint64_t full[kStages];
  uint64_t empty[kStages];
  float red[kNCW][32];
};
static_assert(kXyzBytes % 16 == 0 && kCovBytes % 16 == 0, "bulk-copy alignment");

// Copy the float range [gs, ge) of global memory into shared memory at
// dst + (gs - floor16(gs)): the 16-B aligned interior with one bulk copy
// (issue_bulk), the ragged head and tail (< 16 B each) with 4-byte cp.async
// (!issue_bulk).  Returns the bulk bytes.
__device__ __forceinline__ uint32_t stage_range(unsigned char* dst, uintptr_t gs, uintptr_t ge,
                                                uint64_t* bar, bool issue_bulk, uint64_t policy) {
  const uintptr_t g0 = gs & ~(uintptr_t)15;
  const uintptr_t a = (gs + 15) & ~(uintptr_t)15;
  const uintptr_t b = ge & ~(uintptr_t)15;
  uint32_t bulk = 0;
  uintptr_t h1 = ge, t0 = ge;
  if (b > a) {
    bulk = (uint32_t)(b - a);
    h1 = a;
    t0 = b;
    if (issue_bulk) bulk_g2s(dst + (a - g0), reinterpret_cast<const void*>(a), bulk, bar, policy);
  }
  if (!issue_bulk) {
    for (uintptr_t p = gs; p < h1; p += 4)
      cp_async4(dst + (p - g0), reinterpret_cast<const void*>(p));
    for (uintptr_t p = t0; p < ge; p += 4)
      cp_async4(dst + (p - g0), reinterpret_cast<const void*>(p));
  }
  return bulk;
}

__device__ __forceinline__ void item_bounds(const LinLaunch& L, int it, int& pair, int& b,
                                            int& e) {
  if (L.items) {
    const WorkItem w = L.items[it];
    pair = w.pair;
    b = w.begin;
    e = w.end;
  } else {
    pair = 0;
    b = it * L.item_size;
    e = (int)min((int64_t)b + L.item_size, L.single_src.n);
  }
}

// Warp reduce-scatter of 32 values: afterwards lane l holds the warp total of v[l]
// (31 shuffles instead of 5 per value).
template <int W>
__device__ __forceinline__ void rs_step(float* v, int lane) {
  const bool up = (lane & W) != 0;
#pragma unroll
  for (int j = 0; j < W; ++j) {
    const float send = up ? v[j] : v[j + W];
    const float keep = up ? v[j + W] : v[j];
    v[j] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, W);
  }
}

__global__ void __launch_bounds__(kThreads, VGICP_MIN_BLOCKS) linearize_tma_kernel(const __grid_constant__ LinLaunch L) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem& S = *reinterpret_cast<Smem*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&S.full[s], 2);  // producer arrive + cp.async completion arrive
      mbar_init(&S.empty[s], kNCW);
    }
    mbar_fence_init();
  }
  __syncthreads();

  const uint64_t wait_ns = L.wait_limit_ns > 0 ? (uint64_t)L.wait_limit_ns : kWaitLimitNs;
  if (warp == kNCW) {
    // ---------------- producer ----------------
    if (lane != 0) return;
    const uint64_t stream_pol = policy_evict_first();
    uint32_t u = 0;  // tiles issued
    bool ok = true, withheld = false;
    for (int it = blockIdx.x; it < L.n_items && ok && !withheld; it += gridDim.x) {
      int pair, b, e;
      item_bounds(L, it, pair, b, e);
      const PairDesc* pd = L.pairs ? L.pairs + pair : &L.single;
      const SrcDesc sd = L.srcs ? L.srcs[pd->src] : L.single_src;
      for (int t0 = b; t0 < e; t0 += kTile) {
        const int s = u % kStages;
        if (u >= kStages && !mbar_wait(&S.empty[s], ((u / kStages) - 1) & 1, wait_ns)) {
          ok = false;
          break;
        }
        if (L.test_withhold_tile > 0 && u + 1 == (uint32_t)L.test_withhold_tile) {
          // test launch: this tile is never issued (no copy, no arrival), so the
          // consumers' bounded wait for it runs out
          withheld = true;
          break;
        }
        const int n = min(kTile, e - t0);
        const uintptr_t xs = reinterpret_cast<uintptr_t>(sd.pts + 3 * (int64_t)t0);
        const uintptr_t cs = reinterpret_cast<uintptr_t>(sd.covs + 6 * (int64_t)t0);
        // head/tail cp.async and the descriptor, then the two arrivals, then bulk
        const uintptr_t xe = xs + 12 * (uintptr_t)n, ce = cs + 24 * (uintptr_t)n;
        const uint32_t tx = stage_range(S.xyz[s], xs, xe, &S.full[s], false, stream_pol) +
                            stage_range(S.cov[s], cs, ce, &S.full[s], false, stream_pol);
        TileDesc d;
        d.pair = pair;
        d.begin = t0;
        d.n = n;
        d.item = it;
        d.flags = (t0 == b ? kFirst : 0) | (t0 + kTile >= e ? kLast : 0);
        d.xyz_off = (int)(xs & 15);
        d.cov_off = (int)(cs & 15);
        d.pad = 0;
        S.desc[s] = d;
        cp_async_arrive_noinc(&S.full[s]);
        mbar_arrive_expect_tx(&S.full[s], tx);
        stage_range(S.xyz[s], xs, xe, &S.full[s], true, stream_pol);
        stage_range(S.cov[s], cs, ce, &S.full[s], true, stream_pol);
        ++u;
      }
    }
    if (ok && !withheld) {
      const int s = u % kStages;
      if (u >= kStages && !mbar_wait(&S.empty[s], ((u / kStages) - 1) & 1, wait_ns)) ok = false;
      if (ok) {
        S.desc[s].n = -1;
        mbar_arrive(&S.full[s]);
        mbar_arrive(&S.full[s]);
        ++u;
      }
    }
    if (!ok) atomicExch(L.status, 1);
    if (!ok || withheld) {
      // let copies already in flight land before the block exits
      for (uint32_t v = (u > kStages ? u - kStages : 0); v < u; ++v)
        mbar_wait(&S.full[v % kStages], (v / kStages) & 1, wait_ns);
    }
    return;
  }

  // ---------------- consumers ----------------
  float acc[32];
#pragma unroll
  for (int k = 0; k < 32; ++k) acc[k] = 0.0f;
  Pose32 P;
  MapDesc md;
  const PairDesc* pd = nullptr;
  uint32_t vbase = 0, mask = 0;
  float4* H = S.hits[warp];
  const uint32_t lt_mask = (1u << lane) - 1u;
  const uint64_t map_pol = policy_evict_last();

  for (uint32_t u = 0;; ++u) {
    const int s = u % kStages;
    if (!mbar_wait(&S.full[s], (u / kStages) & 1, wait_ns)) {
      atomicExch(L.status, 1);
      break;
    }
    const TileDesc d = S.desc[s];
    if (d.n < 0) break;
    if (d.flags & kFirst) {
      pd = L.pairs ? L.pairs + d.pair : &L.single;
#pragma unroll
      for (int k = 0; k < 9; ++k) P.R[k] = pd->R[k];
      P.t[0] = pd->t[0];
      P.t[1] = pd->t[1];
      P.t[2] = pd->t[2];
      P.tmax = pd->tmax;
      md = L.maps ? L.maps[pd->map] : L.single_map;
      mask = *md.vmask;
      if (L.corr_out) vbase = *md.vbase;
    }
    const float* X = reinterpret_cast<const float*>(S.xyz[s] + d.xyz_off);
    const float* C = reinterpret_cast<const float*>(S.cov[s] + d.cov_off);

    // ---- lookup: key, first probe (a 256-bit and a 128-bit load) of every point, resolve ----
    int idx[kPtsPerLane];
    int kx[kPtsPerLane], ky[kPtsPerLane], kz[kPtsPerLane];
    bool live[kPtsPerLane];
    unsigned long long key[kPtsPerLane];
    uint32_t h[kPtsPerLane];
    uint32_t sa[kPtsPerLane][8], sb[kPtsPerLane][4];
#pragma unroll
    for (int k = 0; k < kPtsPerLane; ++k) {
      idx[k] = warp * kWarpPts + k * 32 + lane;
      live[k] = idx[k] < d.n;
      kx[k] = ky[k] = kz[k] = kKeyMin - 1;
      if (live[k]) {
        const float x = X[3 * idx[k]], y = X[3 * idx[k] + 1], z = X[3 * idx[k] + 2];
        const float qx = fmaf(P.R[0], x, fmaf(P.R[1], y, fmaf(P.R[2], z, P.t[0])));
        const float qy = fmaf(P.R[3], x, fmaf(P.R[4], y, fmaf(P.R[5], z, P.t[1])));
        const float qz = fmaf(P.R[6], x, fmaf(P.R[7], y, fmaf(P.R[8], z, P.t[2])));
        source_key(P, pd, md, x, y, z, qx, qy, qz, kx[k], ky[k], kz[k]);
        live[k] = key_in_range(kx[k]) && key_in_range(ky[k]) && key_in_range(kz[k]);
      }
      key[k] = live[k] ? pack_key(kx[k], ky[k], kz[k]) : kEmptyKey;
      h[k] = hash_key(kx[k], ky[k], kz[k]) & mask;
      if (live[k]) {
        ld_slot(md.vslots + h[k], map_pol, sa[k], sb[k]);
      } else {
        sa[k][0] = sa[k][1] = 0xFFFFFFFFu;
      }
    }
    int vid[kPtsPerLane];
    float4 r0[kPtsPerLane], r1[kPtsPerLane], r2[kPtsPerLane];
#pragma unroll
    for (int k = 0; k < kPtsPerLane; ++k) {
      vid[k] = -1;
      if (live[k]) {
        unsigned long long t = slot_key(sa[k]);
        uint32_t hh = h[k];
        for (int p = 1; t != key[k] && t != kEmptyKey && (p > 1 || sa[k][kSlotSpill] != 0u) &&
                        p < md.max_probe;
             ++p) {
          hh = (hh + 1) & mask;
          ld_slot(md.vslots + hh, map_pol, sa[k], sb[k]);
          t = slot_key(sa[k]);
        }
        if (t == key[k]) {
          vid[k] = L.corr_out ? (int)__ldg(&md.vslots[hh].vid) : 0;
          slot_gaussian(sa[k], sb[k], r0[k], r1[k], r2[k]);
        }
      }
      if (idx[k] < d.n && (L.corr_out || L.qkey_out)) {
        const int64_t p = (int64_t)d.begin + idx[k];
        if (L.corr_out) L.corr_out[p] = vid[k] < 0 ? -1 : (int)((uint32_t)vid[k] - vbase);
        if (L.qkey_out) {
          L.qkey_out[3 * p + 0] = kx[k];
          L.qkey_out[3 * p + 1] = ky[k];
          L.qkey_out[3 * p + 2] = kz[k];
        }
      }
    }
    // ---- stage the records of the hits, compacted per warp ----
    int nh = 0;
#pragma unroll
    for (int k = 0; k < kPtsPerLane; ++k) {
      const uint32_t m = __ballot_sync(0xFFFFFFFFu, vid[k] >= 0);
      if (vid[k] >= 0) {
        const int pos = nh + __popc(m & lt_mask);
        H[3 * pos + 0] = make_float4(r0[k].x, r0[k].y, r0[k].z, __int_as_float(idx[k]));
        H[3 * pos + 1] = r1[k];
        H[3 * pos + 2] = r2[k];
      }
      nh += __popc(m);
    }
    __syncwarp();
    // ---- terms of the hits, from shared memory ----
    for (int j = lane; j < nh; j += 32) {
      const float4 e0 = H[3 * j], e1 = H[3 * j + 1], e2 = H[3 * j + 2];
      const int i = __float_as_int(e0.w);
      const float x = X[3 * i], y = X[3 * i + 1], z = X[3 * i + 2];
      const float2* cv = reinterpret_cast<const float2*>(C + 6 * i);
      const float2 c01 = cv[0], c23 = cv[1], c45 = cv[2];
      const float c[6] = {c01.x, c01.y, c23.x, c23.y, c45.x, c45.y};
      const float qx = fmaf(P.R[0], x, fmaf(P.R[1], y, fmaf(P.R[2], z, P.t[0])));
      const float qy = fmaf(P.R[3], x, fmaf(P.R[4], y, fmaf(P.R[5], z, P.t[1])));
      const float qz = fmaf(P.R[6], x, fmaf(P.R[7], y, fmaf(P.R[8], z, P.t[2])));
      add_term(acc, P, x, y, z, c, qx, qy, qz, e0, e1, e2);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&S.empty[s]);

    if (d.flags & kLast) {
      rs_step<16>(acc, lane);
      rs_step<8>(acc, lane);
      rs_step<4>(acc, lane);
      rs_step<2>(acc, lane);
      rs_step<1>(acc, lane);
      S.red[warp][lane] = acc[0];
      consumer_bar();
      if (warp == 0 && lane < kAcc) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < kNCW; ++w) t += (double)S.red[w][lane];
        L.partials[(int64_t)d.item * kPartialStride + lane] = t;
      }
      consumer_bar();
#pragma unroll
      for (int k = 0; k < 32; ++k) acc[k] = 0.0f;
    }
  }
}

}  // namespace tma

// ---------------------------------------------------------------------------
// One point per thread (1 or 27 neighbours); the lookups and records come from
// global memory through L1.
// ---------------------------------------------------------------------------
// Cost and gradient of one term, for the differentiable interface:
//   MODE 1: err only;  MODE 2: + g = 2 J^T W d (W held, the Gauss-Newton gradient);
//   MODE 3: + the change of W with the rotation: for omega_i the exact derivative
//           adds -u^T dM/domega_i u = 2 (u' x C_k u')_i, u' = W' d' (source frame).
// Accumulators: 0..5 gradient, 6 err, 28 inlier count.
template <int MODE>
__device__ __forceinline__ void eval_term(float* acc, const Pose32& P, float x, float y, float z,
                                          const float* c, float qx, float qy, float qz,
                                          const float4 r0, const float4 r1, const float4 r2) {
  const float* R = P.R;
  const float tx = r0.x - qx, ty = r0.y - qy, tz = r0.z - qz;
  const float d0 = fmaf(R[0], tx, fmaf(R[3], ty, R[6] * tz));
  const float d1 = fmaf(R[1], tx, fmaf(R[4], ty, R[7] * tz));
  const float d2 = fmaf(R[2], tx, fmaf(R[5], ty, R[8] * tz));
  float m00, m01, m02, m11, m12, m22;
  fused_cov(R, r1, r2, c, m00, m01, m02, m11, m12, m22);
  const float i00 = fmaf(m11, m22, -m12 * m12);
  const float i01 = fmaf(m02, m12, -m01 * m22);
  const float i02 = fmaf(m01, m12, -m02 * m11);
  const float i11 = fmaf(m00, m22, -m02 * m02);
  const float i12 = fmaf(m01, m02, -m00 * m12);
  const float i22 = fmaf(m00, m11, -m01 * m01);
  const float det = fmaf(m00, i00, fmaf(m01, i01, m02 * i02));
  const float sc = rcp_approx(det);
  const float u0 = fmaf(i00, d0, fmaf(i01, d1, i02 * d2)) * sc;
  const float u1 = fmaf(i01, d0, fmaf(i11, d1, i12 * d2)) * sc;
  const float u2 = fmaf(i02, d0, fmaf(i12, d1, i22 * d2)) * sc;
  acc[6] = fmaf(d0, u0, fmaf(d1, u1, fmaf(d2, u2, acc[6])));
  if (MODE >= 2) {
    acc[0] = fmaf(2.0f * u1, z, fmaf(-2.0f * u2, y, acc[0]));
    acc[1] = fmaf(2.0f * u2, x, fmaf(-2.0f * u0, z, acc[1]));
    acc[2] = fmaf(2.0f * u0, y, fmaf(-2.0f * u1, x, acc[2]));
    acc[3] -= 2.0f * u0;
    acc[4] -= 2.0f * u1;
    acc[5] -= 2.0f * u2;
  }
  if (MODE == 3) {
    const float k0 = fmaf(c[0], u0, fmaf(c[1], u1, c[2] * u2));
    const float k1 = fmaf(c[1], u0, fmaf(c[3], u1, c[4] * u2));
    const float k2 = fmaf(c[2], u0, fmaf(c[4], u1, c[5] * u2));
    acc[0] = fmaf(2.0f * u1, k2, fmaf(-2.0f * u2, k1, acc[0]));
    acc[1] = fmaf(2.0f * u2, k0, fmaf(-2.0f * u0, k2, acc[1]));
    acc[2] = fmaf(2.0f * u0, k1, fmaf(-2.0f * u1, k0, acc[2]));
  }
  acc[28] += 1.0f;
}

// MODE 0: linearization (H, b, err); 1-3: cost / gradient / exact gradient;
// 4: overlap (the inlier count only: no term arithmetic, no covariance reads).
template <int MODE>
__device__ __forceinline__ void term(float* acc, const Pose32& P, float x, float y, float z,
                                     const float* c, float qx, float qy, float qz,
                                     const float4 r0, const float4 r1, const float4 r2) {
  if (MODE == 0)
    add_term(acc, P, x, y, z, c, qx, qy, qz, r0, r1, r2);
  else if (MODE == 4)
    acc[28] += 1.0f;
  else
    eval_term<MODE>(acc, P, x, y, z, c, qx, qy, qz, r0, r1, r2);
}

// ---------------------------------------------------------------------------
// Per-point kernel: one source point per thread, dynamically scheduled work
// items.  Occupancy is what hides the DRAM latency of the stream and the L2
// latency of the lookup here, so the kernel keeps its registers for the 28
// accumulators and the term arithmetic: the constants of the current work item
// (pose, map and source descriptors) live in uniform registers across the point
// loop, one per warp instead of one per lane.
// ---------------------------------------------------------------------------

struct __align__(16) ItemConst {
  float R[9];
  float t[3];                 // R, t: 3 float4
  float tmax, inv_r, margin_scale;
  uint32_t mask;              // float4 #3
  const VSlot* vslots;
  const float* pts;           // #4
  const float* covs;
  const PairDesc* pd;         // #5
  double r;
  int32_t max_probe, pad;     // #6
};

__device__ __forceinline__ float4 lds_f4(const void* p) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"((uint32_t)__cvta_generic_to_shared(p)));
  return v;
}
__device__ __forceinline__ void lds_2ptr(const void* p, uint64_t& a, uint64_t& b) {
  asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];"
               : "=l"(a), "=l"(b)
               : "r"((uint32_t)__cvta_generic_to_shared(p)));
}

// A value that is the same in all lanes of the (whole) warp, through a reduction
// whose result the compiler knows to be uniform: it then lives in a uniform register
// instead of one register per lane.
__device__ __forceinline__ uint32_t uniform(uint32_t v) { return __reduce_or_sync(0xFFFFFFFFu, v); }
__device__ __forceinline__ float uniform(float v) {
  return __uint_as_float(uniform(__float_as_uint(v)));
}
template <typename T>
__device__ __forceinline__ T* uniform(T* p) {
  const uint64_t v = reinterpret_cast<uint64_t>(p);
  return reinterpret_cast<T*>((uint64_t)uniform((uint32_t)v) |
                              ((uint64_t)uniform((uint32_t)(v >> 32)) << 32));
}

__device__ __forceinline__ MapDesc md_of_item(MapDesc md, double r) {
  md.r = r;
  return md;
}

// CTAs per SM.  The linearization, the cost and the gradients fit four (64
// registers) with the item's constants in uniform registers, slots of 12 words and the
// key without conversions; the overlap count fits eight.  27 neighbours are slower
// with more CTAs (the L1 holds less of the tables).  3 CTAs, constants re-read from
// shared memory, before: global map 2.85 -> 2.51 ms, 1,000 factors of unsorted clouds
// 812 -> 794 us, cost and gradient of 256 factors 336 -> 244 us, overlap of 3,540
// pairs 1,096 -> 691 us (four CTAs 820).  Three CTAs with the new code 2.82 ms; five
// spill (3.6 ms).
__host__ __device__ constexpr int simple_ctas(int neigh, int mode) {
  return neigh == 27 ? 3 : mode == 4 ? 8 : 4;
}

template <int NEIGH, int MODE, bool DBG>
__global__ void __launch_bounds__(kSimpleThreads, simple_ctas(NEIGH, MODE))
    linearize_simple_kernel(const __grid_constant__ LinLaunch L) {
  __shared__ float red[kSimpleThreads / 32][kAcc];
  // 27 neighbours: each thread's hits (slot offsets) of its current point
  __shared__ uint32_t hits[NEIGH == 27 ? 27 * kSimpleThreads : 1];
  __shared__ ItemConst ic;
  __shared__ int next_item;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t pol = policy_evict_last_l();
  // with occupancy blocks only the items of the maps that have none are left
  if (NEIGH == 27 && L.blocks && *L.blocks_any == 0u) return;

  for (int it = blockIdx.x; it < L.n_items;) {
    int pair, begin, end;
    tma::item_bounds(L, it, pair, begin, end);
    const bool skip = NEIGH == 27 && L.blocks && L.blocks[L.pairs[pair].map].state[0] == 0u;
    if (skip) end = begin;
    if (threadIdx.x == 0) {
      const PairDesc* pd = L.pairs ? L.pairs + pair : &L.single;
      const MapDesc md = L.maps ? L.maps[pd->map] : L.single_map;
      const SrcDesc sd = L.srcs ? L.srcs[pd->src] : L.single_src;
#pragma unroll
      for (int k = 0; k < 9; ++k) ic.R[k] = pd->R[k];
      ic.t[0] = pd->t[0];
      ic.t[1] = pd->t[1];
      ic.t[2] = pd->t[2];
      ic.tmax = pd->tmax;
      ic.inv_r = md.inv_r;
      ic.margin_scale = md.margin_scale;
      ic.mask = *md.vmask;
      ic.vslots = md.vslots;
      ic.pts = sd.pts;
      ic.covs = sd.covs;
      ic.pd = pd;
      ic.r = md.r;
      ic.max_probe = md.max_probe;
    }
    uint32_t vbase = 0;
    if (DBG && L.corr_out) {
      const PairDesc* pd = L.pairs ? L.pairs + pair : &L.single;
      vbase = *(L.maps ? L.maps[pd->map] : L.single_map).vbase;
    }
    __syncthreads();

    float acc[kAcc];
#pragma unroll
    for (int k = 0; k < kAcc; ++k) acc[k] = 0.0f;

    // the item's constants in uniform registers
    Pose32 P;
#pragma unroll
    for (int k = 0; k < 9; ++k) P.R[k] = uniform(ic.R[k]);
#pragma unroll
    for (int k = 0; k < 3; ++k) P.t[k] = uniform(ic.t[k]);
    P.tmax = uniform(ic.tmax);
    MapDesc md;
    md.inv_r = uniform(ic.inv_r);
    md.margin_scale = uniform(ic.margin_scale);
    md.vslots = uniform(ic.vslots);
    const uint32_t mask = uniform(ic.mask);
    // 32-bit offsets from uniform bases, 2^26 points (a whole number of rounds) at a time
    for (int64_t b0 = begin; b0 < end; b0 += 1 << 26) {
      const char* const pts = uniform(reinterpret_cast<const char*>(ic.pts + 3 * b0));
      const char* const covs = uniform(reinterpret_cast<const char*>(ic.covs + 6 * b0));
      const uint32_t n_here = uniform((uint32_t)min((int64_t)1 << 26, end - b0));

      for (uint32_t i = threadIdx.x; i < n_here; i += kSimpleThreads) {
        const float* pt = reinterpret_cast<const float*>(pts + 12u * i);
        const float2* cv = reinterpret_cast<const float2*>(covs + 24u * i);
        const float x = __ldg(pt + 0), y = __ldg(pt + 1), z = __ldg(pt + 2);
        const float2 c01 = __ldg(cv + 0), c23 = __ldg(cv + 1), c45 = __ldg(cv + 2);
        const float c[6] = {c01.x, c01.y, c23.x, c23.y, c45.x, c45.y};
        const float qx = fmaf(P.R[0], x, fmaf(P.R[1], y, fmaf(P.R[2], z, P.t[0])));
        const float qy = fmaf(P.R[3], x, fmaf(P.R[4], y, fmaf(P.R[5], z, P.t[1])));
        const float qz = fmaf(P.R[6], x, fmaf(P.R[7], y, fmaf(P.R[8], z, P.t[2])));
        // Exact key.  y = q / r is split into the nearest integer n and f = y - n (exact)
        // by adding and subtracting 1.5 * 2^23; floor(y) = n - (f < 0), and a face is
        // near when |f| is below the margin of source_key.  From |y| = 2^22 on the split
        // fails, and float32 may be further off than the key range is wide: binary64.  A
        // NaN is no voxel's.
        int kx, ky, kz;
        {
          const float m = fmaf(fabsf(x) + fabsf(y) + fabsf(z) + P.tmax, md.margin_scale,
                               1.1920928955078125e-7f);
          const float yx = qx * md.inv_r, yy = qy * md.inv_r, yz = qz * md.inv_r;
          constexpr float kMagic = 12582912.0f, kFar = 4194304.0f;
          constexpr int kMagicBits = 0x4B400000;
          const float nx = yx + kMagic, ny = yy + kMagic, nz = yz + kMagic;
          const float fx = yx - (nx - kMagic), fy = yy - (ny - kMagic), fz = yz - (nz - kMagic);
          kx = __float_as_int(nx) - kMagicBits + (__float_as_int(fx) >> 31);
          ky = __float_as_int(ny) - kMagicBits + (__float_as_int(fy) >> 31);
          kz = __float_as_int(nz) - kMagicBits + (__float_as_int(fz) >> 31);
          const bool inside = fabsf(yx) < kFar && fabsf(yy) < kFar && fabsf(yz) < kFar;
          const bool ax = fabsf(fx) < m, ay = fabsf(fy) < m, az = fabsf(fz) < m;
          if (!inside || (ax | ay | az)) {  // the binary64 path reads r from shared memory
            if (m != m) {
              kx = 2 * kKeyMin;  // no neighbour is in range either
            } else {
              MapDesc mr;
              mr.r = ic.r;
              if (ax || !inside) kx = axis_key_f64(ic.pd, mr, 0, x, y, z);
              if (ay || !inside) ky = axis_key_f64(ic.pd, mr, 1, x, y, z);
              if (az || !inside) kz = axis_key_f64(ic.pd, mr, 2, x, y, z);
            }
          }
          if (DBG && !inside)
            source_key(P, ic.pd, md_of_item(md, ic.r), x, y, z, qx, qy, qz, kx, ky, kz);
        }
        if (DBG && L.qkey_out) {
          L.qkey_out[3 * (b0 + i) + 0] = kx;
          L.qkey_out[3 * (b0 + i) + 1] = ky;
          L.qkey_out[3 * (b0 + i) + 2] = kz;
        }
        md.max_probe = ic.max_probe;
        if (NEIGH == 1) {
          float4 a0, a1, a2;
          uint32_t h = 0u;
          const bool hit = lookup(md, mask, kx, ky, kz, pol, h, a0, a1, a2);
          if (DBG && L.corr_out) L.corr_out[b0 + i] = hit ? (int)(md.vslots[h].vid - vbase) : -1;
          if (hit) term<MODE>(acc, P, x, y, z, c, qx, qy, qz, a0, a1, a2);
          continue;
        }
        if (DBG && L.corr_out) {
          float4 a0, a1, a2;
          uint32_t h = 0u;
          L.corr_out[b0 + i] = lookup(md, mask, kx, ky, kz, pol, h, a0, a1, a2)
                              ? (int)(md.vslots[h].vid - vbase)
                              : -1;
        }
        // the 27 probes first, hits recorded; then the terms, hit by hit, so a
        // warp evaluates a term while most of its lanes still have one.  The
        // probes go a row of three neighbours at a time, their home slots' first
        // 16 B (key, spill flag) loaded together; a miss whose home slot holds
        // another key with its spill flag set probes on
        int nh = 0;
        for (int dz = -1; dz <= 1; ++dz)
          for (int dy = -1; dy <= 1; ++dy) {
            const int yy = ky + dy, zz = kz + dz;
            const bool row_ok = key_in_range(yy) && key_in_range(zz);
            uint32_t A[3][4];
            uint32_t hh[3];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
              hh[j] = hash_key(kx + j - 1, yy, zz) & mask;
              ld_v4(md.vslots + hh[j], pol, A[j]);
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) {
              const int xx = kx + j - 1;
              if (!row_ok || !key_in_range(xx)) continue;
              const unsigned long long key = pack_key(xx, yy, zz);
              const unsigned long long k0 =
                  (unsigned long long)A[j][0] | ((unsigned long long)A[j][1] << 32);
              int hs = -1;
              if (k0 == key) {
                hs = (int)hh[j];
              } else if (k0 != kEmptyKey && A[j][kSlotSpill] != 0u) {
                uint32_t h = (hh[j] + 1) & mask;  // spilled keys: probe on
                for (int q = 1; q < md.max_probe; ++q) {
                  uint32_t a[4];
                  ld_v4(md.vslots + h, pol, a);
                  const unsigned long long k =
                      (unsigned long long)a[0] | ((unsigned long long)a[1] << 32);
                  if (k == key) { hs = (int)h; break; }
                  if (k == kEmptyKey) break;
                  h = (h + 1) & mask;
                }
              }
              if (hs >= 0) hits[27 * threadIdx.x + nh++] = (uint32_t)hs;
            }
          }
        for (int k = 0; k < nh; ++k) {
          const VSlot* t = md.vslots + hits[27 * threadIdx.x + k];
          uint32_t a[8], b[4];
          float4 a0, a1, a2;
          ld_slot(t, pol, a, b);
          slot_gaussian(a, b, a0, a1, a2);
          term<MODE>(acc, P, x, y, z, c, qx, qy, qz, a0, a1, a2);
        }
      }
    }

#pragma unroll
    for (int k = 0; k < kAcc; ++k) {
      float v = acc[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
      acc[k] = v;
    }
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < kAcc; ++k) red[warp][k] = acc[k];
    }
    // (no status word: a CTA per item)
    if (threadIdx.x == 0)
      next_item = L.status ? (int)gridDim.x + atomicAdd(L.status + 1, 1) : L.n_items;
    __syncthreads();
    if (threadIdx.x < kAcc && !skip) {
      double s = 0.0;
      for (int w = 0; w < kSimpleThreads / 32; ++w) s += (double)red[w][threadIdx.x];
      L.partials[(int64_t)it * kPartialStride + threadIdx.x] = s;
    }
    it = next_item;  // read between the two barriers; rewritten only after the second
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// 27 neighbours from occupancy blocks (vgicp_blocks.cu): one point per thread, work
// items claimed as in the per-point kernel.  The masks of the 1 - 8 blocks around a
// point are shifted so that bit z * 16 + y * 4 + x says whether neighbour (x, y, z) of
// the 3 x 3 x 3 block exists, and its set bits in ascending order are the neighbours in
// the order of the per-point kernel (dz, dy, dx), so the sums are the same bit for bit.
// A neighbour's record is found from its block's mask and first record, which wait in
// shared memory; the next neighbour's record is loaded while the current one's term is
// evaluated.
// Bounded by issue, with 20 of 32 lanes active (a lane has 0 to 27 terms): 96M source
// points of 48 large-map submaps 13.1 -> 9.4 ms, and 0.2 ms to build the blocks; of
// the 9.4 ms the search takes 2.3 (the probes took 8.4), the records' places 1.3, their
// loads 1.2, the terms 4.6.  Four or two CTAs per SM: 10.2, 10.7 ms.
// ---------------------------------------------------------------------------
namespace blocks {
// Moves the cells that a block holds of a window of three, starting at cell `lo` (0..3)
// of the first block, to their place in the window, along the axis whose cells are W
// bits apart (all_lowest: the lowest cell of the axis everywhere): second = false: cells
// lo .. 3 down by lo, true: cells 0 .. lo - 2 up by 4 - lo.
template <int W>
__device__ __forceinline__ uint64_t to_window(uint64_t m, int lo, bool second) {
  // the first three cells of every group of four, along this axis
  constexpr uint64_t kCell = W == 1 ? 0x1111111111111111ull : W == 4 ? 0x000F000F000F000Full
                                                                     : 0x000000000000FFFFull;
  constexpr uint64_t kThree = kCell | (kCell << W) | (kCell << (2 * W));
  if (second) {  // cells 0 .. lo - 2 (lo >= 2)
    const uint64_t keep = lo == 3 ? kCell | (kCell << W) : kCell;
    return (m & keep) << (W * (4 - lo));
  }
  const uint64_t keep = lo == 0 ? kThree : lo == 1 ? kThree << W : lo == 2 ? (kCell | (kCell << W)) << (2 * W)
                                                                          : kCell << (3 * W);
  return (m & keep) >> (W * lo);
}

constexpr int kCtas = 3;  // per SM
template <int MODE>
__global__ void __launch_bounds__(kSimpleThreads, kCtas)
    linearize_blocks_kernel(const __grid_constant__ LinLaunch L) {
  __shared__ float red[kSimpleThreads / 32][kAcc];
  // each thread's half blocks (4 x 4 x 2), hz * 4 + cy * 2 + cx: mask, first record
  __shared__ uint2 s_half[12][kSimpleThreads];
  __shared__ ItemConst ic;
  __shared__ BlockMap bm;
  __shared__ int next_item;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t pol = policy_evict_last_l();

  for (int it = blockIdx.x; it < L.n_items;) {
    int pair, begin, end;
    tma::item_bounds(L, it, pair, begin, end);
    const PairDesc* pd = L.pairs + pair;
    const bool skip = L.blocks[pd->map].state[0] != 0u;  // the same for the CTA
    if (threadIdx.x == 0) {
      const MapDesc md = L.maps[pd->map];
      const SrcDesc sd = L.srcs[pd->src];
#pragma unroll
      for (int k = 0; k < 9; ++k) ic.R[k] = pd->R[k];
      ic.t[0] = pd->t[0];
      ic.t[1] = pd->t[1];
      ic.t[2] = pd->t[2];
      ic.tmax = pd->tmax;
      ic.inv_r = md.inv_r;
      ic.margin_scale = md.margin_scale;
      ic.pts = sd.pts;
      ic.covs = sd.covs;
      ic.pd = pd;
      ic.r = md.r;
      bm = L.blocks[pd->map];
    }
    __syncthreads();
    float acc[kAcc];
#pragma unroll
    for (int k = 0; k < kAcc; ++k) acc[k] = 0.0f;
    Pose32 P;
#pragma unroll
    for (int k = 0; k < 9; ++k) P.R[k] = uniform(ic.R[k]);
#pragma unroll
    for (int k = 0; k < 3; ++k) P.t[k] = uniform(ic.t[k]);
    P.tmax = uniform(ic.tmax);
    MapDesc md;
    md.inv_r = uniform(ic.inv_r);
    md.margin_scale = uniform(ic.margin_scale);
    const BlockSlot* const table = uniform(bm.table);
    const float4* const recs = uniform(bm.recs);
    const uint32_t mask = uniform(bm.mask);

    for (int64_t p = skip ? end : begin + (int)threadIdx.x; p < end; p += kSimpleThreads) {
      const float* pt = ic.pts + 3 * p;
      const float x = __ldg(pt + 0), y = __ldg(pt + 1), z = __ldg(pt + 2);
      const float2* cv = reinterpret_cast<const float2*>(ic.covs + 6 * p);
      const float2 c01 = __ldg(cv + 0), c23 = __ldg(cv + 1), c45 = __ldg(cv + 2);
      const float c[6] = {c01.x, c01.y, c23.x, c23.y, c45.x, c45.y};
      const float qx = fmaf(P.R[0], x, fmaf(P.R[1], y, fmaf(P.R[2], z, P.t[0])));
      const float qy = fmaf(P.R[3], x, fmaf(P.R[4], y, fmaf(P.R[5], z, P.t[1])));
      const float qz = fmaf(P.R[6], x, fmaf(P.R[7], y, fmaf(P.R[8], z, P.t[2])));
      int kx, ky, kz;
      source_key(P, ic.pd, md_of_item(md, ic.r), x, y, z, qx, qy, qz, kx, ky, kz);
      // no neighbour is in the key range beyond one voxel outside it
      if (kx < kKeyMin - 1 || kx > kKeyMax + 1 || ky < kKeyMin - 1 || ky > kKeyMax + 1 ||
          kz < kKeyMin - 1 || kz > kKeyMax + 1)
        continue;
      const int lx = (kx - 1) & 3, ly = (ky - 1) & 3, lz = (kz - 1) & 3;
      const int bx = (kx - 1) >> 2, by = (ky - 1) >> 2, bz = (kz - 1) >> 2;
      uint64_t occ = 0ull;  // window bits
#pragma unroll 1
      for (int cz = 0; cz <= (lz >= 2); ++cz) {
        uint64_t slab = 0ull;
#pragma unroll 1
        for (int cy = 0; cy <= (ly >= 2); ++cy) {
          uint64_t rows = 0ull;
          // the two blocks of a row: their home slots loaded together
          uint32_t a[2][8];
          uint32_t h[2];
#pragma unroll
          for (int cx = 0; cx < 2; ++cx) {
            h[cx] = hash_key(bx + cx, by + cy, bz + cz) & mask;
            if (cx == 0 || lx >= 2) ld_v8(table + h[cx], pol, a[cx]);
          }
#pragma unroll
          for (int cx = 0; cx < 2; ++cx) {
            if (cx == 1 && lx < 2) continue;
            const unsigned long long key = block_key(bx + cx, by + cy, bz + cz);
            unsigned long long k = slot_key(a[cx]);
            for (int q = 1; q < kBlockProbes && k != key && k != 0ull; ++q) {
              h[cx] = (h[cx] + 1) & mask;
              ld_v8(table + h[cx], pol, a[cx]);
              k = slot_key(a[cx]);
            }
            if (k != key) continue;
            const uint64_t bits = (uint64_t)a[cx][2] | ((uint64_t)a[cx][3] << 32);
            // the window reaches half blocks 0 - 2 in z (cells lz .. lz + 2 <= 5)
            const int b = cz * 8 + cy * 2 + cx;
            s_half[b][threadIdx.x] = make_uint2(a[cx][2], a[cx][4]);
            if (cz == 0)
              s_half[b + 4][threadIdx.x] =
                  make_uint2(a[cx][3], a[cx][4] + (uint32_t)__popc(a[cx][2]));
            rows |= to_window<1>(bits, lx, cx == 1);
          }
          slab |= to_window<4>(rows, ly, cy == 1);
        }
        occ |= to_window<16>(slab, lz, cz == 1);
      }
      if (occ == 0ull) continue;
      // the neighbours, two slabs of the window (32 bits) and then the third
      uint32_t now = (uint32_t)occ, then = (uint32_t)(occ >> 32);
      int z0 = lz;
      auto next = [&]() {  // record of the lowest bit, which is cleared
        if (now == 0u) {
          now = then;
          then = 0u;
          z0 = lz + 2;
        }
        const int wbit = __ffs((int)now) - 1;
        now &= now - 1u;
        const int wx = lx + (wbit & 3), wy = ly + ((wbit >> 2) & 3), wz = z0 + (wbit >> 4);
        const int bit = (wz & 1) * 16 + (wy & 3) * 4 + (wx & 3);
        const uint2 m = s_half[(wz >> 1) * 4 + (wy >> 2) * 2 + (wx >> 2)][threadIdx.x];
        return recs + 3 * (m.y + (uint32_t)__popc(m.x & ((1u << bit) - 1u)));
      };
      const float4* rec = next();
      float4 n0 = __ldg(rec), n1 = __ldg(rec + 1), n2 = __ldg(rec + 2);
      while (true) {
        const float4 r0 = n0, r1 = n1, r2 = n2;
        const bool more = (now | then) != 0u;
        if (more) {
          rec = next();
          n0 = __ldg(rec);
          n1 = __ldg(rec + 1);
          n2 = __ldg(rec + 2);
        }
        term<MODE>(acc, P, x, y, z, c, qx, qy, qz, r0, r1, r2);
        if (!more) break;
      }
    }

#pragma unroll
    for (int k = 0; k < kAcc; ++k) {
      float v = acc[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
      acc[k] = v;
    }
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < kAcc; ++k) red[warp][k] = acc[k];
    }
    if (threadIdx.x == 0) next_item = (int)gridDim.x + atomicAdd(L.status + 1, 1);
    __syncthreads();
    if (threadIdx.x < kAcc && !skip) {
      double s = 0.0;
      for (int w = 0; w < kSimpleThreads / 32; ++w) s += (double)red[w][threadIdx.x];
      L.partials[(int64_t)it * kPartialStride + threadIdx.x] = s;
    }
    it = next_item;  // read between the two barriers; rewritten only after the second
    __syncthreads();
  }
}
}  // namespace blocks

template <int NEIGH, int MODE>
void launch_simple(const LinLaunch& L, int grid, cudaStream_t st) {
  if (L.corr_out || L.qkey_out)
    linearize_simple_kernel<NEIGH, MODE, true><<<grid, kSimpleThreads, 0, st>>>(L);
  else
    linearize_simple_kernel<NEIGH, MODE, false><<<grid, kSimpleThreads, 0, st>>>(L);
}

// ---------------------------------------------------------------------------
// Hit-compacting per-warp kernel (1 neighbour).  The lookup phase runs one
// point per lane; the lanes whose voxel exists push (point, covariance, target-
// frame residual mu' - q, voxel covariance) as one 80-B entry into their warp's
// queue in shared memory.  Whenever 32 entries are queued the warp evaluates
// them with every lane busy, so lanes whose point missed do not cost term
// arithmetic.  Item constants live in shared memory as in the per-point kernel.
// ---------------------------------------------------------------------------
namespace compact {
#ifndef VGICP_COMPACT_MIN_BLOCKS
#define VGICP_COMPACT_MIN_BLOCKS 3
#endif
constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kQueue = 64;  // entries per warp (< 32 left after a drain + at most 32 pushed)

__device__ __forceinline__ void eval_entry(float* acc, const float* R, const float4* E) {
  const float4 e0 = E[0], e1 = E[1], e2 = E[2], e3 = E[3], e4 = E[4];
  const float c[6] = {e0.w, e1.x, e1.y, e1.z, e1.w, e2.x};
  add_term_t(acc, R, e0.x, e0.y, e0.z, c, e2.y, e2.z, e2.w, e3, e4);
}

__global__ void __launch_bounds__(kThreads, VGICP_COMPACT_MIN_BLOCKS)
    linearize_compact_kernel(const __grid_constant__ LinLaunch L) {
  __shared__ __align__(16) float4 queue[kWarps][kQueue * 5];
  __shared__ float red[kWarps][kAcc];
  __shared__ ItemConst ic;
  __shared__ int next_item;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t lt_mask = (1u << lane) - 1u;
  const uint64_t pol = policy_evict_last_l();
  float4* Q = queue[warp];

  for (int it = blockIdx.x; it < L.n_items;) {
    int pair, begin, end;
    tma::item_bounds(L, it, pair, begin, end);
    if (threadIdx.x == 0) {
      const PairDesc* pd = L.pairs ? L.pairs + pair : &L.single;
      const MapDesc md = L.maps ? L.maps[pd->map] : L.single_map;
      const SrcDesc sd = L.srcs ? L.srcs[pd->src] : L.single_src;
#pragma unroll
      for (int k = 0; k < 9; ++k) ic.R[k] = pd->R[k];
      ic.t[0] = pd->t[0];
      ic.t[1] = pd->t[1];
      ic.t[2] = pd->t[2];
      ic.tmax = pd->tmax;
      ic.inv_r = md.inv_r;
      ic.margin_scale = md.margin_scale;
      ic.mask = *md.vmask;
      ic.vslots = md.vslots;
      ic.pts = sd.pts;
      ic.covs = sd.covs;
      ic.pd = pd;
      ic.r = md.r;
      ic.max_probe = md.max_probe;
    }
    __syncthreads();

    float acc[kAcc];
#pragma unroll
    for (int k = 0; k < kAcc; ++k) acc[k] = 0.0f;
    int qn = 0;  // queued entries (warp-uniform)
    const int n = end - begin;

    for (int base = warp * 32; base < n; base += kThreads) {
      const int p = begin + base + lane;
      bool hit = false;
      float x = 0.f, y = 0.f, z = 0.f, tx = 0.f, ty = 0.f, tz = 0.f;
      float2 c01, c23, c45;
      float4 a1, a2;
      if (p < end) {
        const float4 g0 = lds_f4(&ic.R[0]), g1 = lds_f4(&ic.R[4]), g2 = lds_f4(&ic.R[8]);
        const float4 g3 = lds_f4(&ic.tmax);
        uint64_t vs, ps, cs, pds;
        lds_2ptr(&ic.vslots, vs, ps);
        lds_2ptr(&ic.covs, cs, pds);
        const float* pt = reinterpret_cast<const float*>(ps) + 3 * (int64_t)p;
        x = __ldg(pt + 0);
        y = __ldg(pt + 1);
        z = __ldg(pt + 2);
        const float2* cv = reinterpret_cast<const float2*>(reinterpret_cast<const float*>(cs) +
                                                           6 * (int64_t)p);
        c01 = __ldg(cv + 0);
        c23 = __ldg(cv + 1);
        c45 = __ldg(cv + 2);
        const float qx = fmaf(g0.x, x, fmaf(g0.y, y, fmaf(g0.z, z, g2.y)));
        const float qy = fmaf(g0.w, x, fmaf(g1.x, y, fmaf(g1.y, z, g2.z)));
        const float qz = fmaf(g1.z, x, fmaf(g1.w, y, fmaf(g2.x, z, g2.w)));
        const float S = fabsf(x) + fabsf(y) + fabsf(z) + g3.x;
        const float m = fmaf(S, g3.z, 1.1920928955078125e-7f);
        const float yx = qx * g3.y, yy = qy * g3.y, yz = qz * g3.y;
        const float fx = floorf(yx), fy = floorf(yy), fz = floorf(yz);
        const float rx = yx - fx, ry = yy - fy, rz = yz - fz;
        const bool ax = (rx < m) | (rx > 1.0f - m);
        const bool ay = (ry < m) | (ry > 1.0f - m);
        const bool az = (rz < m) | (rz > 1.0f - m);
        int kx = clamp_to_int(fx), ky = clamp_to_int(fy), kz = clamp_to_int(fz);
        if (ax | ay | az) {
          const PairDesc* pd = reinterpret_cast<const PairDesc*>(pds);
          MapDesc mr;
          mr.r = ic.r;
          if (ax) kx = axis_key_f64(pd, mr, 0, x, y, z);
          if (ay) ky = axis_key_f64(pd, mr, 1, x, y, z);
          if (az) kz = axis_key_f64(pd, mr, 2, x, y, z);
        }
        MapDesc md;
        md.vslots = reinterpret_cast<const VSlot*>(vs);
        md.max_probe = ic.max_probe;
        float4 a0;
        uint32_t h = 0u;
        hit = lookup(md, __float_as_uint(g3.w), kx, ky, kz, pol, h, a0, a1, a2);
        tx = a0.x - qx;
        ty = a0.y - qy;
        tz = a0.z - qz;
      }
      const uint32_t hm = __ballot_sync(0xFFFFFFFFu, hit);
      if (hit) {
        float4* E = Q + 5 * (qn + __popc(hm & lt_mask));
        E[0] = make_float4(x, y, z, c01.x);
        E[1] = make_float4(c01.y, c23.x, c23.y, c45.x);
        E[2] = make_float4(c45.y, tx, ty, tz);
        E[3] = a1;
        E[4] = a2;
      }
      if (lane == 0) acc[28] += (float)__popc(hm);
      qn += __popc(hm);
      __syncwarp();
      if (qn >= 32) {  // one full warp of terms: lane l takes entry qn - 32 + l
        const float4 g0 = lds_f4(&ic.R[0]), g1 = lds_f4(&ic.R[4]), g2 = lds_f4(&ic.R[8]);
        const float R[9] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w, g2.x};
        eval_entry(acc, R, Q + 5 * (qn - 32 + lane));
        qn -= 32;
        __syncwarp();
      }
    }
    if (lane < qn) {  // drain the partially filled queue
      const float4 g0 = lds_f4(&ic.R[0]), g1 = lds_f4(&ic.R[4]), g2 = lds_f4(&ic.R[8]);
      const float R[9] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w, g2.x};
      eval_entry(acc, R, Q + 5 * lane);
    }
    __syncwarp();

#pragma unroll
    for (int k = 0; k < kAcc; ++k) {
      float v = acc[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
      acc[k] = v;
    }
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < kAcc; ++k) red[warp][k] = acc[k];
    }
    if (threadIdx.x == 0) next_item = (int)gridDim.x + atomicAdd(L.status + 1, 1);
    __syncthreads();
    if (threadIdx.x < kAcc) {
      double t = 0.0;
      for (int w = 0; w < kWarps; ++w) t += (double)red[w][threadIdx.x];
      L.partials[(int64_t)it * kPartialStride + threadIdx.x] = t;
    }
    it = next_item;  // read between the two barriers; rewritten only after the second
    __syncthreads();
  }
}
}  // namespace compact


// ---------------------------------------------------------------------------
// Few long work items (1 neighbour): one cluster of 8 CTAs per item.
//
// A thread of the per-point kernel takes its points of an item one after the other
// (64 of a 16K item), and a factor set of a few items, a sliding window for
// instance, lasts as long as that chain: 72 us for ten factors of 20,000 points on
// 20 of 152 SMs.  Here CTA w of the cluster takes what warp w of the per-point
// kernel takes.  Its 8 warps look up and invert 16 points of every lane at once (two
// per thread, in flight together) and leave them in shared memory; then each
// accumulator is summed over them by one thread per lane, in the order in which the
// per-point kernel adds them, so every sum is the same bit for bit.  The
// accumulators are dealt to warps 0 - 4; the CTAs' sums meet in the first CTA
// through distributed shared memory.
//
// The SMs do more work per point this way (all threads wait for the sums), so it
// is for few items (split_items).  Bounded by the latency of a round (two loads, a
// barrier) and by the sums' shared-memory reads.
// ---------------------------------------------------------------------------
namespace split {
constexpr int kCtas = 8;          // CTAs per item = warps of the per-point kernel
constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;
constexpr int kPer = 2;           // points per thread and round
constexpr int kRound = kWarps * kPer;
static_assert(kCtas * 32 == kSimpleThreads, "one CTA per warp of the per-point kernel");

// What the sums need of a point: MODE 0: adj(M') (6), 1 / det, u (3), d (3), x, y,
// z; modes 1 - 3: u, d, x, y, z and C_k u.
__host__ __device__ constexpr int values(int mode) { return mode == 0 ? 16 : mode == 3 ? 12 : mode == 2 ? 9 : 6; }

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::
                   : "memory");
}
// Address of a shared-memory object of CTA `rank` of the cluster, and a store there.
__device__ __forceinline__ uint32_t map_rank(const void* p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void store_cluster(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

template <int MODE>
__global__ void __cluster_dims__(kCtas, 1, 1) __launch_bounds__(kThreads, 2)
    linearize_split_kernel(const __grid_constant__ LinLaunch L) {
  constexpr int NV = values(MODE);
  __shared__ float val[kRound][NV][32];
  __shared__ float red[kCtas][kAcc];  // the first CTA's receives every CTA's sums
  __shared__ float mine[kAcc];
  __shared__ ItemConst ic;
  __shared__ int hits;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int it = blockIdx.x / kCtas;
  const uint32_t w = cluster_rank();
  const uint64_t pol = policy_evict_last_l();
  int pair, begin, end;
  tma::item_bounds(L, it, pair, begin, end);
  if (threadIdx.x == 0) {
    const PairDesc* pd = L.pairs ? L.pairs + pair : &L.single;
    const MapDesc md = L.maps ? L.maps[pd->map] : L.single_map;
    const SrcDesc sd = L.srcs ? L.srcs[pd->src] : L.single_src;
#pragma unroll
    for (int k = 0; k < 9; ++k) ic.R[k] = pd->R[k];
    ic.t[0] = pd->t[0];
    ic.t[1] = pd->t[1];
    ic.t[2] = pd->t[2];
    ic.tmax = pd->tmax;
    ic.inv_r = md.inv_r;
    ic.margin_scale = md.margin_scale;
    ic.mask = *md.vmask;
    ic.vslots = md.vslots;
    ic.pts = sd.pts;
    ic.covs = sd.covs;
    ic.pd = pd;
    ic.r = md.r;
    ic.max_probe = md.max_probe;
    hits = 0;
  }
  if (threadIdx.x < kAcc) mine[threadIdx.x] = 0.0f;
  __syncthreads();
  Pose32 P;
#pragma unroll
  for (int k = 0; k < 9; ++k) P.R[k] = ic.R[k];
  P.t[0] = ic.t[0];
  P.t[1] = ic.t[1];
  P.t[2] = ic.t[2];
  P.tmax = ic.tmax;
  MapDesc md;
  md.vslots = ic.vslots;
  md.inv_r = ic.inv_r;
  md.margin_scale = ic.margin_scale;
  md.r = ic.r;
  md.max_probe = ic.max_probe;
  const uint32_t mask = ic.mask;
  const float* R = P.R;

  float acc[kAcc];
#pragma unroll
  for (int k = 0; k < kAcc; ++k) acc[k] = 0.0f;
  const int p0 = begin + (int)w * 32 + lane;
  // points of the longest lane (lane 0)
  const int n0 = end - begin - (int)w * 32;
  const int steps = n0 > 0 ? (n0 + kSimpleThreads - 1) / kSimpleThreads : 0;
  int my_hits = 0;
  for (int j0 = 0; j0 < steps; j0 += kRound) {
    // ---- kPer points per thread: key, first probe of each, resolve, terms ----
    float x[kPer], y[kPer], z[kPer], c[kPer][6], q[kPer][3];
    int kx[kPer], ky[kPer], kz[kPer];
    uint32_t h[kPer], sa[kPer][8], sb[kPer][4];
    unsigned long long key[kPer];
    bool live[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int64_t p = (int64_t)p0 + (int64_t)kSimpleThreads * (j0 + warp * kPer + u);
      live[u] = p < end;
      if (live[u]) {
        const float* pt = ic.pts + 3 * p;
        x[u] = __ldg(pt + 0);
        y[u] = __ldg(pt + 1);
        z[u] = __ldg(pt + 2);
        const float2* cv = reinterpret_cast<const float2*>(ic.covs + 6 * p);
        const float2 c01 = __ldg(cv + 0), c23 = __ldg(cv + 1), c45 = __ldg(cv + 2);
        c[u][0] = c01.x; c[u][1] = c01.y; c[u][2] = c23.x;
        c[u][3] = c23.y; c[u][4] = c45.x; c[u][5] = c45.y;
      }
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      key[u] = kEmptyKey;
      if (live[u]) {
        q[u][0] = fmaf(R[0], x[u], fmaf(R[1], y[u], fmaf(R[2], z[u], P.t[0])));
        q[u][1] = fmaf(R[3], x[u], fmaf(R[4], y[u], fmaf(R[5], z[u], P.t[1])));
        q[u][2] = fmaf(R[6], x[u], fmaf(R[7], y[u], fmaf(R[8], z[u], P.t[2])));
        source_key(P, ic.pd, md, x[u], y[u], z[u], q[u][0], q[u][1], q[u][2], kx[u], ky[u], kz[u]);
        live[u] = key_in_range(kx[u]) && key_in_range(ky[u]) && key_in_range(kz[u]);
      }
      if (live[u]) {
        key[u] = pack_key(kx[u], ky[u], kz[u]);
        h[u] = hash_key(kx[u], ky[u], kz[u]) & mask;
        ld_slot(md.vslots + h[u], pol, sa[u], sb[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      bool hit = false;
      if (live[u]) {
        unsigned long long t = slot_key(sa[u]);
        for (int p = 1; t != key[u] && t != kEmptyKey && (p > 1 || sa[u][kSlotSpill] != 0u) &&
                        p < md.max_probe;
             ++p) {
          h[u] = (h[u] + 1) & mask;
          ld_slot(md.vslots + h[u], pol, sa[u], sb[u]);
          t = slot_key(sa[u]);
        }
        hit = t == key[u];
      }
      float v[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) v[k] = 0.0f;  // a miss adds zeros
      if (hit) {
        float4 r0, r1, r2;
        slot_gaussian(sa[u], sb[u], r0, r1, r2);
        const float tx = r0.x - q[u][0], ty = r0.y - q[u][1], tz = r0.z - q[u][2];
        const float d0 = fmaf(R[0], tx, fmaf(R[3], ty, R[6] * tz));
        const float d1 = fmaf(R[1], tx, fmaf(R[4], ty, R[7] * tz));
        const float d2 = fmaf(R[2], tx, fmaf(R[5], ty, R[8] * tz));
        float m00, m01, m02, m11, m12, m22;
        fused_cov(R, r1, r2, c[u], m00, m01, m02, m11, m12, m22);
        const float i00 = fmaf(m11, m22, -m12 * m12);
        const float i01 = fmaf(m02, m12, -m01 * m22);
        const float i02 = fmaf(m01, m12, -m02 * m11);
        const float i11 = fmaf(m00, m22, -m02 * m02);
        const float i12 = fmaf(m01, m02, -m00 * m12);
        const float i22 = fmaf(m00, m11, -m01 * m01);
        const float det = fmaf(m00, i00, fmaf(m01, i01, m02 * i02));
        const float sc = rcp_approx(det);
        if (MODE == 0) {
          const float w00 = __fmul_rn(i00, sc), w01 = __fmul_rn(i01, sc), w02 = __fmul_rn(i02, sc);
          const float w11 = __fmul_rn(i11, sc), w12 = __fmul_rn(i12, sc), w22 = __fmul_rn(i22, sc);
          v[0] = i00; v[1] = i01; v[2] = i02; v[3] = i11; v[4] = i12; v[5] = i22; v[6] = sc;
          v[7] = fmaf(w00, d0, fmaf(w01, d1, w02 * d2));
          v[8] = fmaf(w01, d0, fmaf(w11, d1, w12 * d2));
          v[9] = fmaf(w02, d0, fmaf(w12, d1, w22 * d2));
          v[10] = d0; v[11] = d1; v[12] = d2;
          v[13] = x[u]; v[14] = y[u]; v[15] = z[u];
        } else {
          const float u0 = fmaf(i00, d0, fmaf(i01, d1, i02 * d2)) * sc;
          const float u1 = fmaf(i01, d0, fmaf(i11, d1, i12 * d2)) * sc;
          const float u2 = fmaf(i02, d0, fmaf(i12, d1, i22 * d2)) * sc;
          v[0] = u0; v[1] = u1; v[2] = u2; v[3] = d0; v[4] = d1; v[5] = d2;
          if (MODE >= 2) {
            v[NV > 6 ? 6 : 0] = x[u]; v[NV > 6 ? 7 : 0] = y[u]; v[NV > 6 ? 8 : 0] = z[u];
          }
          if (MODE == 3) {
            v[NV > 9 ? 9 : 0] = fmaf(c[u][0], u0, fmaf(c[u][1], u1, c[u][2] * u2));
            v[NV > 9 ? 10 : 0] = fmaf(c[u][1], u0, fmaf(c[u][3], u1, c[u][4] * u2));
            v[NV > 9 ? 11 : 0] = fmaf(c[u][2], u0, fmaf(c[u][4], u1, c[u][5] * u2));
          }
        }
        ++my_hits;
      }
#pragma unroll
      for (int k = 0; k < NV; ++k) val[warp * kPer + u][k][lane] = v[k];
    }
    __syncthreads();
    // ---- the sums, point after point (the expressions of add_term / eval_term) ----
    const int n = min(kRound, steps - j0);
    if (MODE == 0) {
      if (warp < 3) {
        for (int j = 0; j < n; ++j) {
          const float s = val[j][6][lane];
          const float px = val[j][13][lane], py = val[j][14][lane], pz = val[j][15][lane];
          const float w00 = __fmul_rn(val[j][0][lane], s), w01 = __fmul_rn(val[j][1][lane], s);
          const float w02 = __fmul_rn(val[j][2][lane], s), w11 = __fmul_rn(val[j][3][lane], s);
          const float w12 = __fmul_rn(val[j][4][lane], s), w22 = __fmul_rn(val[j][5][lane], s);
          if (warp == 0) {
            const float p00 = fmaf(py, w02, -pz * w01), p01 = fmaf(py, w12, -pz * w11),
                        p02 = fmaf(py, w22, -pz * w12);
            acc[6] += p00; acc[7] += p01; acc[8] += p02;
            acc[0] = fmaf(p02, py, fmaf(-p01, pz, acc[0]));
            acc[1] = fmaf(p00, pz, fmaf(-p02, px, acc[1]));
            acc[2] = fmaf(p01, px, fmaf(-p00, py, acc[2]));
          } else if (warp == 1) {
            const float p10 = fmaf(pz, w00, -px * w02), p11 = fmaf(pz, w01, -px * w12),
                        p12 = fmaf(pz, w02, -px * w22);
            acc[9] += p10; acc[10] += p11; acc[11] += p12;
            acc[3] = fmaf(p10, pz, fmaf(-p12, px, acc[3]));
            acc[4] = fmaf(p11, px, fmaf(-p10, py, acc[4]));
          } else {
            const float p20 = fmaf(px, w01, -py * w00), p21 = fmaf(px, w11, -py * w01),
                        p22 = fmaf(px, w12, -py * w02);
            acc[12] += p20; acc[13] += p21; acc[14] += p22;
            acc[5] = fmaf(p21, px, fmaf(-p20, py, acc[5]));
          }
        }
      } else if (warp == 3) {
        for (int j = 0; j < n; ++j) {
          const float s = val[j][6][lane];
#pragma unroll
          for (int k = 0; k < 6; ++k)
            acc[15 + k] = __fadd_rn(acc[15 + k], __fmul_rn(val[j][k][lane], s));
        }
      } else if (warp == 4) {
        for (int j = 0; j < n; ++j) {
          const float u0 = val[j][7][lane], u1 = val[j][8][lane], u2 = val[j][9][lane];
          const float d0 = val[j][10][lane], d1 = val[j][11][lane], d2 = val[j][12][lane];
          const float px = val[j][13][lane], py = val[j][14][lane], pz = val[j][15][lane];
          acc[27] = fmaf(d0, u0, fmaf(d1, u1, fmaf(d2, u2, acc[27])));
          acc[21] = fmaf(u1, pz, fmaf(-u2, py, acc[21]));
          acc[22] = fmaf(u2, px, fmaf(-u0, pz, acc[22]));
          acc[23] = fmaf(u0, py, fmaf(-u1, px, acc[23]));
          acc[24] -= u0;
          acc[25] -= u1;
          acc[26] -= u2;
        }
      }
    } else if (warp == 0) {
      for (int j = 0; j < n; ++j) {
        const float u0 = val[j][0][lane], u1 = val[j][1][lane], u2 = val[j][2][lane];
        const float d0 = val[j][3][lane], d1 = val[j][4][lane], d2 = val[j][5][lane];
        acc[6] = fmaf(d0, u0, fmaf(d1, u1, fmaf(d2, u2, acc[6])));
        if (MODE >= 2) {
          const float px = val[j][NV > 6 ? 6 : 0][lane], py = val[j][NV > 6 ? 7 : 0][lane],
                      pz = val[j][NV > 6 ? 8 : 0][lane];
          acc[0] = fmaf(2.0f * u1, pz, fmaf(-2.0f * u2, py, acc[0]));
          acc[1] = fmaf(2.0f * u2, px, fmaf(-2.0f * u0, pz, acc[1]));
          acc[2] = fmaf(2.0f * u0, py, fmaf(-2.0f * u1, px, acc[2]));
          acc[3] -= 2.0f * u0;
          acc[4] -= 2.0f * u1;
          acc[5] -= 2.0f * u2;
        }
        if (MODE == 3) {
          const float k0 = val[j][NV > 9 ? 9 : 0][lane], k1 = val[j][NV > 9 ? 10 : 0][lane],
                      k2 = val[j][NV > 9 ? 11 : 0][lane];
          acc[0] = fmaf(2.0f * u1, k2, fmaf(-2.0f * u2, k1, acc[0]));
          acc[1] = fmaf(2.0f * u2, k0, fmaf(-2.0f * u0, k2, acc[1]));
          acc[2] = fmaf(2.0f * u0, k1, fmaf(-2.0f * u1, k0, acc[2]));
        }
      }
    }
    __syncthreads();  // val is rewritten by the next round
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) my_hits += __shfl_xor_sync(0xFFFFFFFFu, my_hits, o);
  if (lane == 0 && my_hits) atomicAdd(&hits, my_hits);
  // the warp tree of the per-point kernel; an accumulator is nonzero in one warp only
#pragma unroll
  for (int k = 0; k < kAcc - 1; ++k) {
    const int owner = MODE != 0 ? 0
                      : k < 3 ? 0 : k < 5 ? 1 : k < 6 ? 2 : k < 9 ? 0 : k < 12 ? 1 : k < 15 ? 2
                      : k < 21 ? 3 : 4;
    if (MODE != 0 && k > 6) continue;
    if (warp == owner) {
      float v = acc[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
      if (lane == 0) mine[k] = v;
    }
  }
  cluster_sync();  // every CTA of the cluster runs, and its own sums are in place
  if (threadIdx.x < kAcc)
    store_cluster(map_rank(&red[w][threadIdx.x], 0),
                  threadIdx.x == kAcc - 1 ? (float)hits : mine[threadIdx.x]);
  cluster_sync();
  if (w == 0 && threadIdx.x < kAcc) {
    double s = 0.0;
    for (int k = 0; k < kCtas; ++k) s += (double)red[k][threadIdx.x];
    L.partials[(int64_t)it * kPartialStride + threadIdx.x] = s;
  }
}
}  // namespace split

// ---------------------------------------------------------------------------
// Work items for at most two CTAs per SM (one neighbour): a CTA per item, four points
// per thread at a time (two with two CTAs per SM) with their lookups in flight
// together, and the next ones loaded while these are evaluated.
//
// The per-point kernel hides its loads behind other warps.  With one or two CTAs per SM
// there are too few, and a thread's 64 points of a 16K item, each waiting for its
// stream and then for its lookup, set the time.  At two CTAs per SM a thread may have
// 128 registers, at one 255: room for the lookups of two or four points and for the next
// points.  Each thread keeps its points and adds their terms in their order, so the
// sums are those of the per-point kernel bit for bit.  Bounded by the latency of a
// round (a lookup, the terms).  A plan's execution, factors of 16,000 points, maps as
// sources / unsorted clouds: 152 factors 102 / 104 -> 63 / 66 us, 300 factors
// 113 / 129 -> 86 / 98 us.
// ---------------------------------------------------------------------------
namespace ahead {
// kPer: points per thread and round
template <int MODE, int kPer>
__global__ void __launch_bounds__(kSimpleThreads, 4 / kPer)
    linearize_ahead_kernel(const __grid_constant__ LinLaunch L) {
  __shared__ float red[kSimpleThreads / 32][kAcc];
  __shared__ ItemConst ic;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int it = blockIdx.x;
  const uint64_t pol = policy_evict_last_l();
  int pair, begin, end;
  tma::item_bounds(L, it, pair, begin, end);
  if (threadIdx.x == 0) {
    const PairDesc* pd = L.pairs ? L.pairs + pair : &L.single;
    const MapDesc md = L.maps ? L.maps[pd->map] : L.single_map;
    const SrcDesc sd = L.srcs ? L.srcs[pd->src] : L.single_src;
#pragma unroll
    for (int k = 0; k < 9; ++k) ic.R[k] = pd->R[k];
    ic.t[0] = pd->t[0];
    ic.t[1] = pd->t[1];
    ic.t[2] = pd->t[2];
    ic.tmax = pd->tmax;
    ic.inv_r = md.inv_r;
    ic.margin_scale = md.margin_scale;
    ic.mask = *md.vmask;
    ic.vslots = md.vslots;
    ic.pts = sd.pts;
    ic.covs = sd.covs;
    ic.pd = pd;
    ic.r = md.r;
    ic.max_probe = md.max_probe;
  }
  __syncthreads();
  Pose32 P;
#pragma unroll
  for (int k = 0; k < 9; ++k) P.R[k] = uniform(ic.R[k]);
#pragma unroll
  for (int k = 0; k < 3; ++k) P.t[k] = uniform(ic.t[k]);
  P.tmax = uniform(ic.tmax);
  MapDesc md;
  md.inv_r = uniform(ic.inv_r);
  md.margin_scale = uniform(ic.margin_scale);
  md.vslots = uniform(ic.vslots);
  const uint32_t mask = uniform(ic.mask);
  const float* const pts = uniform(ic.pts + 3 * (int64_t)begin);
  const float* const covs = uniform(ic.covs + 6 * (int64_t)begin);
  const int64_t n = end - begin;

  float acc[kAcc];
#pragma unroll
  for (int k = 0; k < kAcc; ++k) acc[k] = 0.0f;

  float next[kPer][9];  // the points of the round to come: mean, covariance
  auto load = [&](int64_t i0) {
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int64_t i = i0 + u * kSimpleThreads;
      if (i < n) {
        const float* pt = pts + 3 * i;
        const float2* cv = reinterpret_cast<const float2*>(covs + 6 * i);
        next[u][0] = __ldg(pt + 0);
        next[u][1] = __ldg(pt + 1);
        next[u][2] = __ldg(pt + 2);
        const float2 c01 = __ldg(cv + 0), c23 = __ldg(cv + 1), c45 = __ldg(cv + 2);
        next[u][3] = c01.x; next[u][4] = c01.y; next[u][5] = c23.x;
        next[u][6] = c23.y; next[u][7] = c45.x; next[u][8] = c45.y;
      }
    }
  };
  load(threadIdx.x);
  for (int64_t i0 = threadIdx.x; i0 < n; i0 += kPer * kSimpleThreads) {
    float s[kPer][9], q[kPer][3];
    uint32_t h[kPer], a[kPer][8], b[kPer][4];
    unsigned long long key[kPer];
    bool live[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
#pragma unroll
      for (int k = 0; k < 9; ++k) s[u][k] = next[u][k];
      live[u] = i0 + u * kSimpleThreads < n;
      if (!live[u]) continue;
      const float x = s[u][0], y = s[u][1], z = s[u][2];
      q[u][0] = fmaf(P.R[0], x, fmaf(P.R[1], y, fmaf(P.R[2], z, P.t[0])));
      q[u][1] = fmaf(P.R[3], x, fmaf(P.R[4], y, fmaf(P.R[5], z, P.t[1])));
      q[u][2] = fmaf(P.R[6], x, fmaf(P.R[7], y, fmaf(P.R[8], z, P.t[2])));
      int kx, ky, kz;
      source_key(P, ic.pd, md_of_item(md, ic.r), x, y, z, q[u][0], q[u][1], q[u][2], kx, ky, kz);
      live[u] = key_in_range(kx) && key_in_range(ky) && key_in_range(kz);
      if (live[u]) {
        key[u] = pack_key(kx, ky, kz);
        h[u] = hash_key(kx, ky, kz) & mask;
        ld_slot(md.vslots + h[u], pol, a[u], b[u]);
      }
    }
    load(i0 + kPer * kSimpleThreads);
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      if (!live[u]) continue;
      unsigned long long t = slot_key(a[u]);
      for (int p = 1; t != key[u] && t != kEmptyKey && (p > 1 || a[u][kSlotSpill] != 0u) &&
                      p < ic.max_probe;
           ++p) {
        h[u] = (h[u] + 1) & mask;
        ld_slot(md.vslots + h[u], pol, a[u], b[u]);
        t = slot_key(a[u]);
      }
      if (t != key[u]) continue;
      float4 r0, r1, r2;
      slot_gaussian(a[u], b[u], r0, r1, r2);
      term<MODE>(acc, P, s[u][0], s[u][1], s[u][2], s[u] + 3, q[u][0], q[u][1], q[u][2], r0, r1, r2);
    }
  }

#pragma unroll
  for (int k = 0; k < kAcc; ++k) {
    float v = acc[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if (lane == 0) red[warp][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < kAcc) {
    double v = 0.0;
    for (int w = 0; w < kSimpleThreads / 32; ++w) v += (double)red[w][threadIdx.x];
    L.partials[(int64_t)it * kPartialStride + threadIdx.x] = v;
  }
}
}  // namespace ahead

// Term `lane` (its sum s) of a linearization to its places in the 43-value result.
__device__ __forceinline__ void write_result(int lane, double s, bool failed, double* o,
                                             int64_t* inliers) {
  constexpr int ww_r[6] = {0, 0, 0, 1, 1, 2}, ww_c[6] = {0, 1, 2, 1, 2, 2};
  if (lane < 6) {
    o[6 * ww_r[lane] + ww_c[lane]] = s;
    o[6 * ww_c[lane] + ww_r[lane]] = s;
  } else if (lane < 15) {
    const int i = (lane - 6) / 3, j = (lane - 6) % 3;
    o[6 * i + 3 + j] = s;
    o[6 * (3 + j) + i] = s;
  } else if (lane < 21) {
    const int k = lane - 15;
    o[6 * (3 + ww_r[k]) + 3 + ww_c[k]] = s;
    o[6 * (3 + ww_c[k]) + 3 + ww_r[k]] = s;
  } else if (lane < 27) {
    o[36 + (lane - 21)] = s;
  } else if (lane == 27) {
    o[42] = s;
  } else if (lane == 28) {
    *inliers = failed ? -1 : (int64_t)llrint(s);
  }
}

// ---------------------------------------------------------------------------
// A small factor on its own (1 neighbour): one cluster of 8 CTAs of 1,024 threads does
// all of vgicp_linearize, four work items per CTA at a time.  The items' sums meet in
// the scratch array behind a cluster barrier and the first CTA adds them up, in the
// order of the reduction kernel: one launch where there were three (status word,
// items, reduction).  The call is bound by the host: 8,192 points 32.5 -> 29.5 us a
// call, of which the GPU works 10.6 -> 9.6 us.
// Pose and descriptors come from the kernel parameters (constant bank).
// ---------------------------------------------------------------------------
namespace factor {
constexpr int kCtas = 8, kGroups = 4, kThreads = kGroups * kSimpleThreads;
constexpr int kMaxItems = 2 * kCtas * kGroups;  // two rounds
constexpr int kWarps = kSimpleThreads / 32;

__global__ void __cluster_dims__(kCtas, 1, 1) __launch_bounds__(kThreads)
    linearize_factor_kernel(const __grid_constant__ LinLaunch L, double* __restrict__ out,
                            int64_t* __restrict__ inliers) {
  __shared__ float red[kGroups][kWarps][kAcc];
  const int lane = threadIdx.x & 31, group = threadIdx.x / kSimpleThreads;
  const int t = threadIdx.x % kSimpleThreads, warp = t >> 5;
  const uint64_t pol = policy_evict_last_l();
  const uint32_t rank = split::cluster_rank();
  Pose32 P;
#pragma unroll
  for (int k = 0; k < 9; ++k) P.R[k] = L.single.R[k];
#pragma unroll
  for (int k = 0; k < 3; ++k) P.t[k] = L.single.t[k];
  P.tmax = L.single.tmax;
  const uint32_t mask = *L.single_map.vmask;
  const int64_t n = L.single_src.n;
  for (int first = (int)rank * kGroups; first < L.n_items; first += kCtas * kGroups) {
    const int it = first + group;
    float acc[kAcc];
#pragma unroll
    for (int k = 0; k < kAcc; ++k) acc[k] = 0.0f;
    const int64_t begin = (int64_t)it * L.item_size, end = min(begin + L.item_size, n);
    for (int64_t p = begin + t; p < end; p += kSimpleThreads) {
      const float* pt = L.single_src.pts + 3 * p;
      const float x = __ldg(pt + 0), y = __ldg(pt + 1), z = __ldg(pt + 2);
      const float2* cv = reinterpret_cast<const float2*>(L.single_src.covs + 6 * p);
      const float2 c01 = __ldg(cv + 0), c23 = __ldg(cv + 1), c45 = __ldg(cv + 2);
      const float c[6] = {c01.x, c01.y, c23.x, c23.y, c45.x, c45.y};
      const float qx = fmaf(P.R[0], x, fmaf(P.R[1], y, fmaf(P.R[2], z, P.t[0])));
      const float qy = fmaf(P.R[3], x, fmaf(P.R[4], y, fmaf(P.R[5], z, P.t[1])));
      const float qz = fmaf(P.R[6], x, fmaf(P.R[7], y, fmaf(P.R[8], z, P.t[2])));
      int kx, ky, kz;
      source_key(P, &L.single, L.single_map, x, y, z, qx, qy, qz, kx, ky, kz);
      float4 r0, r1, r2;
      uint32_t h = 0u;
      if (lookup(L.single_map, mask, kx, ky, kz, pol, h, r0, r1, r2))
        add_term(acc, P, x, y, z, c, qx, qy, qz, r0, r1, r2);
    }
#pragma unroll
    for (int k = 0; k < kAcc; ++k) {
      float v = acc[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
      if (lane == 0) red[group][warp][k] = v;
    }
    __syncthreads();
    if (t < kAcc && it < L.n_items) {
      double s = 0.0;
      for (int w = 0; w < kWarps; ++w) s += (double)red[group][w][t];
      L.partials[(int64_t)it * kPartialStride + t] = s;
    }
    __syncthreads();
  }
  __threadfence();
  split::cluster_sync();  // the sums of every CTA are visible
  if (rank == 0 && threadIdx.x < 32) {
    double s = 0.0;
    if (lane < kAcc)
      for (int it = 0; it < L.n_items; ++it)
        s += __ldcg(L.partials + (int64_t)it * kPartialStride + lane);
    write_result(lane, s, false, out, inliers);
  }
}
}  // namespace factor

// One warp per pair: lane k sums term k over the pair's items in order.  For the
// gradient modes, an optional right Jacobian per pair (jr, 36 doubles, row-major)
// maps the gradient g of the right perturbation to that of the pose increment,
// J_r^T g, and an optional per-pair scale multiplies it (the incoming gradient of
// a reverse-mode pass).
__global__ void reduce_kernel(const double* __restrict__ partials, const int2* __restrict__ span,
                              int32_t n_items_single, int64_t n_pairs,
                              const int32_t* __restrict__ status, double* __restrict__ out,
                              int64_t* __restrict__ inliers, int32_t mode,
                              const double* __restrict__ jr, const double* __restrict__ gscale,
                              int32_t bad) {
  const int64_t pair = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (pair >= n_pairs) return;
  const int32_t a = span ? span[pair].x : 0;
  const int32_t b = span ? span[pair].y : n_items_single;
  double s = 0.0;
  if (lane < kAcc)
    for (int32_t it = a; it < b; ++it) s += partials[(int64_t)it * kPartialStride + lane];
  const bool failed = status && (bad ? *status == bad : *status != 0);
  if (failed) s = __longlong_as_double(0x7FF8000000000000ll);  // NaN
  if (mode == 4) {  // overlap: the inlier count only
    if (lane == 28) inliers[pair] = failed ? -1 : (int64_t)llrint(s);
    return;
  }
  if (mode != 0) {  // gradient (6) and err (1)
    if (jr && mode >= 2) {
      double g[6];
#pragma unroll
      for (int i = 0; i < 6; ++i) g[i] = __shfl_sync(0xFFFFFFFFu, s, i);
      if (lane < 6) {
        const double* J = jr + pair * 36;
        double v = 0.0;
#pragma unroll
        for (int i = 0; i < 6; ++i) v = fma(J[6 * i + lane], g[i], v);
        s = gscale ? v * gscale[pair] : v;
      }
    } else if (gscale && lane < 6 && mode >= 2) {
      s *= gscale[pair];
    }
    if (lane < 7) out[pair * 7 + lane] = s;
    if (lane == 28) inliers[pair] = failed ? -1 : (int64_t)llrint(s);
    return;
  }
  write_result(lane, s, failed, out + pair * 43, inliers + pair);
}

}  // namespace

// One-shot test state for the staged kernel's bounded waits
// (vgicp_test_expire_waits): the tile its producers withhold (+1; 0 = none) and
// the wait limit of that one launch.
std::mutex g_wait_test_mu;
int32_t g_wait_test_tile = 0;
int64_t g_wait_test_ns = 0;

void take_wait_test(LinLaunch& L) {
  std::lock_guard<std::mutex> lock(g_wait_test_mu);
  if (g_wait_test_tile > 0) {
    L.test_withhold_tile = g_wait_test_tile;
    L.wait_limit_ns = g_wait_test_ns;
    g_wait_test_tile = 0;
    g_wait_test_ns = 0;
  }
}

int arm_wait_test(int32_t tile, int64_t limit_ns) {
  if (tile < 0 || limit_ns <= 0 || limit_ns > 2000000000ll)
    return set_error(VGICP_ERR_INVALID_ARG, "tile must be >= 0 and the limit in (0, 2 s]");
  std::lock_guard<std::mutex> lock(g_wait_test_mu);
  g_wait_test_tile = tile + 1;
  g_wait_test_ns = limit_ns;
  return VGICP_OK;
}

int default_item_size() { return 16384; }

int default_variant() { return 1; }

// Work items a single factor is spread over (which fixes the order of its sums, so
// it stays when a kernel's CTAs per SM change).
int single_factor_items() { return device_sm_count() * 3; }

int linearize_grid(int neighbours, int variant, int mode) {
  if (variant == 0) variant = default_variant();
  if (neighbours == 27 || variant == 1 || mode != 0)
    return device_sm_count() * simple_ctas(neighbours, mode);
  if (variant == 3) return device_sm_count() * VGICP_COMPACT_MIN_BLOCKS;
  return device_sm_count() * VGICP_MIN_BLOCKS;
}

// Whether a launch goes to the cluster-per-item kernel: the per-point kernel's
// results (variant 1), at least four points per thread in a full item, and at most
// three items to eight SMs, that is three of its CTAs to an SM.  A plan's execution,
// factors of 16,000 points, cluster per item against the kernel of namespace ahead:
// 40 items 48 / 51 us, 56 items 50 / 51, 76 items 71 / 53, 112 items 100 / 60.
static bool split_items(const LinLaunch& L, int variant) {
  return L.neighbours != 27 && variant == 1 && L.mode <= 3 && L.grid <= 0 && !L.corr_out &&
         !L.qkey_out && L.item_size >= 4 * kSimpleThreads && 8 * L.n_items <= 3 * device_sm_count();
}

// Points per thread of a launch that goes to the kernel of namespace ahead instead of the
// per-point one, or 0: four where every item has an SM of its own, two up to two items
// per SM.  Four against two points: 76 items 53 / 57 us, 152 items 63 / 70.  Above two items
// per SM the items' waves count (350 items: 126 us by the per-point kernel, two waves here),
// and for full grids the per-point kernel's 32 warps per SM hide more.
static int ahead_items(const LinLaunch& L, int variant) {
  if (L.neighbours == 27 || variant != 1 || L.mode > 3 || L.grid > 0 || L.corr_out || L.qkey_out ||
      L.item_size < 4 * kSimpleThreads)
    return 0;
  return L.n_items <= device_sm_count() ? 4 : L.n_items <= 2 * device_sm_count() ? 2 : 0;
}

template <int MODE>
static void launch_ahead(const LinLaunch& L, int per, cudaStream_t st) {
  const unsigned ctas = (unsigned)L.n_items;
  if (per == 4) ahead::linearize_ahead_kernel<MODE, 4><<<ctas, kSimpleThreads, 0, st>>>(L);
  else ahead::linearize_ahead_kernel<MODE, 2><<<ctas, kSimpleThreads, 0, st>>>(L);
}

// Whether a launch needs its status word and work-item counter zeroed: the staged
// kernel's waits and dynamically claimed items do, a CTA per item does not.
bool needs_status(const LinLaunch& L) {
  const int variant = L.mode != 0 ? 1 : (L.variant ? L.variant : default_variant());
  if (L.neighbours != 27 && variant != 1) return true;
  const int grid = L.grid > 0 ? L.grid : linearize_grid(L.neighbours, variant, L.mode);
  return grid < L.n_items;
}

// Up to 64 items of one or two rounds of points each.
bool factor_in_one_launch(const LinLaunch& L) {
  return !L.items && !L.pairs && L.neighbours == 1 && L.mode == 0 && L.variant <= 1 &&
         L.grid <= 0 && !L.corr_out && !L.qkey_out && L.n_items >= 1 &&
         L.n_items <= factor::kMaxItems && L.item_size <= 2 * kSimpleThreads;
}

int launch_factor(const LinLaunch& L, double* out, int64_t* inliers, cudaStream_t st) {
  if (L.ev_start) VGICP_CUDA_TRY(cudaEventRecord(L.ev_start, st));
  factor::linearize_factor_kernel<<<factor::kCtas, factor::kThreads, 0, st>>>(L, out, inliers);
  VGICP_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  if (L.ev_stop) VGICP_CUDA_TRY(cudaEventRecord(L.ev_stop, st));
  return VGICP_OK;
}

int launch_linearize(const LinLaunch& L, cudaStream_t st) {
  if (L.n_items <= 0) return VGICP_OK;
  const int variant = L.mode != 0 ? 1 : (L.variant ? L.variant : default_variant());
  int grid = L.grid > 0 ? L.grid : linearize_grid(L.neighbours, variant, L.mode);
  grid = std::min(grid, L.n_items);
  if (L.ev_start) VGICP_CUDA_TRY(cudaEventRecord(L.ev_start, st));
  LinLaunch Lb = L;
  if (L.neighbours == 27 && L.blocks) {
    // the maps with occupancy blocks, then (below) the items of those without
    const int bgrid = L.grid > 0 ? grid : std::min(device_sm_count() * blocks::kCtas, L.n_items);
    if (L.mode == 0) blocks::linearize_blocks_kernel<0><<<bgrid, kSimpleThreads, 0, st>>>(L);
    else if (L.mode == 1) blocks::linearize_blocks_kernel<1><<<bgrid, kSimpleThreads, 0, st>>>(L);
    else if (L.mode == 2) blocks::linearize_blocks_kernel<2><<<bgrid, kSimpleThreads, 0, st>>>(L);
    else blocks::linearize_blocks_kernel<3><<<bgrid, kSimpleThreads, 0, st>>>(L);
    count_launches(1);
    Lb.status = L.status + 1;  // the second work-item counter
  }
  const int ahead = ahead_items(L, variant);
  if (split_items(L, variant)) {
    const unsigned ctas = (unsigned)L.n_items * split::kCtas;
    if (L.mode == 0) split::linearize_split_kernel<0><<<ctas, split::kThreads, 0, st>>>(L);
    else if (L.mode == 1) split::linearize_split_kernel<1><<<ctas, split::kThreads, 0, st>>>(L);
    else if (L.mode == 2) split::linearize_split_kernel<2><<<ctas, split::kThreads, 0, st>>>(L);
    else split::linearize_split_kernel<3><<<ctas, split::kThreads, 0, st>>>(L);
  } else if (ahead > 0) {
    if (L.mode == 0) launch_ahead<0>(L, ahead, st);
    else if (L.mode == 1) launch_ahead<1>(L, ahead, st);
    else if (L.mode == 2) launch_ahead<2>(L, ahead, st);
    else launch_ahead<3>(L, ahead, st);
  } else if (L.mode != 0) {
    // cost / gradient evaluations use the per-point kernel
    if (L.neighbours == 27) {
      if (L.mode == 1) launch_simple<27, 1>(Lb, grid, st);
      else if (L.mode == 2) launch_simple<27, 2>(Lb, grid, st);
      else launch_simple<27, 3>(Lb, grid, st);
    } else {
      if (L.mode == 1) launch_simple<1, 1>(L, grid, st);
      else if (L.mode == 2) launch_simple<1, 2>(L, grid, st);
      else if (L.mode == 3) launch_simple<1, 3>(L, grid, st);
      else launch_simple<1, 4>(L, grid, st);
    }
  } else if (L.neighbours == 27) {
    launch_simple<27, 0>(Lb, grid, st);
  } else if (variant == 1) {
    launch_simple<1, 0>(L, grid, st);
  } else if (variant == 3 && !L.corr_out && !L.qkey_out) {
    compact::linearize_compact_kernel<<<grid, compact::kThreads, 0, st>>>(L);
  } else if (variant == 3) {
    launch_simple<1, 0>(L, grid, st);  // the per-point kernel writes the debug outputs

  } else {
    // the dynamic shared-memory limit is a per-device function attribute: set it
    // once per device, under a lock (host threads may launch concurrently)
    static std::mutex attr_mu;
    static bool attr_set[kMaxDevices] = {false};
    int dev = 0;
    VGICP_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices)
      return set_error(VGICP_ERR_INVALID_ARG, "device index beyond the supported range");
    {
      std::lock_guard<std::mutex> lock(attr_mu);
      if (!attr_set[dev]) {
        VGICP_CUDA_TRY(cudaFuncSetAttribute(tma::linearize_tma_kernel,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)sizeof(tma::Smem)));
        attr_set[dev] = true;
      }
    }
    LinLaunch Lt = L;
    take_wait_test(Lt);
    tma::linearize_tma_kernel<<<grid, tma::kThreads, sizeof(tma::Smem), st>>>(Lt);
  }
  VGICP_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  if (L.ev_stop) VGICP_CUDA_TRY(cudaEventRecord(L.ev_stop, st));
  return VGICP_OK;
}

int launch_reduce(const double* partials, const int2* span, int32_t n_items_single,
                  int64_t n_pairs, const int32_t* status, double* out, int64_t* inliers,
                  cudaStream_t st, int32_t mode, const double* jr, const double* gscale,
                  int32_t bad) {
  if (n_pairs <= 0) return VGICP_OK;
  const int warps = 8;
  const int64_t blocks = (n_pairs + warps - 1) / warps;
  reduce_kernel<<<(unsigned)blocks, warps * 32, 0, st>>>(partials, span, n_items_single, n_pairs,
                                                         status, out, inliers, mode, jr, gscale,
                                                         bad);
  VGICP_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return VGICP_OK;
}

}  // namespace vgicp
