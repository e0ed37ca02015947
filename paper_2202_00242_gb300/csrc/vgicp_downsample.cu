// Voxel-grid downsampling with timestamp averaging (arXiv 2202.00242 Sec. III-C:
// the input clouds are downsampled by a voxel grid; each voxel averages the
// timestamps of its points as well as their positions, and a point whose time
// lies far from its voxel's is put in another, new voxel so that the first and
// last points of a scan are not fused).
//
// Reading (deterministic): a point's voxel is floor(p / r) (binary64
// semantics); the voxel's reference time is that of its first point in index
// order; a point more than `split` away from it in time goes to the voxel's
// second output voxel.  Output voxels are numbered in order of first
// appearance, cloud by cloud; each holds the mean of its points' positions and
// times, the binary64 mean rounded to float32 (of the double-float sum in index order
// where that is exact, else of the binary64 sum in that order).
//
//   insert   per point: exact key, CAS into the cloud's table, first index
//   group    per point: sub-voxel from the first point's time; first index and
//            count of each (voxel, sub) group
//   mark     first points in a bitmap; places for the groups' point lists
//   scatter  the points of each group, contiguous; beside it, the scan of the
//            bitmap's words (a group's output voxel is the number of first points
//            before its own) and the clouds' output offsets
//   finalize per first point: exact sums of its group's list, means.  Short lists are
//            sorted; a long one is summed by a warp as it comes, and sorted only if its
//            sums round in that order, or if another order's could give another mean
// Six launches, one copy in and one out: a sweep of 60,000 points is bound by their
// latency and the host's (290 -> 215 us a call, of which the kernels take 33 us; before,
// 14 kernels, three fills and five copies, 65 us, and a thread per voxel that sorted
// and summed lists of thousands).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "vgicp.h"
#include "vgicp_device.cuh"
#include "vgicp_internal.h"
#include "vgicp_sort.cuh"

namespace vgicp {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxProbe = 64;
constexpr uint32_t kNone = 0xFFFFFFFFu;

struct __align__(16) DsSlot {
  unsigned long long key;
  uint32_t first;  // smallest point index (global) in the cell
  uint32_t pad;
};

// A (voxel, sub) group: G per slot, G = 2 with a time split, else 1.
struct __align__(16) DsGroup {
  uint32_t first;  // smallest point index
  uint32_t count;
  uint32_t end;    // of its list, once the scatter is done
  uint32_t pad;
};

__device__ __forceinline__ int cloud_of(const int64_t* __restrict__ off, int32_t n, int64_t i) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(off + mid) <= i) lo = mid; else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ void set_status(int32_t* status, int32_t code) {
  atomicCAS(status, 0, code);
}

#define DS_LOOP(i, n)                                                         \
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n); \
       i += (int64_t)gridDim.x * blockDim.x)

__global__ void ds_init_kernel(uint4* slots, int64_t cap, uint4* groups, int64_t n_groups) {
  DS_LOOP(s, n_groups) {
    if (s < cap) slots[s] = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, kNone, 0u);
    groups[s] = make_uint4(kNone, 0u, 0u, 0u);
  }
}

__global__ void ds_insert_kernel(const float* __restrict__ pts, int64_t n,
                                 const int64_t* __restrict__ off, int32_t n_clouds, float inv_r,
                                 double r, const int64_t* __restrict__ base,
                                 const uint32_t* __restrict__ mask, DsSlot* slots,
                                 uint32_t* __restrict__ pt_slot, int32_t* status) {
  DS_LOOP(i, n) {
    const int c = cloud_of(off, n_clouds, i);
    const int kx = axis_key_target(pts[3 * i], inv_r, r);
    const int ky = axis_key_target(pts[3 * i + 1], inv_r, r);
    const int kz = axis_key_target(pts[3 * i + 2], inv_r, r);
    if (!key_in_range(kx) || !key_in_range(ky) || !key_in_range(kz)) {
      pt_slot[i] = kNone;
      set_status(status, VGICP_ERR_KEY_RANGE);
      continue;
    }
    const unsigned long long key = pack_key(kx, ky, kz);
    DsSlot* t = slots + base[c];
    const uint32_t m = mask[c];
    uint32_t h = hash_key(kx, ky, kz) & m;
    uint32_t found = kNone;
    for (int p = 0; p < kMaxProbe; ++p) {
      unsigned long long cur = *reinterpret_cast<volatile unsigned long long*>(&t[h].key);
      if (cur == kEmptyKey) {
        cur = atomicCAS(&t[h].key, kEmptyKey, key);
        if (cur == kEmptyKey) cur = key;
      }
      if (cur == key) {
        found = h;
        break;
      }
      h = (h + 1) & m;
    }
    if (found == kNone) {
      pt_slot[i] = kNone;
      set_status(status, VGICP_ERR_HASH_FULL);
      continue;
    }
    atomicMin(&t[found].first, (uint32_t)i);
    pt_slot[i] = (uint32_t)(base[c] + found);
  }
}

__global__ void ds_group_kernel(int64_t n, const float* __restrict__ times, double split, int G,
                                const DsSlot* __restrict__ slots,
                                const uint32_t* __restrict__ pt_slot, DsGroup* groups,
                                uint32_t* __restrict__ pt_group) {
  DS_LOOP(i, n) {
    const uint32_t s = pt_slot[i];
    if (s == kNone) {
      pt_group[i] = kNone;
      continue;
    }
    uint32_t g = s;
    if (G == 2) {
      const double t0 = (double)times[slots[s].first];
      g = 2u * s + (fabs((double)times[i] - t0) > split ? 1u : 0u);
    }
    atomicMin(&groups[g].first, (uint32_t)i);
    atomicAdd(&groups[g].count, 1u);
    pt_group[i] = g;
  }
}

// CTAs [0, n_mark): first points, one bit each (n_words words, the last one holds
// point n's).  The others: places of the groups' lists, a range per CTA and the
// groups' own inside it (the order of the lists does not matter).
constexpr int kPlacePer = 4;
__global__ void __launch_bounds__(kThreads) ds_mark_kernel(int64_t n, int64_t n_words, int n_mark,
                                                           const uint32_t* __restrict__ pt_group,
                                                           DsGroup* groups, int64_t n_groups,
                                                           uint32_t* __restrict__ bitmap,
                                                           uint32_t* cursor) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if ((int)blockIdx.x < n_mark) {
    const int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x;
    bool f = false;
    if (i < n) {
      const uint32_t g = pt_group[i];
      f = g != kNone && groups[g].first == (uint32_t)i;
    }
    const uint32_t b = __ballot_sync(0xFFFFFFFFu, f);
    if (lane == 0 && (i >> 5) < n_words) bitmap[i >> 5] = b;
    return;
  }
  __shared__ uint32_t warp_sum[kThreads / 32];
  __shared__ uint32_t base;
  const int64_t g0 = ((int64_t)blockIdx.x - n_mark) * (kThreads * kPlacePer) + threadIdx.x;
  uint32_t cnt[kPlacePer], sum = 0u;
#pragma unroll
  for (int j = 0; j < kPlacePer; ++j) {
    const int64_t g = g0 + (int64_t)j * kThreads;
    cnt[j] = g < n_groups ? groups[g].count : 0u;
    sum += cnt[j];
  }
  uint32_t inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) warp_sum[w] = inc;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0u;
    for (int k = 0; k < kThreads / 32; ++k) {
      const uint32_t x = warp_sum[k];
      warp_sum[k] = t;
      t += x;
    }
    base = t > 0u ? atomicAdd(cursor, t) : 0u;
  }
  __syncthreads();
  uint32_t run = base + warp_sum[w] + inc - sum;
#pragma unroll
  for (int j = 0; j < kPlacePer; ++j) {
    if (cnt[j] > 0u) groups[g0 + (int64_t)j * kThreads].end = run;  // the list's start, for now
    run += cnt[j];
  }
}

__device__ __forceinline__ uint32_t rank_of(const uint32_t* __restrict__ bitmap,
                                            const uint32_t* __restrict__ wscan, int64_t i) {
  return wscan[i >> 5] + (uint32_t)__popc(bitmap[i >> 5] & ((1u << (i & 31)) - 1u));
}

__device__ __forceinline__ void scatter_point(int64_t i, const uint32_t* __restrict__ pt_group,
                                              DsGroup* groups, uint32_t* __restrict__ list) {
  const uint32_t g = pt_group[i];
  if (g != kNone) list[atomicAdd(&groups[g].end, 1u)] = (uint32_t)i;
}

// CTA 0 scans the words' popcounts and writes the clouds' output offsets (and the
// status word behind them); the others scatter the points.  For up to kScanWords
// words, which one CTA scans while the others work.
constexpr int64_t kScanWords = 16384;
__global__ void __launch_bounds__(kThreads) ds_scatter_kernel(
    int64_t n, const uint32_t* __restrict__ pt_group, DsGroup* groups, uint32_t* __restrict__ list,
    int64_t n_words, const uint32_t* __restrict__ bitmap, uint32_t* __restrict__ wscan,
    int32_t n_clouds, const int64_t* __restrict__ off, const int32_t* __restrict__ status,
    uint32_t* __restrict__ oo) {
  if (blockIdx.x > 0) {
    const int64_t i = ((int64_t)blockIdx.x - 1) * kThreads + threadIdx.x;
    if (i < n) scatter_point(i, pt_group, groups, list);
    return;
  }
  constexpr int kPer = 8;
  __shared__ uint32_t warp_sum[kThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t carry = 0u;
  for (int64_t w0 = 0; w0 < n_words; w0 += kThreads * kPer) {
    const int64_t a = w0 + (int64_t)threadIdx.x * kPer;
    uint32_t c[kPer], sum = 0u;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      c[k] = a + k < n_words ? (uint32_t)__popc(bitmap[a + k]) : 0u;
      sum += c[k];
    }
    uint32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) warp_sum[w] = inc;
    __syncthreads();
    uint32_t run = carry + inc - sum;
    for (int k = 0; k < kThreads / 32; ++k) {
      const uint32_t x = warp_sum[k];
      if (k < w) run += x;
      carry += x;
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      if (a + k < n_words) wscan[a + k] = run;
      run += c[k];
    }
    __syncthreads();  // also: this CTA's words are visible to it below
  }
  for (int c = threadIdx.x; c <= n_clouds; c += kThreads) oo[c] = rank_of(bitmap, wscan, off[c]);
  if (threadIdx.x == 0) oo[n_clouds + 1] = (uint32_t)*status;
}

// The same steps apart, for more words.
__global__ void ds_popc_kernel(int64_t n_words, const uint32_t* __restrict__ bitmap,
                               uint32_t* __restrict__ out) {
  DS_LOOP(w, n_words) out[w] = (uint32_t)__popc(bitmap[w]);
}
__global__ void ds_scatter_large_kernel(int64_t n, const uint32_t* __restrict__ pt_group,
                                        DsGroup* groups, uint32_t* __restrict__ list,
                                        const uint32_t* __restrict__ bitmap,
                                        const uint32_t* __restrict__ wscan, int32_t n_clouds,
                                        const int64_t* __restrict__ off,
                                        const int32_t* __restrict__ status,
                                        uint32_t* __restrict__ oo) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) scatter_point(i, pt_group, groups, list);
  if (i <= n_clouds) oo[i] = rank_of(bitmap, wscan, off[i]);
  if (i == 0) oo[n_clouds + 1] = (uint32_t)*status;
}

// (hi, lo) += the same of the lane at distance `delta`, exactly (checked).
__device__ __forceinline__ void ds_add_lane(float* hi, float* lo, bool& exact, int delta) {
  const bool other = __shfl_xor_sync(0xFFFFFFFFu, (int)exact, delta) != 0;
  exact = exact && other;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float h = __shfl_xor_sync(0xFFFFFFFFu, hi[k], delta);
    const float l = __shfl_xor_sync(0xFFFFFFFFu, lo[k], delta);
    float t, e, u, e2, v, e3;
    two_sum(hi[k], h, t, e);
    two_sum(lo[k], l, u, e2);
    two_sum(u, e, v, e3);
    exact = exact && e2 == 0.0f && e3 == 0.0f;
    two_sum(t, v, hi[k], lo[k]);
  }
}

// Whether every value within `error` of s has the mean q = RN32(s / n) (m: s / n in
// binary64): the distance of m to the ends of what rounds to q, in float32.
__device__ __forceinline__ bool mean_is_certain(double m, float q, float error_of_mean) {
  const uint32_t b = __float_as_uint(q) & 0x7FFFFFFFu;
  if (b < (27u << 23) || b >= 0x7F800000u) return false;
  const float spacing = __uint_as_float((b & 0x7F800000u) - (23u << 23));
  const float half = (b & 0x007FFFFFu) ? 0.5f * spacing : 0.25f * spacing;  // a power of two: below
  const float off = fabsf((float)(m - (double)q));
  return half - off > error_of_mean + 0x1p-22f * spacing;
}

// Whether c values have the same binary64 sum in every order, an exact one: every partial
// sum is a multiple of the last bit of the smallest above zero (as bits, less one), and
// below 2^53 of them.
__device__ __forceinline__ bool any_order(uint32_t c, float largest, uint32_t smallest) {
  if (largest == 0.f) return true;
  const int top = max((int)(__float_as_uint(largest) >> 23), 1);
  const int low = max((int)((smallest + 1u) >> 23), 1);
  return top < 255 && top - low + 32 - __clz((int)(c - 1u)) <= 29;
}

// One lane per point; the lanes of first points take their group's list, lists
// longer than kSerial the whole warp.  Lists are in the order in which their points came,
// so what depends on the order of a sum must not reach the output.  A sum in double-float
// that is exact in this order is the true one; the sum in index order, exact or in
// binary64, is within c^2 max |v| 2^-53 of it, and nearly always has the same mean.
// The kernel, sweeps of 60,000 points at 0.25 / 1.0 m: 16 / 30 us, of 250,000: 42 / 92;
// with every sum taken in the order of its list 17 / 34 and 37 / 110; with the smallest
// magnitude of every long list taken along with its sums 15 / 37 and 44 / 123.
constexpr uint32_t kSerial = 8;  // as many as the sorting network takes
__global__ void __launch_bounds__(kThreads) ds_finalize_kernel(
    int64_t n, const uint32_t* __restrict__ bitmap, const uint32_t* __restrict__ wscan,
    const uint32_t* __restrict__ pt_group, const DsGroup* __restrict__ groups,
    const float* __restrict__ pts, const float* __restrict__ times, uint32_t* __restrict__ list,
    float* __restrict__ out_pts, float* __restrict__ out_times, int32_t* __restrict__ out_counts) {
  const int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool mine = i < n && ((bitmap[i >> 5] >> (i & 31)) & 1u);
  uint32_t c = 0u, at = 0u;
  if (mine) {
    const uint4 g = *reinterpret_cast<const uint4*>(groups + pt_group[i]);
    c = g.y;
    at = g.z - g.y;
  }
  float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
  float largest[4] = {0.f, 0.f, 0.f, 0.f};
  bool exact = true;
  for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, c > kSerial); todo; todo &= todo - 1u) {
    const int b = __ffs(todo) - 1;
    const uint32_t ab = __shfl_sync(0xFFFFFFFFu, at, b), cb = __shfl_sync(0xFFFFFFFFu, c, b);
    float h[4] = {0.f, 0.f, 0.f, 0.f}, l[4] = {0.f, 0.f, 0.f, 0.f}, g[4] = {0.f, 0.f, 0.f, 0.f};
    bool ex = true;
    for (uint32_t a = lane; a < cb; a += 32) {
      const int64_t j = list[ab + a];
      const float f[4] = {pts[3 * j], pts[3 * j + 1], pts[3 * j + 2], times ? times[j] : 0.f};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (k == 3 && !times) break;
        df_add(h[k], l[k], f[k], ex);
        g[k] = fmaxf(g[k], fabsf(f[k]));
      }
    }
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) ds_add_lane(h, l, ex, d);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t m = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(g[k]));
      if (lane == b) {
        hi[k] = h[k];
        lo[k] = l[k];
        largest[k] = __uint_as_float(m);
      }
    }
    if (lane == b) exact = ex;
  }
  // A long list's mean is certain if no sum within the error rounds to another, or (the
  // quotient on a midpoint, mostly) if every order has the same sum.
  const double N = (double)c, y = __drcp_rn(N);
  float mean[4];
  bool certain = exact && c > kSerial, same_mean = certain;
  if (certain) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double m = div_rn(__dadd_rn((double)hi[k], (double)lo[k]), N, y);
      mean[k] = __double2float_rn(m);
      same_mean = same_mean && (largest[k] == 0.f ||
                                mean_is_certain(m, mean[k], (float)c * largest[k] * 0x1p-52f));
    }
  }
  for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, certain && !same_mean); todo; todo &= todo - 1u) {
    const int b = __ffs(todo) - 1;
    const uint32_t ab = __shfl_sync(0xFFFFFFFFu, at, b), cb = __shfl_sync(0xFFFFFFFFu, c, b);
    uint32_t smallest[4] = {kNone, kNone, kNone, kNone};  // above zero, as bits less one
    for (uint32_t a = lane; a < cb; a += 32) {
      const int64_t j = list[ab + a];
      const float f[4] = {pts[3 * j], pts[3 * j + 1], pts[3 * j + 2], times ? times[j] : 0.f};
#pragma unroll
      for (int k = 0; k < 4; ++k)
        smallest[k] = min(smallest[k], (__float_as_uint(f[k]) & 0x7FFFFFFFu) - 1u);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t m = __reduce_min_sync(0xFFFFFFFFu, smallest[k]);
      if (lane == b) certain = certain && any_order(c, largest[k], m);
    }
  }
  if (!mine) return;
  if (!certain) {  // in ascending point index
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    exact = true;
#pragma unroll
    for (int k = 0; k < 4; ++k) hi[k] = lo[k] = 0.f;
    auto add_exact = [&](int64_t j) {
#pragma unroll
      for (int k = 0; k < 3; ++k) df_add(hi[k], lo[k], pts[3 * j + k], exact);
      if (times) df_add(hi[3], lo[3], times[j], exact);
    };
    auto add_64 = [&](int64_t j) {
#pragma unroll
      for (int k = 0; k < 3; ++k) s[k] = __dadd_rn(s[k], (double)pts[3 * j + k]);
      if (times) s[3] = __dadd_rn(s[3], (double)times[j]);
    };
    if (c <= kSerial) {
      uint32_t e[kSerial];
#pragma unroll
      for (int a = 0; a < (int)kSerial; ++a) e[a] = a < (int)c ? list[at + a] : kNone;
      // odd-even merge network
      constexpr int kPairs[19][2] = {{0, 1}, {2, 3}, {4, 5}, {6, 7}, {0, 2}, {1, 3}, {4, 6},
                                     {5, 7}, {1, 2}, {5, 6}, {0, 4}, {1, 5}, {2, 6}, {3, 7},
                                     {2, 4}, {3, 5}, {1, 2}, {3, 4}, {5, 6}};
#pragma unroll
      for (int q = 0; q < 19; ++q) {
        uint32_t &l = e[kPairs[q][0]], &h = e[kPairs[q][1]];
        const uint32_t low = min(l, h);
        h = max(l, h);
        l = low;
      }
#pragma unroll
      for (int a = 0; a < (int)kSerial; ++a)
        if (a < (int)c) add_exact(e[a]);
      if (!exact)
#pragma unroll
        for (int a = 0; a < (int)kSerial; ++a)
          if (a < (int)c) add_64(e[a]);
    } else {
      uint32_t* L = list + at;
      sort_list(L, c);
      for (uint32_t a = 0; a < c; ++a) add_exact(L[a]);
      if (!exact)
        for (uint32_t a = 0; a < c; ++a) add_64(L[a]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (exact) s[k] = __dadd_rn((double)hi[k], (double)lo[k]);
      mean[k] = __double2float_rn(div_rn(s[k], N, y));
    }
  }
  const int64_t v = rank_of(bitmap, wscan, i);
#pragma unroll
  for (int k = 0; k < 3; ++k) out_pts[3 * v + k] = mean[k];
  if (out_times) out_times[v] = mean[3];
  if (out_counts) out_counts[v] = (int32_t)c;
}

int grid_of(int64_t n) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + kThreads - 1) / kThreads, 0x7FFFFFFF));
}

}  // namespace
}  // namespace vgicp

extern "C" {

int vgicp_downsample(const float* points, const float* times, const int64_t* offsets,
                     int32_t n_clouds, double resolution, double split, float* out_points,
                     float* out_times, int32_t* out_counts, int64_t* out_offsets,
                     vgicp_stream_t stream) {
  using namespace vgicp;
  if (!(resolution > 0.0) || !std::isfinite(resolution))
    return set_error(VGICP_ERR_INVALID_ARG, "resolution must be positive and finite");
  if (n_clouds <= 0 || !offsets || !out_offsets)
    return set_error(VGICP_ERR_INVALID_ARG, "n_clouds >= 1, offsets and out_offsets required");
  if (offsets[0] != 0) return set_error(VGICP_ERR_INVALID_ARG, "offsets[0] must be 0");
  for (int32_t c = 0; c < n_clouds; ++c)
    if (offsets[c + 1] < offsets[c])
      return set_error(VGICP_ERR_INVALID_ARG, "offsets must be non-decreasing");
  if (!std::isfinite(split)) return set_error(VGICP_ERR_INVALID_ARG, "split must be finite");
  const int64_t n = offsets[n_clouds];
  if (n >= (int64_t)0xFFFFFFFFll) return set_error(VGICP_ERR_INVALID_ARG, "more than 2^32-1 points");
  if (n == 0) {
    for (int32_t c = 0; c <= n_clouds; ++c) out_offsets[c] = 0;
    return VGICP_OK;
  }
  if (!points || !out_points) return set_error(VGICP_ERR_INVALID_ARG, "null points");
  std::vector<int64_t> base((size_t)n_clouds);
  std::vector<uint32_t> mask((size_t)n_clouds);
  int64_t cap = 0;
  for (int32_t c = 0; c < n_clouds; ++c) {
    uint64_t k = 16;
    while (k < 2ull * (uint64_t)std::max<int64_t>(offsets[c + 1] - offsets[c], 1)) k <<= 1;
    base[(size_t)c] = cap;
    mask[(size_t)c] = (uint32_t)(k - 1);
    cap += (int64_t)k;
  }
  if (2 * cap >= (int64_t)0xFFFFFFFFll)
    return set_error(VGICP_ERR_INVALID_ARG, "more than 2^31-1 table slots");
  // one buffer; its front is filled by the host in one copy: offsets, tables, and the
  // zeroed counters
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = (off + std::max<size_t>(bytes, 1) + 255) & ~size_t(255);
    return o;
  };
  const int G = times && split > 0.0 ? 2 : 1;
  const int64_t n_groups = cap * G, n_words = n / 32 + 1;
  const size_t o_off = take(sizeof(int64_t) * (n_clouds + 1));
  const size_t o_base = take(sizeof(int64_t) * n_clouds);
  const size_t o_mask = take(sizeof(uint32_t) * n_clouds);
  const size_t o_cursor = take(sizeof(uint32_t));
  const size_t o_status = take(sizeof(int32_t));
  const size_t upload = off;
  const size_t o_oo = take(sizeof(uint32_t) * (n_clouds + 2));
  const size_t o_slots = take(sizeof(DsSlot) * cap);
  const size_t o_groups = take(sizeof(DsGroup) * n_groups);
  const size_t o_ptslot = take(sizeof(uint32_t) * n);
  const size_t o_ptgroup = take(sizeof(uint32_t) * n);
  const size_t o_list = take(sizeof(uint32_t) * n);
  const size_t o_bitmap = take(sizeof(uint32_t) * n_words);
  const size_t o_wscan = take(sizeof(uint32_t) * n_words);
  const size_t o_scan = take(sizeof(uint32_t) * scan_tmp_elems(n_words));
  std::vector<char> host(upload, 0);
  std::memcpy(host.data() + o_off, offsets, sizeof(int64_t) * (n_clouds + 1));
  std::memcpy(host.data() + o_base, base.data(), sizeof(int64_t) * n_clouds);
  std::memcpy(host.data() + o_mask, mask.data(), sizeof(uint32_t) * n_clouds);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  char* d = nullptr;
  VGICP_CUDA_TRY(device_malloc(reinterpret_cast<void**>(&d), off, st, true));
  auto U = [&](size_t o) { return reinterpret_cast<uint32_t*>(d + o); };
  int64_t* d_off = reinterpret_cast<int64_t*>(d + o_off);
  int64_t* d_base = reinterpret_cast<int64_t*>(d + o_base);
  int32_t* d_status = reinterpret_cast<int32_t*>(d + o_status);
  DsSlot* d_slots = reinterpret_cast<DsSlot*>(d + o_slots);
  DsGroup* d_groups = reinterpret_cast<DsGroup*>(d + o_groups);
  int rc = VGICP_OK;
  // (a copy from pageable memory returns once the source is staged)
  cudaError_t e = cudaMemcpyAsync(d, host.data(), upload, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) rc = check_cuda(e, "downsample setup");
  const float inv_r = (float)(1.0 / resolution);
  const int g = grid_of(n);
  const bool fused = n_words <= kScanWords;
  if (rc == VGICP_OK) {
    ds_init_kernel<<<grid_of(n_groups), kThreads, 0, st>>>(reinterpret_cast<uint4*>(d_slots), cap,
                                                          reinterpret_cast<uint4*>(d_groups),
                                                          n_groups);
    ds_insert_kernel<<<g, kThreads, 0, st>>>(points, n, d_off, n_clouds, inv_r, resolution,
                                             d_base, U(o_mask), d_slots, U(o_ptslot), d_status);
    ds_group_kernel<<<g, kThreads, 0, st>>>(n, times, split, G, d_slots, U(o_ptslot), d_groups,
                                            U(o_ptgroup));
    const int n_mark = grid_of(n_words * 32);
    const int n_place = grid_of((n_groups + kPlacePer - 1) / kPlacePer);
    ds_mark_kernel<<<n_mark + n_place, kThreads, 0, st>>>(n, n_words, n_mark, U(o_ptgroup),
                                                         d_groups, n_groups, U(o_bitmap),
                                                         U(o_cursor));
    count_launches(4);
    if (fused) {
      ds_scatter_kernel<<<g + 1, kThreads, 0, st>>>(n, U(o_ptgroup), d_groups, U(o_list), n_words,
                                                   U(o_bitmap), U(o_wscan), n_clouds, d_off,
                                                   d_status, U(o_oo));
      count_launches(1);
    } else {
      ds_popc_kernel<<<grid_of(n_words), kThreads, 0, st>>>(n_words, U(o_bitmap), U(o_wscan));
      rc = launch_exclusive_scan(U(o_wscan), U(o_wscan), n_words, nullptr, U(o_scan), nullptr, st);
      ds_scatter_large_kernel<<<grid_of(std::max<int64_t>(n, n_clouds + 1)), kThreads, 0, st>>>(
          n, U(o_ptgroup), d_groups, U(o_list), U(o_bitmap), U(o_wscan), n_clouds, d_off, d_status,
          U(o_oo));
      count_launches(2);
    }
  }
  if (rc == VGICP_OK) {
    ds_finalize_kernel<<<g, kThreads, 0, st>>>(n, U(o_bitmap), U(o_wscan), U(o_ptgroup), d_groups,
                                               points, times, U(o_list), out_points, out_times,
                                               out_counts);
    count_launches(1);
    e = cudaGetLastError();
    if (e != cudaSuccess) rc = check_cuda(e, "downsample kernels");
  }
  std::vector<uint32_t> oo((size_t)n_clouds + 2, 0u);  // the offsets, then the status
  if (rc == VGICP_OK) {
    e = cudaMemcpyAsync(oo.data(), U(o_oo), sizeof(uint32_t) * oo.size(), cudaMemcpyDeviceToHost,
                        st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) rc = check_cuda(e, "downsample results");
  }
  const int32_t status = (int32_t)oo[(size_t)n_clouds + 1];
  e = cudaFreeAsync(d, st);
  if (rc == VGICP_OK && e != cudaSuccess) rc = check_cuda(e, "cudaFreeAsync");
  if (rc == VGICP_OK && status == VGICP_ERR_KEY_RANGE)
    return set_error(status, "a point's voxel key is outside [-2^20, 2^20)");
  if (rc == VGICP_OK && status == VGICP_ERR_HASH_FULL)
    return set_error(status, "voxel table probe limit exceeded");
  if (rc == VGICP_OK)
    for (int32_t c = 0; c <= n_clouds; ++c) out_offsets[c] = oo[(size_t)c];
  return rc;
}

}  // extern "C"
