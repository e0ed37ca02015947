// Voxel-map build kernels (arXiv 2202.00242 Sec. III-A: the target cloud is
// discretised into voxels; each voxel aggregates the means and covariances of
// its points).
//
// Pipeline for a batch of maps built from concatenated clouds (one launch per
// step for the whole batch):
//   reset     table slots <- empty: every slot on the first build; afterwards
//             the lookup-table slots the previous build's voxels occupy, by CTAs
//             of the insertion (the build table is left empty by the scatter)
//   insert    per point: exact key, open-addressing insert (CAS on the 64-bit
//             key, bounded linear probe), count, smallest point index
//   number    first points (the smallest index of their voxel) marked in a
//             bitmap; voxel id = number of first points before the voxel's
//             (a scan of the words' popcounts), so voxels are numbered in order
//             of first appearance, map by map; each first point gives its voxel
//             its count, key and, in the slot, its id
//             (and per map: lookup-table capacity from the voxel count)
//   sort      per map chunk: the voxels in Morton order of their keys (rank), and
//             the offsets of their point lists, in rank order and by voxel (for
//             maps of many chunks after a kernel that counts the chunks' points)
//   scatter   per point: append its index to its voxel's list; the voxel's
//             last point empties its build-table slot (a point without a voxel is
//             marked behind its map's last list)
//   finalize  per voxel, in rank order: sort its list, sum means and
//             covariances (exactly, else in binary64 in ascending point index),
//             divide by N, round to float32; copy the points into the voxel-
//             grouped cloud (the lists laid end to end); insert the voxel into
//             its map's lookup table (inline records)
// The result is deterministic and bit-identical to the binary64 definition
// rounded once to float32.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>
#include <string>
#include <vector>

#include "vgicp_device.cuh"
#include "vgicp_internal.h"
#include "vgicp_mean.h"
#include "vgicp_sort.cuh"

namespace vgicp {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ int find_map(const int64_t* __restrict__ off, int32_t n_maps,
                                        int64_t i) {
  // last m with off[m] <= i (empty maps are skipped)
  int lo = 0, hi = n_maps;  // answer in [lo, hi)
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (__ldg(off + mid) <= i) lo = mid; else hi = mid;
  }
  return lo;
}

// find_map for the points of one warp, which are consecutive: the first active
// lane searches, the others walk forward from its map (a warp spans few maps).
__device__ __forceinline__ int find_map_warp(const int64_t* __restrict__ off, int32_t n_maps,
                                             int64_t i) {
  const unsigned am = __activemask();
  const int leader = __ffs(am) - 1;
  int m = ((int)(threadIdx.x & 31) == leader) ? find_map(off, n_maps, i) : 0;
  m = __shfl_sync(am, m, leader);
  while (m + 1 < n_maps && __ldg(off + m + 1) <= i) ++m;
  return m;
}

__device__ __forceinline__ void set_status(int32_t* status, int32_t code) {
  atomicCAS(status, 0, code);
}

// The status of the insertion becomes the build's; its own word is ready for the next.
__device__ __forceinline__ void take_status(int32_t* status) {
  status[0] = status[1];
  status[1] = 0;
}

__global__ void init_slots_kernel(Slot* __restrict__ slots, int64_t cap_total, int32_t* status) {
  if (blockIdx.x == 0 && threadIdx.x < 2) status[threadIdx.x] = 0;
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < cap_total;
       s += (int64_t)gridDim.x * blockDim.x) {
    Slot e;
    e.key = kEmptyKey;
    e.vid = 0xFFFFFFFFu;
    e.count = 0u;
    slots[s] = e;
  }
}

// Rebuild: empty the lookup-table slots the previous build's voxels occupy
// (every slot a build claims belongs to one of its voxels, and spill flags are
// set only on claimed slots), which leaves the tables empty.  (The build table
// is emptied by the scatter of every build.)
__device__ void reset_lookup(int cta, int ctas, int64_t n_max, const uint32_t* __restrict__ n_vox,
                             const uint32_t* __restrict__ lslot_of, VSlot* vslots) {
  const int64_t V = *n_vox;
  for (int64_t v = cta * (int64_t)blockDim.x + threadIdx.x; v < V && v < n_max;
       v += (int64_t)ctas * blockDim.x) {
    const uint32_t ls = lslot_of[v];
    if (ls != kNoSlot)
      asm volatile("st.global.v8.b32 [%0], {%1, %1, %2, %2, %2, %2, %2, %2};" ::"l"(vslots + ls),
                   "r"(0xFFFFFFFFu), "r"(0u)
                   : "memory");
  }
}

// One CTA in kResetEvery empties lookup slots on a rebuild (a first build passes no CTAs
// for it): the lookup tables are next written by finalize, and the previous build's
// voxel count by the numbering, so the reset needs no launch of its own.  Ten maps of
// 20,000 points rebuilt and ten factors, r 0.25 / 1.0: 118.8 / 104.8 us with a reset
// kernel, 115.8 / 101.5 so; three maps of 3,000 points 84.7 / 80.2; 500 submaps (25.8M
// points): insert 598 us with the reset inside, 494 + 114 apart.
// Errors go to the second status word, which the numbering moves to the first.
constexpr int kResetEvery = 9;
__global__ void insert_kernel(const float* __restrict__ pts, int64_t n_total,
                              const int64_t* __restrict__ point_off, int32_t n_maps,
                              const int64_t* __restrict__ slot_base,
                              const uint32_t* __restrict__ cap_mask, float inv_r, double r,
                              int32_t max_probe, Slot* slots, uint32_t* __restrict__ pt_slot,
                              int32_t* status, int reset_ctas, const uint32_t* __restrict__ n_vox,
                              const uint32_t* __restrict__ lslot_of, VSlot* vslots) {
  int cta = blockIdx.x;
  const int ctas = gridDim.x - reset_ctas;
  if (reset_ctas > 0) {
    const int k = cta / kResetEvery;
    if (cta % kResetEvery == 0 && k < reset_ctas) {
      reset_lookup(k, reset_ctas, n_total, n_vox, lslot_of, vslots);
      return;
    }
    cta -= min(k + 1, reset_ctas);
  }
  for (int64_t i = cta * (int64_t)blockDim.x + threadIdx.x; i < n_total;
       i += (int64_t)ctas * blockDim.x) {
    const int m = find_map_warp(point_off, n_maps, i);
    const int kx = axis_key_target(__ldg(pts + 3 * i + 0), inv_r, r);
    const int ky = axis_key_target(__ldg(pts + 3 * i + 1), inv_r, r);
    const int kz = axis_key_target(__ldg(pts + 3 * i + 2), inv_r, r);
    if (!key_in_range(kx) || !key_in_range(ky) || !key_in_range(kz)) {
      pt_slot[i] = kNoSlot;
      set_status(status, VGICP_ERR_KEY_RANGE);
      continue;
    }
    const unsigned long long key = pack_key(kx, ky, kz);
    const uint32_t mask = __ldg(cap_mask + m);
    const int64_t base = __ldg(slot_base + m);
    uint32_t h = hash_key(kx, ky, kz) & mask;
    uint32_t found = kNoSlot;
    for (int p = 0; p < max_probe; ++p) {
      // one round trip: the CAS either claims an empty slot or returns its key
      const unsigned long long cur = atomicCAS(&slots[base + h].key, kEmptyKey, key);
      if (cur == kEmptyKey || cur == key) {
        found = (uint32_t)(base + h);
        break;
      }
      h = (h + 1) & mask;
    }
    if (found == kNoSlot) {
      pt_slot[i] = kNoSlot;
      set_status(status, VGICP_ERR_HASH_FULL);
      continue;
    }
    atomicAdd(&slots[found].count, 1u);
    atomicMin(&slots[found].vid, (uint32_t)i);
    pt_slot[i] = found;
  }
}


// Per point: append its index to its voxel's list.  The voxel's last point
// (the one whose fill count reaches the voxel's count; every other point of the
// voxel has read the slot before its own increment) empties the build-table
// slot, whose sector it has just read: the build table is empty again when the
// scatter ends, ready for the next build.
// A point without a voxel (outside the key range, which the build reports) is in no list:
// it leaves kNoSlot at the end of its map's range of plist, behind the map's last list.
__global__ void scatter_kernel(int64_t n_total, const uint32_t* __restrict__ pt_slot, Slot* slots,
                               unsigned long long* bfill, uint32_t* __restrict__ plist,
                               const int64_t* __restrict__ point_off, int32_t n_maps,
                               uint32_t* dropped) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t s = pt_slot[i];
    if (s == kNoSlot) {
      const int m = find_map(point_off, n_maps, i);
      plist[point_off[m + 1] - 1 - (int64_t)atomicAdd(dropped + m, 1u)] = kNoSlot;
      continue;
    }
    // one read of the slot: voxel id and count
    const uint4 w = *reinterpret_cast<const uint4*>(slots + s);
    const uint32_t v = w.z, c = w.w;
    // (list base << 32 | fill): one atomic gives the point its place
    const unsigned long long bf = atomicAdd(bfill + v, 1ull);
    const uint32_t f = (uint32_t)bf;
    plist[(uint32_t)(bf >> 32) + f] = (uint32_t)i;
    if (f + 1u == c) {
      Slot e;
      e.key = kEmptyKey;
      e.vid = 0xFFFFFFFFu;
      e.count = 0u;
      slots[s] = e;
    }
  }
}

// Inserts voxel v (its key, count, mean and the Cholesky factor of its
// covariance) into its map's lookup table: linear probing from the key's home
// slot, claiming a slot with a CAS on the key; a key placed past its home sets
// the home slot's spill flag.  lslot_of[v] records the slot (kNoSlot if the
// probe limit was reached, which is reported as VGICP_ERR_HASH_FULL).
// lo: the voxel's map.
__device__ __forceinline__ void insert_lookup(uint32_t v, unsigned long long key, uint32_t c,
                                              const float* q, int lo,
                                              const int64_t* __restrict__ slot_base,
                                              const uint32_t* __restrict__ vmask,
                                              int32_t max_probe, VSlot* vslots,
                                              uint32_t* __restrict__ lslot_of, int32_t* status) {
  const unsigned long long fm = (1ull << kKeyBits) - 1ull;
  const int kx = (int)((key >> (2 * kKeyBits)) & fm) - kKeyBias;
  const int ky = (int)((key >> kKeyBits) & fm) - kKeyBias;
  const int kz = (int)(key & fm) - kKeyBias;
  // the Cholesky factor L of C' (the linearization forms R^T C' R as (R^T L)(R^T L)^T);
  // a non-positive pivot (a semi-definite C') leaves its column zero
  const float l00 = q[3] > 0.f ? sqrtf(q[3]) : 0.f;
  const float il0 = l00 > 0.f ? 1.0f / l00 : 0.f;
  const float l10 = q[4] * il0, l20 = q[5] * il0;
  const float p11 = q[6] - l10 * l10;
  const float l11 = p11 > 0.f ? sqrtf(p11) : 0.f;
  const float l21 = l11 > 0.f ? (q[7] - l20 * l10) / l11 : 0.f;
  const float p22 = q[8] - l20 * l20 - l21 * l21;
  const float l22 = p22 > 0.f ? sqrtf(p22) : 0.f;
  const uint32_t mask = vmask[lo];
  VSlot* t = vslots + slot_base[lo];
  const uint32_t home = hash_key(kx, ky, kz) & mask;
  uint32_t h = home;
  bool placed = false;
  for (int p = 0; p < max_probe; ++p) {
    if (atomicCAS(&t[h].key, kEmptyKey, key) == kEmptyKey) {
      placed = true;
      break;
    }
    h = (h + 1) & mask;
  }
  if (placed && h != home) atomicOr(&t[home].spill, 1u);
  lslot_of[v] = placed ? (uint32_t)(slot_base[lo] + h) : kNoSlot;
  if (!placed) {
    set_status(status, VGICP_ERR_HASH_FULL);
    return;
  }
  // the slot (key and spill aside) in three stores, the second sector in one: as words
  // finalize of one map of 4M voxels took 631 us, as 16-byte words 483, so 416
  char* sl = reinterpret_cast<char*>(t + h);
  reinterpret_cast<VSlot*>(sl)->mu[0] = q[0];
  *reinterpret_cast<float4*>(sl + 16) = make_float4(q[1], q[2], l00, l10);
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %7};" ::"l"(sl + 32),
               "r"(__float_as_uint(l20)), "r"(__float_as_uint(l11)), "r"(__float_as_uint(l21)),
               "r"(__float_as_uint(l22)), "r"(v), "r"(c), "r"(0u)
               : "memory");
}

// Per-voxel sums and the grouped cloud.  A CTA takes 128 consecutive ranks,
// whose point lists are one contiguous segment of plist:
//   1. the segment is loaded into shared memory (coalesced) and each thread
//      sorts its voxel's short list there by point index (segments longer than
//      the staging buffer sort in place in global memory);
//   2. point-parallel: every thread gathers points of the segment and writes
//      them to the grouped cloud at their list positions (balanced, coalesced
//      writes; the random reads all in flight at once);
//   3. voxel-parallel: each thread sums its voxel's points from the grouped copy
//      just written (L2-resident) and writes the voxel record.
constexpr int kFinThreads = 128;
constexpr int kFinStage = 3072;  // indices staged per CTA

// Map of rank (or voxel id) r: the last m with vbase[m] <= r.
__device__ __forceinline__ int map_of_rank(const uint32_t* __restrict__ vbase, int32_t n_maps,
                                           int64_t r) {
  int lo = 0, hi = n_maps;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if ((int64_t)vbase[mid] <= r) lo = mid; else hi = mid;
  }
  return lo;
}

// Least magnitude above zero among covariance entries off the diagonal (f: a point, then
// xx xy xz yy yz zz), as twice the bits less one: zeros last.
__device__ __forceinline__ uint32_t least_off_diagonal(uint32_t low, const float* f) {
  const uint32_t xy = 2u * __float_as_uint(f[4]) - 1u, xz = 2u * __float_as_uint(f[5]) - 1u,
                 yz = 2u * __float_as_uint(f[7]) - 1u;
  return min(min(low, xy), min(xz, yz));
}

// Exact sums of list entries o + first, o + first + step, ... < o + c of the grouped
// cloud (plain loads: written by the caller's kernel), in double-float: hi + lo stays
// the exact sum while each TwoSum error adds exactly to lo (checked).
template <bool LOW>
__device__ __forceinline__ void sum_entries(const float* gpts, const float* gcovs, uint32_t o,
                                            uint32_t c, uint32_t first, uint32_t step, float* hi,
                                            float* lo, bool& exact, uint32_t& low) {
  for (uint32_t a = first; a < c; a += step) {
    const int64_t d = (int64_t)o + a;
    float f[9];
#pragma unroll
    for (int k = 0; k < 3; ++k) f[k] = gpts[3 * d + k];
    const float2* gc = reinterpret_cast<const float2*>(gcovs + 6 * d);
    const float2 c0 = gc[0], c1 = gc[1], c2 = gc[2];
    f[3] = c0.x; f[4] = c0.y; f[5] = c1.x; f[6] = c1.y; f[7] = c2.x; f[8] = c2.y;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      float t, e, u, e2;
      two_sum(hi[k], f[k], t, e);
      two_sum(lo[k], e, u, e2);
      exact = exact && (e2 == 0.0f);
      hi[k] = t;
      lo[k] = u;
    }
    if (LOW) low = least_off_diagonal(low, f);
  }
}

// A binary64 sum in the two words of (hi, lo).
__device__ __forceinline__ void put_sum64(double s, float& hi, float& lo) {
  hi = __int_as_float(__double2hiint(s));
  lo = __int_as_float(__double2loint(s));
}
__device__ __forceinline__ double get_sum64(float hi, float lo) {
  return __hiloint2double(__float_as_int(hi), __float_as_int(lo));
}

// The binary64 sums of a list in ascending point index (the grouped order), where those in
// double-float are not exact (rare: large dynamic range).
__device__ __forceinline__ void sum_entries64(const float* gpts, const float* gcovs, uint32_t o,
                                              uint32_t c, float* hi, float* lo) {
  double sum[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) sum[k] = 0.0;
  for (uint32_t a = 0; a < c; ++a) {
    const int64_t d = (int64_t)o + a;
#pragma unroll
    for (int k = 0; k < 3; ++k) sum[k] = __dadd_rn(sum[k], (double)gpts[3 * d + k]);
#pragma unroll
    for (int k = 0; k < 6; ++k) sum[3 + k] = __dadd_rn(sum[3 + k], (double)gcovs[6 * d + k]);
  }
#pragma unroll
  for (int k = 0; k < 9; ++k) put_sum64(sum[k], hi[k], lo[k]);
}

// The record of voxel v (c points) from its sums: exact ones in double-float, else (words
// of) the binary64 ones; q: the means of the nine components.
__device__ __forceinline__ void write_record(uint32_t v, uint32_t c, float* hi, float* lo,
                                             bool exact, float4* __restrict__ recs, float* q) {
  // q = RN32(RN64(sum / N)) per component: from the exact float pair in
  // float32 where certified, else (rare) from the binary64 definition
  uint32_t need64 = exact ? 0u : 0x1FFu;
  if (exact) {
#pragma unroll
    for (int k = 0; k < 9; ++k) {  // hi = RN(hi + lo), lo = the exact remainder
      float t, e;
      two_sum(hi[k], lo[k], t, e);
      hi[k] = t;
      lo[k] = e;
    }
    const float rN = __frcp_rn((float)c);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      bool ok;
      q[k] = mean_rn32(hi[k], lo[k], c, rN, ok);
      if (!ok) need64 |= 1u << k;
    }
  }
  if (need64) {
    const double N = (double)c;
    const double y = __drcp_rn(N);
#pragma unroll
    for (int k = 0; k < 9; ++k)
      if (need64 & (1u << k)) {
        const double sum = exact ? __dadd_rn((double)hi[k], (double)lo[k])  // exact
                                 : get_sum64(hi[k], lo[k]);
        q[k] = __double2float_rn(div_rn(sum, N, y));
      }
  }
  recs[3 * v + 0] = make_float4(q[0], q[1], q[2], __uint_as_float(c));
  recs[3 * v + 1] = make_float4(q[3], q[4], q[5], q[6]);
  recs[3 * v + 2] = make_float4(q[7], q[8], 0.0f, 0.0f);
}

// One read of a word that other CTAs may be setting, whose value then stays.  (A relaxed
// load, which the kernel's other loads wait for, takes the rebuild of 500 maps of 50,000
// points 10 us more, of 3.1 ms, a volatile one 20.)
__device__ __forceinline__ int32_t read_once(const int32_t* p) {
  int32_t v;
  asm("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

// Row d of the grouped cloud without a point: NaN, which is no voxel's.
__device__ __forceinline__ void empty_row(float* gpts, float* gcovs, int64_t d) {
  const float nan = __uint_as_float(0x7FFFFFFFu);
#pragma unroll
  for (int k = 0; k < 3; ++k) gpts[3 * d + k] = nan;
#pragma unroll
  for (int k = 0; k < 6; ++k) gcovs[6 * d + k] = nan;
}

// Lists lie end to end but for the points without a voxel, which follow their map's last
// list (or fill the range of a map that has no voxel).  Those exist only after an
// insertion that reported an error, and only then is a list's length read from its
// voxel's count instead of the next offset: the read costs a dependent load.
__global__ void __launch_bounds__(kFinThreads) finalize_kernel(
    int64_t n_max, const uint32_t* __restrict__ n_vox, const float* __restrict__ pts,
    const float* __restrict__ covs, const uint32_t* __restrict__ vorder,
    const uint32_t* __restrict__ vcount, const uint32_t* __restrict__ goff,
    uint32_t* __restrict__ plist, float4* __restrict__ recs, float* gpts, float* gcovs,
    const unsigned long long* __restrict__ vkeys, int32_t n_maps,
    const uint32_t* __restrict__ vbase, const int64_t* __restrict__ slot_base,
    const uint32_t* __restrict__ vmask, int32_t max_probe, VSlot* vslots,
    uint32_t* __restrict__ lslot_of, int32_t* status) {
  __shared__ uint32_t stage[kFinStage];
  __shared__ int seg_map[2];
  const int64_t V = min((int64_t)*n_vox, n_max);
  const uint32_t total = (uint32_t)n_max;  // end of the last list (goff[V] is not stored)
  const bool dropped = read_once(status) != 0;
  if (V == 0)  // no point has a voxel
    for (int64_t i = blockIdx.x * (int64_t)kFinThreads + threadIdx.x; i < n_max;
         i += (int64_t)gridDim.x * kFinThreads)
      empty_row(gpts, gcovs, i);
  for (int64_t r0 = (int64_t)blockIdx.x * kFinThreads; r0 < V; r0 += (int64_t)gridDim.x * kFinThreads) {
    const int64_t r1 = min(V, r0 + kFinThreads);
    // list bounds from consecutive offsets: no dependent load through vorder
    const uint32_t seg0 = r0 > 0 ? goff[r0] : 0u;
    const uint32_t seg1 = r1 < V ? goff[r1] : total;
    const uint32_t len = seg1 - seg0;
    const bool staged = len <= (uint32_t)kFinStage;
    const int64_t r = r0 + threadIdx.x;
    const bool mine = r < r1;
    if (threadIdx.x == 0) {  // the maps of the CTA's first and last ranks
      seg_map[0] = map_of_rank(vbase, n_maps, r0);
      seg_map[1] = map_of_rank(vbase, n_maps, r1 - 1);
    }
    const uint32_t v = mine ? vorder[r] : 0u;
    const uint32_t o = mine ? goff[r] : 0u;
    const uint32_t c =
        !mine ? 0u : dropped ? vcount[v] : (r + 1 < V ? goff[r + 1] : total) - o;
    // 1. sort the lists by point index
    if (staged) {
      for (uint32_t i = threadIdx.x; i < len; i += kFinThreads) stage[i] = plist[seg0 + i];
      __syncthreads();
      if (mine) insertion_sort(stage + (o - seg0), c);
    } else if (mine) {
      sort_list(plist + o, c);
    }
    __syncthreads();
    // 2. gather into the grouped cloud
    const uint32_t* lst = staged ? stage : plist + seg0;
    for (uint32_t i = threadIdx.x; i < len; i += kFinThreads) {
      const int64_t j = min(lst[i], total - 1u);  // (kNoSlot: the row is emptied below)
      const float x = __ldg(pts + 3 * j), y = __ldg(pts + 3 * j + 1), z = __ldg(pts + 3 * j + 2);
      const float2* cv = reinterpret_cast<const float2*>(covs + 6 * j);
      const float2 c0 = __ldg(cv), c1 = __ldg(cv + 1), c2 = __ldg(cv + 2);
      const int64_t d = (int64_t)seg0 + i;
      gpts[3 * d + 0] = x;
      gpts[3 * d + 1] = y;
      gpts[3 * d + 2] = z;
      float2* gc = reinterpret_cast<float2*>(gcovs + 6 * d);
      gc[0] = c0;
      gc[1] = c1;
      gc[2] = c2;
    }
    if (dropped)
      for (uint32_t i = threadIdx.x; i < len; i += kFinThreads)
        if (lst[i] == kNoSlot) empty_row(gpts, gcovs, (int64_t)seg0 + i);
    __syncthreads();  // the CTA's global writes are visible to the CTA after this
    // 3. sums from the grouped copy (plain loads: written by this kernel)
    if (mine) {
      float hi[9], lo[9], q[9];
#pragma unroll
      for (int k = 0; k < 9; ++k) hi[k] = lo[k] = 0.0f;
      bool exact = true;
      uint32_t low = 0u;
      sum_entries<false>(gpts, gcovs, o, c, 0u, 1u, hi, lo, exact, low);
      if (!exact) sum_entries64(gpts, gcovs, o, c, hi, lo);
      write_record(v, c, hi, lo, exact, recs, q);
      // the voxel's map (ranks and voxel ids of a map share its range
      // [vbase[m], vbase[m + 1])): a CTA's ranks rarely span two maps
      int m = seg_map[0];
      while (m < seg_map[1] && (int64_t)vbase[m + 1] <= r) ++m;
      insert_lookup(v, vkeys[v], c, q, m, slot_base, vmask, max_probe, vslots,
                    lslot_of, status);
    }
    __syncthreads();  // the stage is reused by the next batch
  }
}

// (hi, lo) += the same of the lane at distance `delta`, exactly (checked).
__device__ __forceinline__ void add_lane(float* hi, float* lo, bool& exact, int delta) {
  const bool other = __shfl_xor_sync(0xFFFFFFFFu, (int)exact, delta) != 0;
  exact = exact && other;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const float h = __shfl_xor_sync(0xFFFFFFFFu, hi[k], delta);
    const float l = __shfl_xor_sync(0xFFFFFFFFu, lo[k], delta);
    float t, e, u, e2, v, e3;
    two_sum(hi[k], h, t, e);
    two_sum(lo[k], l, u, e2);
    two_sum(u, e, v, e3);
    exact = exact && e2 == 0.0f && e3 == 0.0f;
    hi[k] = t;
    lo[k] = v;
  }
}

// The sums of the nine components of list entries o .. o + c - 1 in ascending point index,
// one by each of a warp's first lanes: as sum_entries, or (words of) the binary64 sums where
// one of those is not exact.  Returns whether they all are.
__device__ __forceinline__ bool sum_components(const float* gpts, const float* gcovs, int lane,
                                               uint32_t o, uint32_t c, float& hi, float& lo) {
  const float* const f = lane < 3 ? gpts + 3 * (int64_t)o + lane : gcovs + 6 * (int64_t)o + (lane - 3);
  const int step = lane < 3 ? 3 : 6;
  const uint32_t n = lane < 9 ? c : 0u;
  bool exact = true;
#pragma unroll 4
  for (uint32_t a = 0; a < n; ++a) {
    float t, e, u, e2;
    two_sum(hi, f[(int64_t)step * a], t, e);
    two_sum(lo, e, u, e2);
    exact = exact && e2 == 0.0f;
    hi = t;
    lo = u;
  }
  if (__all_sync(0xFFFFFFFFu, exact)) return true;
  double sum = 0.0;
#pragma unroll 4
  for (uint32_t a = 0; a < n; ++a) sum = __dadd_rn(sum, (double)f[(int64_t)step * a]);
  put_sum64(sum, hi, lo);
  return false;
}

// Whether the order of a list's exact sums cannot matter (hi: the sums, low: the least
// off-diagonal magnitude): the partial sums, below the largest diagonal sum (covariances are
// positive semi-definite), are multiples of the last bit of the smallest and at most 2^53 of
// them, so that the sums in ascending point index are exact too.  (Coordinates, which have
// one sign in a voxel, and diagonal entries do not cancel.)
__device__ __forceinline__ bool any_order(const float* hi, uint32_t low) {
  const float top = fmaxf(fabsf(hi[3]), fmaxf(fabsf(hi[6]), fabsf(hi[8])));
  const int e = (int)(__float_as_uint(top) >> 23) + 1;
  return low == 0xFFFFFFFFu || (e < 255 && e - max((int)((low + 1u) >> 24), 1) <= 30);
}

// What any_order leaves open, by component, `per` lanes to a list: whether the entries off
// the diagonal are multiples of the last bit of their component's smallest and their
// partial sums, at most c times the largest, below 2^53 of those.  (Off-diagonal entries
// that are all tiny, of planes along an axis, stay open above.)
__device__ __forceinline__ bool off_diagonals_fit(const float* gcovs, uint32_t o, uint32_t c,
                                                  int part, int per) {
  uint32_t low[3], top[3];  // bits less one (zeros last), bits
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    low[k] = 0xFFFFFFFFu;
    top[k] = 0u;
  }
  for (uint32_t a = part; a < c; a += per) {
    const float* const f = gcovs + 6 * ((int64_t)o + a);
    const float v[3] = {f[1], f[2], f[4]};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const uint32_t b = __float_as_uint(v[k]) & 0x7FFFFFFFu;
      low[k] = min(low[k], b - 1u);
      top[k] = max(top[k], b);
    }
  }
  bool fits = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    for (int d = 1; d < per; d <<= 1) {
      low[k] = min(low[k], __shfl_xor_sync(0xFFFFFFFFu, low[k], d));
      top[k] = max(top[k], __shfl_xor_sync(0xFFFFFFFFu, top[k], d));
    }
    const int e_top = max((int)(top[k] >> 23), 1), e_low = max((int)((low[k] + 1u) >> 23), 1);
    fits = fits && (top[k] == 0u ||
                    (e_top < 255 && e_top - e_low + 32 - __clz((int)(c - 1u)) <= 29));
  }
  return fits;
}

// The same for long lists: R consecutive ranks per CTA, 128 / R threads per voxel, R
// the power of two that makes about 512 points per CTA.  The lists are not sorted
// first: a point's position in the grouped cloud is the number of smaller indices in
// its list, counted by the thread that copies it.  A voxel's threads sum its points
// (exact partial sums, joined exactly); a list longer than 64 points per thread is
// summed by the whole warp.  Where the order of the points may matter, or the sums are not
// exact, nine lanes sum the list once more in ascending point index, a component each (a
// list of 160 points that one lane summed in binary64 took 100 us; rebuild of ten maps of
// 20,000 points at 100 per voxel, one such list 185 -> 99 us, none 86).  A segment longer
// than the staging buffer (a voxel of thousands of points) is sorted in place by one thread
// per voxel, as above.
// Bounded by the latency of the chain offsets - indices - gather - sums on few CTAs.
// This kernel / the one above (points per voxel on average): ten maps of 20,000
// points 19 / 18 us (2.0), 20 / 28 (5.7), 19 / 55 (11), 21 / 148 (23), 49 / 1554 (91);
// 20 maps of 40,000 52 / 66 (11); 100 maps of 50,000 252 / 230 (3.8), 226 / 212 (8.1),
// 233 / 314 (15), 322 / 781 (33).  More registers (80 against 56) cost it the large
// sets of short lists (six CTAs per SM asked for: the compiler takes 96 otherwise).
constexpr uint32_t kFinSerial = 64;
__global__ void __launch_bounds__(kFinThreads, 6) finalize_long_kernel(
    int64_t n_max, const uint32_t* __restrict__ n_vox, const float* __restrict__ pts,
    const float* __restrict__ covs, const uint32_t* __restrict__ vorder,
    const uint32_t* __restrict__ vcount, const uint32_t* __restrict__ goff,
    uint32_t* __restrict__ plist, float4* __restrict__ recs, float* gpts, float* gcovs,
    const unsigned long long* __restrict__ vkeys, int32_t n_maps,
    const uint32_t* __restrict__ vbase, const int64_t* __restrict__ slot_base,
    const uint32_t* __restrict__ vmask, int32_t max_probe, VSlot* vslots,
    uint32_t* __restrict__ lslot_of, int32_t* status) {
  __shared__ uint32_t stage[kFinStage];
  __shared__ uint32_t list_at[kFinThreads];  // first entry of each list, in the segment
  const int64_t V = min((int64_t)*n_vox, n_max);
  const uint32_t total = (uint32_t)n_max;  // end of the last list (goff[V] is not stored)
  const bool dropped = read_once(status) != 0;
  if (V == 0)  // no point has a voxel
    for (int64_t i = blockIdx.x * (int64_t)kFinThreads + threadIdx.x; i < n_max;
         i += (int64_t)gridDim.x * kFinThreads)
      empty_row(gpts, gcovs, i);
  const uint32_t avg = (uint32_t)(n_max / max((int64_t)1, V));
  int R = kFinThreads;
  while (R > 4 && (uint32_t)R * avg > 512u) R >>= 1;
  const int per = kFinThreads / R;  // threads per voxel (1 .. 32)
  const int lane = threadIdx.x & 31, part = (int)threadIdx.x & (per - 1);
  for (int64_t r0 = (int64_t)blockIdx.x * R; r0 < V; r0 += (int64_t)gridDim.x * R) {
    const int64_t r1 = min(V, r0 + R);
    const uint32_t seg0 = r0 > 0 ? goff[r0] : 0u;
    const uint32_t seg1 = r1 < V ? goff[r1] : total;
    const uint32_t len = seg1 - seg0;
    const bool staged = len <= (uint32_t)kFinStage;
    const int64_t r = r0 + (int)threadIdx.x / per;
    const bool ours = r < r1, mine = ours && part == 0;
    const uint32_t v = mine || (ours && dropped) ? vorder[r] : 0u;
    const uint32_t o = ours ? goff[r] : 0u;
    const uint32_t c =
        !ours ? 0u : dropped ? vcount[v] : (r + 1 < V ? goff[r + 1] : total) - o;
    if (staged) {
      for (uint32_t i = threadIdx.x; i < len; i += kFinThreads) stage[i] = plist[seg0 + i];
      if (mine) list_at[r - r0] = o - seg0;
    } else if (mine) {
      sort_list(plist + o, c);
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < len; i += kFinThreads) {
      const uint32_t id = staged ? stage[i] : plist[seg0 + i];
      const int64_t j = min(id, total - 1u);  // (kNoSlot: the row is emptied below)
      const float x = __ldg(pts + 3 * j), y = __ldg(pts + 3 * j + 1), z = __ldg(pts + 3 * j + 2);
      const float2* cv = reinterpret_cast<const float2*>(covs + 6 * j);
      const float2 c0 = __ldg(cv), c1 = __ldg(cv + 1), c2 = __ldg(cv + 2);
      int64_t d = (int64_t)seg0 + i;
      if (staged && id != kNoSlot) {
        int q = 0, end = (int)(r1 - r0);  // the entry's list: the last with list_at <= i
        while (end - q > 1) {
          const int mid = (q + end) >> 1;
          if (list_at[mid] <= i) q = mid; else end = mid;
        }
        const uint32_t a = list_at[q], e = q + 1 < (int)(r1 - r0) ? list_at[q + 1] : len;
        uint32_t smaller = 0u;
#pragma unroll 4
        for (uint32_t t = a; t < e; ++t) smaller += stage[t] < id ? 1u : 0u;
        d = (int64_t)seg0 + a + smaller;
      }
      gpts[3 * d + 0] = x;
      gpts[3 * d + 1] = y;
      gpts[3 * d + 2] = z;
      float2* gc = reinterpret_cast<float2*>(gcovs + 6 * d);
      gc[0] = c0;
      gc[1] = c1;
      gc[2] = c2;
    }
    if (dropped)
      for (uint32_t i = threadIdx.x; i < len; i += kFinThreads)
        if ((staged ? stage[i] : plist[seg0 + i]) == kNoSlot)
          empty_row(gpts, gcovs, (int64_t)seg0 + i);
    __syncthreads();  // the CTA's global writes are visible to the CTA after this
    float hi[9], lo[9], q[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) hi[k] = lo[k] = 0.0f;
    bool exact = true;
    uint32_t low = 0xFFFFFFFFu;
    const bool by_warp = c > kFinSerial * (uint32_t)per;
    if (!by_warp) sum_entries<true>(gpts, gcovs, o, c, part, per, hi, lo, exact, low);
    for (int d = 1; d < per; d <<= 1) {
      add_lane(hi, lo, exact, d);
      low = min(low, __shfl_xor_sync(0xFFFFFFFFu, low, d));
    }
    for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, mine && by_warp); todo; todo &= todo - 1u) {
      const int b = __ffs(todo) - 1;  // the whole warp sums the list of lane b
      const uint32_t ob = __shfl_sync(0xFFFFFFFFu, o, b), cb = __shfl_sync(0xFFFFFFFFu, c, b);
      float h[9], l[9];
      bool ex = true;
      uint32_t lw = 0xFFFFFFFFu;
#pragma unroll
      for (int k = 0; k < 9; ++k) h[k] = l[k] = 0.0f;
      sum_entries<true>(gpts, gcovs, ob, cb, lane, 32u, h, l, ex, lw);
#pragma unroll 1
      for (int d = 1; d < 32; d <<= 1) add_lane(h, l, ex, d);
      lw = __reduce_min_sync(0xFFFFFFFFu, lw);
      if (lane == b) {
        low = lw;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          hi[k] = h[k];
          lo[k] = l[k];
        }
        exact = ex;
      }
    }
    bool open = mine && exact && (per > 1 || by_warp) && !any_order(hi, low);
    if (__any_sync(0xFFFFFFFFu, open)) {  // by component, by the lists' threads
      open = __shfl_sync(0xFFFFFFFFu, (int)open, lane & ~(per - 1)) != 0;
      const bool fits = off_diagonals_fit(gcovs, o, open ? c : 0u, part, per);
      open = open && !fits;
    }
    const bool again = mine && (!exact || open);
    for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, again); todo; todo &= todo - 1u) {
      const int b = __ffs(todo) - 1;  // the list of lane b in ascending index, by nine lanes
      const uint32_t ob = __shfl_sync(0xFFFFFFFFu, o, b), cb = __shfl_sync(0xFFFFFFFFu, c, b);
      float h = 0.0f, l = 0.0f;
      const bool ex = sum_components(gpts, gcovs, lane, ob, cb, h, l);
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const float hk = __shfl_sync(0xFFFFFFFFu, h, k), lk = __shfl_sync(0xFFFFFFFFu, l, k);
        if (lane == b) {
          hi[k] = hk;
          lo[k] = lk;
        }
      }
      if (lane == b) exact = ex;
    }
    if (mine) {
      write_record(v, c, hi, lo, exact, recs, q);
      insert_lookup(v, vkeys[v], c, q, map_of_rank(vbase, n_maps, r), slot_base, vmask, max_probe,
                    vslots, lslot_of, status);
    }
    __syncthreads();  // the stage is reused by the next ranks
  }
}

// 10 bits per axis of the key, interleaved (a locality order, not a unique code).
__device__ __forceinline__ uint32_t spread10(uint32_t x) {
  x &= 1023u;
  x = (x | (x << 16)) & 0x030000FFu;
  x = (x | (x << 8)) & 0x0300F00Fu;
  x = (x | (x << 4)) & 0x030C30C3u;
  x = (x | (x << 2)) & 0x09249249u;
  return x;
}
// One CTA (of 1024 threads) or one cluster of 8 CTAs (of 256) per (map, chunk): the
// chunk's voxels sorted by Morton code (ties by voxel id); vorder[rank] = v, goff[rank] =
// the offset of its point list (the map's first point plus the counts of the ranks
// before; the lists of a map fill its range of points), also stored by voxel for the
// scatter, as (offset << 32 | fill 0).
//
// A stable radix sort, least significant digit first, the elements spread evenly
// over the CTAs' shared memory.  A warp holds 32 J consecutive elements, J per lane
// in registers; for each, the lanes with the same digit are found by one ballot per
// digit bit, and the warp's counter of that digit gives the element's rank among the
// warp's.  The CTAs exchange their digit counts through distributed shared memory; a
// scan over (digit, CTA, warp) turns counters into places, and the elements are
// scattered to the CTAs that own the places.  Up to 2,048 voxels are sorted by the
// cluster's first CTA alone.
// The code is shortened first: in each axis the bits above the largest magnitude
// are copies of the sign (bit 9), which never decide an order by themselves, so
// m + 1 bits per axis are sorted (a map within +-64 voxels: 21 bits, three passes of
// 7) instead of 10.
// Bounded by issue (about 60 instructions per element and pass) and, for few
// chunks, by the passes' barriers; clusters pay for scattering between SMs, so many
// chunks are sorted by one CTA each.  Cluster / single CTA, maps of n points (V
// voxels): 10 maps of 20,000 (V = 19,000) 27 / 58 us, 10 of 20,000 (9,700) 17 / 36,
// 20 of 40,000 (37,000) 56 / 58, 20 of 80,000 (41,000) 52 / 49, 100 of 50,000
// (12,000) 76 / 47, 500 of 50,000 264 / 169.  A bitonic sort (29 passes through shared
// memory for 16K elements) took 65 us for 10 maps of 20,000 and 278 us for the 500
// maps of the global map.
constexpr int kDigitBits = 8;
constexpr int kDigits = 1 << kDigitBits;
constexpr int kSortElems = 2048;  // elements a CTA of a cluster holds

template <int CTAS, int THREADS>
struct SortSmem {
  static constexpr int kWarps = THREADS / 32, kGroups = THREADS / kDigits;
  uint32_t key[kMortonChunk / CTAS];
  uint16_t idx[kMortonChunk / CTAS];
  uint32_t count[kWarps][kDigits];   // then: place of the warp's first of the digit
  uint32_t part[kGroups][kDigits];   // the same per 8 warps
  uint32_t total[CTAS][kDigits];     // digit counts of every CTA of the cluster
  uint32_t bits[CTAS];
  uint32_t warp[kWarps];
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::
                   : "memory");
}
__device__ __forceinline__ uint32_t smem_of_rank(const void* p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(a)
               : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_cluster16(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(addr), "h"((uint16_t)v) : "memory");
}

// Points of each chunk, for maps of many chunks: a chunk's list offsets start behind its
// map's earlier chunks, whose voxels it otherwise counts itself, which is quadratic in the
// map.  Rebuild of one map of n points (V voxels), counting itself / by this kernel: 50,000
// (46,000) 81 / 91 us, 100,000 (92,000) 92 / 95, 200,000 (184,000) 117 / 111, 1M 414 / 355,
// 4M 1,312 / 1,185, 16M 6,571 / 5,167; 100 maps of 100,000 2,164 / 2,193.
constexpr uint32_t kOwnCount = 8 * kMortonChunk;  // up to that many voxels in a map
__global__ void __launch_bounds__(kThreads) chunk_points_kernel(
    const int2* __restrict__ chunks, const uint32_t* __restrict__ vbase,
    const uint32_t* __restrict__ vcount, uint32_t* __restrict__ chunk_points) {
  const int2 ch = chunks[blockIdx.x];
  const uint32_t v0 = vbase[ch.x], V = vbase[ch.x + 1] - v0, lo = (uint32_t)ch.y * kMortonChunk;
  if (lo >= V) return;
  const uint32_t hi = min(V, lo + kMortonChunk);
  uint32_t sum = 0u;
#pragma unroll 8
  for (uint32_t i = lo + threadIdx.x; i < hi; i += kThreads) sum += vcount[v0 + i];
  __shared__ uint32_t warp_sum[kThreads / 32];
  sum = __reduce_add_sync(0xFFFFFFFFu, sum);
  if ((threadIdx.x & 31) == 0) warp_sum[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int i = 1; i < kThreads / 32; ++i) sum += warp_sum[i];
  chunk_points[blockIdx.x] = sum;
}

template <int CTAS, int THREADS>
__global__ void __launch_bounds__(THREADS) morton_sort_kernel(
    const int2* __restrict__ chunks, const uint32_t* __restrict__ chunk_points,
    const uint32_t* __restrict__ vbase,
    const unsigned long long* __restrict__ vkeys, const uint32_t* __restrict__ vcount,
    const int64_t* __restrict__ point_off, uint32_t* __restrict__ vorder,
    uint32_t* __restrict__ goff, unsigned long long* __restrict__ bfill) {
  constexpr int kWarps = THREADS / 32, kGroups = THREADS / kDigits, kEach = kWarps / kGroups;
  constexpr int kItems = kMortonChunk / (CTAS * THREADS);
  static_assert(kEach == 8 && kItems % 2 == 0, "scan and register layout");
  extern __shared__ __align__(16) unsigned char sort_smem[];
  auto& S = *reinterpret_cast<SortSmem<CTAS, THREADS>*>(sort_smem);
  const int2 ch = chunks[blockIdx.x / CTAS];
  const int m = ch.x;
  const uint32_t v0 = vbase[m], V = vbase[m + 1] - v0;
  const uint32_t lo = (uint32_t)ch.y * kMortonChunk;
  if (lo >= V) return;
  const uint32_t cnt = min((uint32_t)kMortonChunk, V - lo);
  const uint32_t first = v0 + lo;
  const uint32_t rank = CTAS > 1 ? cluster_rank() : 0u;
  const uint32_t ctas = cnt <= (uint32_t)kSortElems ? 1u : (uint32_t)CTAS;
  if (rank >= ctas) return;  // the first CTA sorts alone: no cluster barrier below
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t J = (cnt + ctas * THREADS - 1) / (ctas * THREADS);  // elements per lane
  const uint32_t c0 = rank * (J * THREADS);                          // this CTA's first
  const uint32_t mine = cnt > c0 ? min(J * (uint32_t)THREADS, cnt - c0) : 0u;
  const uint32_t e0 = (uint32_t)w * 32u * J + (uint32_t)lane;  // element j: c0 + e0 + 32 j

  // keys: 10 bits per axis, and the bits that differ from their axis' sign
  uint32_t key[kItems];
  uint32_t diff = 0u;
#pragma unroll
  for (int j = 0; j < kItems; ++j) {
    const uint32_t e = e0 + 32u * j;
    key[j] = 0u;
    if (j < (int)J && e < mine) {
      const unsigned long long k = vkeys[first + c0 + e];
      const uint32_t x = (uint32_t)(k >> (2 * kKeyBits)) & 1023u, y = (uint32_t)(k >> kKeyBits) & 1023u,
                     z = (uint32_t)k & 1023u;
      key[j] = x | (y << 10) | (z << 20);
      diff |= (x ^ (0u - (x >> 9))) | (y ^ (0u - (y >> 9))) | (z ^ (0u - (z >> 9)));
    }
  }
  diff = __reduce_or_sync(0xFFFFFFFFu, diff & 511u);
  if (lane == 0) S.warp[w] = diff;
  __syncthreads();
  uint32_t bits = 0u;
  for (int i = 0; i < kWarps; ++i) bits |= S.warp[i];
  if (ctas > 1u) {
    cluster_sync();  // every CTA of the cluster runs
    if (threadIdx.x < ctas) st_cluster(smem_of_rank(&S.bits[rank], threadIdx.x), bits);
    cluster_sync();
    for (uint32_t i = 0; i < ctas; ++i) bits |= S.bits[i];
  }
  const int mag = 32 - __clz((int)bits);               // magnitude bits kept (0 .. 9)
  const int total_bits = 3 * (mag + 1);
  const int passes = (total_bits + kDigitBits - 1) / kDigitBits;
  const int digit_bits = (total_bits + passes - 1) / passes;
  const uint32_t low = (1u << mag) - 1u;
#pragma unroll
  for (int j = 0; j < kItems; ++j) {
    const uint32_t x = key[j] & 1023u, y = (key[j] >> 10) & 1023u, z = key[j] >> 20;
    key[j] = spread10((x & low) | ((x >> 9) << mag)) | (spread10((y & low) | ((y >> 9) << mag)) << 1) |
             (spread10((z & low) | ((z >> 9) << mag)) << 2);
  }
  uint32_t idx[kItems / 2];  // index in the chunk, two 16-bit values a word
#pragma unroll
  for (int j = 0; j < kItems; j += 2) {
    const uint32_t i = c0 + e0 + 32u * j;
    idx[j / 2] = i | ((i + 32u) << 16);
  }

  const uint32_t digit_mask = (1u << digit_bits) - 1u;
  const uint32_t lower = (1u << lane) - 1u;
  const uint32_t inv_j = 65536u / J + 1u;  // (p / 256) / J for p / 256 < 64 and J <= 8
  for (int pass = 0; pass < passes; ++pass) {
    const int shift = pass * digit_bits;
    if (pass > 0) {
#pragma unroll
      for (int j = 0; j < kItems; ++j) {
        const uint32_t e = e0 + 32u * j;
        if (j < (int)J && e < mine) {
          key[j] = S.key[e];
          const uint32_t v = S.idx[e];
          idx[j / 2] = (j & 1) ? (idx[j / 2] & 0xFFFFu) | (v << 16) : (idx[j / 2] & 0xFFFF0000u) | v;
        }
      }
    }
    for (int d = lane; d < kDigits; d += 32) S.count[w][d] = 0u;
    __syncwarp();
    uint32_t rk[kItems / 2];  // rank among the warp's elements of the digit, 16 bits
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      if (j < (int)J) {  // the same for all lanes
        const bool live = e0 + 32u * j < mine;
        const uint32_t d = (key[j] >> shift) & digit_mask;
        uint32_t peers = __ballot_sync(0xFFFFFFFFu, live);
#pragma unroll
        for (int b = 0; b < kDigitBits; ++b) {
          const uint32_t bit = 0u - ((d >> b) & 1u);
          peers &= ~(__ballot_sync(0xFFFFFFFFu, bit != 0u) ^ bit);
        }
        const uint32_t seen = live ? S.count[w][d] : 0u;
        __syncwarp();
        if (live && (peers & lower) == 0u) S.count[w][d] = seen + (uint32_t)__popc(peers);
        __syncwarp();
        const uint32_t r = seen + (uint32_t)__popc(peers & lower);
        rk[j / 2] = (j & 1) ? rk[j / 2] | (r << 16) : r;
      }
    }
    __syncthreads();
    // counters -> places, in the order (digit, CTA, warp); thread = (digit, 8 warps)
    const int d = threadIdx.x % kDigits, g = threadIdx.x / kDigits;
    uint32_t c[kEach], sum = 0u;
#pragma unroll
    for (int i = 0; i < kEach; ++i) {
      c[i] = S.count[g * kEach + i][d];
      sum += c[i];
    }
    if (kGroups > 1) {
      S.part[g][d] = sum;
      __syncthreads();
      if (g == 0)
#pragma unroll
        for (int i = 1; i < kGroups; ++i) sum += S.part[i][d];
    }
    uint32_t all = sum, before = 0u, inc = 0u;  // of the digit (threads of group 0)
    if (ctas > 1u) {
      for (uint32_t r = 0; r < ctas; ++r) st_cluster(smem_of_rank(&S.total[rank][d], r), sum);
      cluster_sync();
      all = 0u;
#pragma unroll
      for (int r = 0; r < CTAS; ++r) {
        const uint32_t t = S.total[r][d];
        all += t;
        if (r < (int)rank) before += t;
      }
    }
    if (g == 0) {  // whole warps
      inc = all;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
      }
      if (lane == 31) S.warp[w] = inc;
    }
    __syncthreads();
    uint32_t run = 0u;
    if (g == 0) {
      run = inc - all + before;
      for (int i = 0; i < w; ++i) run += S.warp[i];
    }
    if (kGroups > 1) {
      if (g == 0) {  // part <- first place of (digit, group)
        const uint32_t p0 = c[0] + c[1] + c[2] + c[3] + c[4] + c[5] + c[6] + c[7];
        uint32_t at = run + p0;
#pragma unroll
        for (int i = 1; i < kGroups; ++i) {
          const uint32_t x = S.part[i][d];
          S.part[i][d] = at;
          at += x;
        }
      }
      __syncthreads();
      if (g > 0) run = S.part[g][d];
    }
#pragma unroll
    for (int i = 0; i < kEach; ++i) {
      S.count[g * kEach + i][d] = run;
      run += c[i];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      if (j < (int)J && e0 + 32u * j < mine) {
        const uint32_t p = S.count[w][(key[j] >> shift) & digit_mask] +
                           ((rk[j / 2] >> (16 * (j & 1))) & 0xFFFFu);
        const uint32_t i = (idx[j / 2] >> (16 * (j & 1))) & 0xFFFFu;
        if (CTAS == 1 || ctas == 1u) {
          S.key[p] = key[j];
          S.idx[p] = (uint16_t)i;
        } else {
          const uint32_t to = ((p / THREADS) * inv_j) >> 16;
          const uint32_t o = p - to * (J * THREADS);
          st_cluster(smem_of_rank(&S.key[o], to), key[j]);
          st_cluster16(smem_of_rank(&S.idx[o], to), i);
        }
      }
    }
    if (ctas > 1u) cluster_sync();
    else __syncthreads();
  }
  // points of the map's earlier chunks
  uint32_t base = 0u;
  if (chunk_points)
    for (uint32_t i = threadIdx.x; i < (uint32_t)ch.y; i += THREADS)
      base += chunk_points[blockIdx.x / CTAS - 1u - i];
  else
    for (uint32_t i = threadIdx.x; i < lo; i += THREADS) base += vcount[v0 + i];
  base = __reduce_add_sync(0xFFFFFFFFu, base);
  if (lane == 0) S.warp[w] = base;
  __syncthreads();
  base = (uint32_t)point_off[m];
  for (int i = 0; i < kWarps; ++i) base += S.warp[i];
  // list offsets: a scan of the counts in rank order, 32 ranks of the warp's at a time,
  // then over the warps and the CTAs before
  uint32_t off[kItems], run = 0u;
#pragma unroll
  for (int j = 0; j < kItems; ++j) {
    off[j] = 0u;
    if (j < (int)J) {  // the same for all lanes
      const uint32_t e = e0 + 32u * j;
      uint32_t n = 0u;
      if (e < mine) {
        const uint32_t v = first + (uint32_t)S.idx[e];
        vorder[first + c0 + e] = v;
        n = vcount[v];
      }
      uint32_t inc = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
      }
      off[j] = run + inc - n;
      run += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
  }
  __syncthreads();  // S.warp has been read
  if (lane == 0) S.warp[w] = run;
  __syncthreads();
  uint32_t all = 0u;
  for (int i = 0; i < kWarps; ++i) {
    if (i < w) base += S.warp[i];
    all += S.warp[i];
  }
  if (ctas > 1u) {
    if (threadIdx.x < ctas) st_cluster(smem_of_rank(&S.bits[rank], threadIdx.x), all);
    cluster_sync();
#pragma unroll
    for (int i = 0; i < CTAS; ++i)
      if (i < (int)rank) base += S.bits[i];
  }
#pragma unroll
  for (int j = 0; j < kItems; ++j) {
    const uint32_t e = e0 + 32u * j;
    if (j < (int)J && e < mine) {
      const uint32_t o = base + off[j];
      goff[first + c0 + e] = o;
      bfill[first + (uint32_t)S.idx[e]] = (unsigned long long)o << 32;
    }
  }
}

// Launches the sort with CTAS CTAs of THREADS threads per chunk.
template <int CTAS, int THREADS>
int launch_sort(const MapSet* s, const uint32_t* chunk_points, uint32_t* vorder,
                unsigned long long* bfill, cudaStream_t st) {
  constexpr int kBytes = (int)sizeof(SortSmem<CTAS, THREADS>);
  auto* kernel = morton_sort_kernel<CTAS, THREADS>;
  if (kBytes > 48 * 1024) {  // above the default limit: opt in once per device
    static std::mutex attr_mu;
    static bool attr_set[kMaxDevices] = {false};
    int dev = 0;
    VGICP_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices)
      return set_error(VGICP_ERR_INVALID_ARG, "device index beyond the supported range");
    std::lock_guard<std::mutex> lock(attr_mu);
    if (!attr_set[dev]) {
      VGICP_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBytes));
      attr_set[dev] = true;
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)s->n_chunks * CTAS);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = kBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = CTAS;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = CTAS > 1 ? 1 : 0;
  VGICP_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, (const int2*)s->d_chunks, chunk_points,
                                    (const uint32_t*)s->d_vbase,
                                    (const unsigned long long*)s->d_vkeys,
                                    (const uint32_t*)s->d_vcount, (const int64_t*)s->d_point_off,
                                    vorder, s->d_goff, bfill));
  return VGICP_OK;
}

__device__ __forceinline__ uint32_t lookup_capacity(uint32_t nvox) {
  uint32_t c = 16;
  while (c < kLookupLoad * nvox) c <<= 1;
  return c;
}

// Slots a build uses of a map's region, which the first build sized; a rebuild with
// more voxels runs at a higher load factor (an insertion past max_probe reports
// VGICP_ERR_HASH_FULL).
__device__ __forceinline__ uint32_t table_capacity(uint32_t nvox, uint32_t region) {
  return min(lookup_capacity(nvox), region);
}

// First build (and empty sets), per map (blockIdx.y): lookup-table capacity from its
// voxel count; with clear_all, every slot of the map's region emptied (fresh memory;
// later builds find the region empty after the reset).
__global__ void vslot_init_kernel(const int64_t* __restrict__ slot_base,
                                  const uint32_t* __restrict__ vbase, VSlot* vslots,
                                  uint32_t* __restrict__ vmask, int32_t clear_all) {
  const int m = blockIdx.y;
  const uint32_t region = (uint32_t)(slot_base[m + 1] - slot_base[m]);
  const uint32_t cap = table_capacity(vbase[m + 1] - vbase[m], region);
  if (clear_all) {
    VSlot* t = vslots + slot_base[m];
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < region;
         i += gridDim.x * blockDim.x) {
      // the whole first 32-B sector (key = empty, spill = 0): no read-modify-write
      asm volatile("st.global.v8.b32 [%0], {%1, %1, %2, %2, %2, %2, %2, %2};" ::"l"(t + i),
                   "r"(0xFFFFFFFFu), "r"(0u)
                   : "memory");
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) vmask[m] = cap - 1u;
}

// ---- exclusive scan of uint32 (three phases) --------------------------------
constexpr int kScanThreads = 256;
constexpr int kScanPerThread = 8;
constexpr int kScanTile = kScanThreads * kScanPerThread;

__device__ __forceinline__ int64_t scan_len(int64_t n_max, const uint32_t* n_dev) {
  return n_dev ? min(n_max, (int64_t)*n_dev) : n_max;
}

// Block-wide exclusive scan of one value per thread (T threads); returns the
// thread's exclusive prefix and writes the block total to *total.
template <int T>
__device__ __forceinline__ uint32_t block_exclusive(uint32_t x, uint32_t* total) {
  static_assert(T % 32 == 0 && T <= 1024, "block size");
  __shared__ uint32_t warp_sum[T / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) warp_sum[w] = inc;
  __syncthreads();
  if (w == 0) {
    uint32_t ws = lane < T / 32 ? warp_sum[lane] : 0u;
    uint32_t wi = ws;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(0xFFFFFFFFu, wi, o);
      if (lane >= o) wi += y;
    }
    if (lane < T / 32) warp_sum[lane] = wi - ws;
    if (lane == T / 32 - 1) *total = wi;
  }
  __syncthreads();
  uint32_t r = warp_sum[w] + inc - x;
  __syncthreads();
  return r;
}

__global__ void scan_tile_sums_kernel(const uint32_t* __restrict__ in, int64_t n_max,
                                      const uint32_t* n_dev, uint32_t* __restrict__ sums) {
  const int64_t n = scan_len(n_max, n_dev);
  const int64_t base = (int64_t)blockIdx.x * kScanTile + threadIdx.x * kScanPerThread;
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < kScanPerThread; ++k)
    if (base + k < n) s += in[base + k];
  __shared__ uint32_t total;
  block_exclusive<kScanThreads>(s, &total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// One CTA: each thread scans a contiguous run of the tile sums.
constexpr int kScanSumsThreads = 1024;
__global__ void __launch_bounds__(kScanSumsThreads) scan_sums_kernel(
    uint32_t* __restrict__ sums, int64_t nb, uint32_t* __restrict__ total_dev) {
  __shared__ uint32_t total;
  const int64_t per = (nb + kScanSumsThreads - 1) / kScanSumsThreads;
  const int64_t a = min(nb, (int64_t)threadIdx.x * per), b = min(nb, a + per);
  uint32_t s = 0;
  for (int64_t i = a; i < b; ++i) s += sums[i];
  uint32_t run = block_exclusive<kScanSumsThreads>(s, &total);
  for (int64_t i = a; i < b; ++i) {
    const uint32_t x = sums[i];
    sums[i] = run;
    run += x;
  }
  if (threadIdx.x == 0 && total_dev) *total_dev = total;
}

__global__ void scan_tiles_kernel(const uint32_t* in, uint32_t* out, int64_t n_max,
                                  const uint32_t* n_dev, const uint32_t* __restrict__ sums) {
  const int64_t n = scan_len(n_max, n_dev);
  const int64_t base = (int64_t)blockIdx.x * kScanTile + threadIdx.x * kScanPerThread;
  uint32_t v[kScanPerThread];
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < kScanPerThread; ++k) {
    v[k] = (base + k < n) ? in[base + k] : 0u;
    s += v[k];
  }
  __shared__ uint32_t total;
  uint32_t run = block_exclusive<kScanThreads>(s, &total) + sums[blockIdx.x];
#pragma unroll
  for (int k = 0; k < kScanPerThread; ++k) {
    if (base + k < n) out[base + k] = run;
    run += v[k];
  }
}

// ---- first-appearance numbering -----------------------------------------
// A point is its voxel's first if its index is the smallest of the voxel (the
// build-table slot holds that index after the insert).  The first points are
// marked in a bitmap (one warp ballot per 32 points); a voxel's id is the number
// of marked points before its first point (an exclusive scan of the words'
// popcounts), so voxels are numbered in order of first appearance, map by map.

// One thread per point; every warp is whole, so the ballot sees all 32 lanes.  The
// grid covers the word of index n, which the ranks below read.
__global__ void first_bits_kernel(const uint32_t* __restrict__ pt_slot,
                                  const Slot* __restrict__ slots, int64_t n,
                                  uint32_t* __restrict__ bitmap) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  bool f = false;
  if (i < n) {
    const uint32_t ps = pt_slot[i];
    f = ps != kNoSlot && slots[ps].vid == (uint32_t)i;
  }
  const unsigned b = __ballot_sync(0xFFFFFFFFu, f);
  if ((threadIdx.x & 31) == 0 && (i >> 5) <= (n >> 5)) bitmap[i >> 5] = b;
}

__global__ void popc_words_kernel(const uint32_t* __restrict__ bitmap, int64_t n_words,
                                  uint32_t* __restrict__ out) {
  for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < n_words;
       w += (int64_t)gridDim.x * blockDim.x)
    out[w] = (uint32_t)__popc(bitmap[w]);
}

// Number of first points before point i (wscan: the exclusive scan of the words'
// popcounts; the word of index n exists and has no bit at or above n).
__device__ __forceinline__ uint32_t first_rank(const uint32_t* __restrict__ bitmap,
                                               const uint32_t* __restrict__ wscan, uint32_t i) {
  const uint32_t w = i >> 5;
  return wscan[w] + (uint32_t)__popc(bitmap[w] & ((1u << (i & 31u)) - 1u));
}

// Each first point gives its voxel its id: the voxel's count and key are
// recorded by id and the id replaces the index in the build-table slot.
__global__ void assign_ids_kernel(const uint32_t* __restrict__ bitmap,
                                  const uint32_t* __restrict__ wscan, int64_t n,
                                  const uint32_t* __restrict__ pt_slot, Slot* slots,
                                  uint32_t* __restrict__ vcount,
                                  unsigned long long* __restrict__ vkeys) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (!((bitmap[i >> 5] >> (i & 31)) & 1u)) continue;
    const uint32_t id = first_rank(bitmap, wscan, (uint32_t)i);
    Slot* sl = slots + pt_slot[i];
    vcount[id] = sl->count;
    vkeys[id] = sl->key;
    sl->vid = id;
  }
}

// vbase[m] = voxels of the maps before m; vbase[n_maps] and *n_vox = all.  With vmask
// (a rebuild) also each map's lookup-table mask.  The scatter's counters start at zero.
__device__ __forceinline__ void map_ranges(int m, int32_t n_maps, int64_t n_total,
                                           const int64_t* __restrict__ point_off,
                                           const uint32_t* bitmap, const uint32_t* wscan,
                                           uint32_t* __restrict__ vbase,
                                           uint32_t* __restrict__ n_vox,
                                           const int64_t* __restrict__ vslot_base,
                                           uint32_t* __restrict__ vmask,
                                           uint32_t* __restrict__ dropped) {
  const uint32_t v =
      first_rank(bitmap, wscan, (uint32_t)(m < n_maps ? point_off[m] : n_total));
  vbase[m] = v;
  if (m < n_maps) dropped[m] = 0u;
  if (m == n_maps) {
    *n_vox = v;
  } else if (vmask) {
    const uint32_t next =
        first_rank(bitmap, wscan, (uint32_t)(m + 1 < n_maps ? point_off[m + 1] : n_total));
    vmask[m] = table_capacity(next - v, (uint32_t)(vslot_base[m + 1] - vslot_base[m])) - 1u;
  }
}
__global__ void vbase_kernel(int32_t n_maps, int64_t n_total, const int64_t* __restrict__ point_off,
                             const uint32_t* __restrict__ bitmap,
                             const uint32_t* __restrict__ wscan, uint32_t* __restrict__ vbase,
                             uint32_t* __restrict__ n_vox, const int64_t* __restrict__ vslot_base,
                             uint32_t* __restrict__ vmask, int32_t* status,
                             uint32_t* __restrict__ dropped) {
  if (blockIdx.x == 0 && threadIdx.x == 0) take_status(status);
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m <= n_maps)
    map_ranges(m, n_maps, n_total, point_off, bitmap, wscan, vbase, n_vox, vslot_base, vmask,
               dropped);
}

// The words' popcounts scanned and the maps' ranges, by one CTA: five launches in one
// while the words are few (200,000 points: 2 us; kNumberWords take 6 us, the scan's
// launches for as many 9).
constexpr int64_t kNumberWords = 32768;
constexpr int kNumberThreads = 1024, kNumberPer = 8;
__global__ void __launch_bounds__(kNumberThreads) number_kernel(
    const uint32_t* bitmap, int64_t n_words, uint32_t* wscan, int32_t n_maps, int64_t n_total,
    const int64_t* __restrict__ point_off, uint32_t* __restrict__ vbase,
    uint32_t* __restrict__ n_vox, const int64_t* __restrict__ vslot_base,
    uint32_t* __restrict__ vmask, int32_t* status, uint32_t* __restrict__ dropped) {
  __shared__ uint32_t total;
  if (threadIdx.x == 0) take_status(status);
  uint32_t carry = 0u;
  for (int64_t w0 = 0; w0 < n_words; w0 += kNumberThreads * kNumberPer) {
    const int64_t a = w0 + (int64_t)threadIdx.x * kNumberPer;
    uint32_t c[kNumberPer], sum = 0u;
#pragma unroll
    for (int k = 0; k < kNumberPer; ++k) {
      c[k] = a + k < n_words ? (uint32_t)__popc(bitmap[a + k]) : 0u;
      sum += c[k];
    }
    uint32_t run = carry + block_exclusive<kNumberThreads>(sum, &total);
#pragma unroll
    for (int k = 0; k < kNumberPer; ++k) {
      if (a + k < n_words) wscan[a + k] = run;
      run += c[k];
    }
    carry += total;
    __syncthreads();  // the CTA's words are visible to it; `total` may be rewritten
  }
  for (int m = threadIdx.x; m <= n_maps; m += kNumberThreads)
    map_ranges(m, n_maps, n_total, point_off, bitmap, wscan, vbase, n_vox, vslot_base, vmask,
               dropped);
}

// One thread per element (no grid-stride cap): CTAs are dispatched roughly in
// index order, so the maps being worked on at any moment are a few consecutive
// ones whose clouds and tables stay in L2 while their random accesses land.
int grid_for(int64_t n, int threads) {
  const int64_t g = (n + threads - 1) / threads;
  return (int)std::max<int64_t>(1, std::min<int64_t>(g, 0x7FFFFFFF));
}

}  // namespace

size_t scan_tmp_elems(int64_t n_max) { return (size_t)((n_max + kScanTile - 1) / kScanTile) + 1; }

int launch_exclusive_scan(const uint32_t* in, uint32_t* out, int64_t n_max, const uint32_t* n_dev,
                          uint32_t* block_tmp, uint32_t* total_dev, cudaStream_t st) {
  if (n_max <= 0) {
    if (total_dev) VGICP_CUDA_TRY(cudaMemsetAsync(total_dev, 0, sizeof(uint32_t), st));
    return VGICP_OK;
  }
  const int64_t nb = (n_max + kScanTile - 1) / kScanTile;
  scan_tile_sums_kernel<<<(unsigned)nb, kScanThreads, 0, st>>>(in, n_max, n_dev, block_tmp);
  scan_sums_kernel<<<1, kScanSumsThreads, 0, st>>>(block_tmp, nb, total_dev);
  scan_tiles_kernel<<<(unsigned)nb, kScanThreads, 0, st>>>(in, out, n_max, n_dev, block_tmp);
  VGICP_CUDA_TRY(cudaGetLastError());
  count_launches(3);
  return VGICP_OK;
}

// First build of a set: reads the per-map voxel counts back (one stream
// synchronization) and allocates each map's lookup-table region at
// next_pow2(max(16, kLookupLoad V, 2 n)) slots; a build uses
// min(next_pow2(kLookupLoad V), region) of it.
int size_lookup_tables(MapSet* s, cudaStream_t st) {
  std::vector<uint32_t> vb((size_t)s->n_maps + 1);
  VGICP_CUDA_TRY(cudaMemcpyAsync(vb.data(), s->d_vbase, sizeof(uint32_t) * vb.size(),
                                 cudaMemcpyDeviceToHost, st));
  VGICP_CUDA_TRY(cudaStreamSynchronize(st));
  s->vslot_base.assign((size_t)s->n_maps + 1, 0);
  s->vox.assign((size_t)s->n_maps, 0u);
  int64_t total = 0;
  for (int32_t m = 0; m < s->n_maps; ++m) {
    const uint64_t V = vb[m + 1] >= vb[m] ? vb[m + 1] - vb[m] : 0;
    // at least 2 n slots, so that a rebuild with up to V = n voxels still fits
    // (load factor <= 1/2); the first build's capacity next_pow2(kLookupLoad V)
    // when larger
    const uint64_t nm = (uint64_t)(s->point_off[m + 1] - s->point_off[m]);
    uint64_t c = 16;
    while (c < kLookupLoad * V || c < 2 * nm) c <<= 1;
    s->vslot_base[m] = total;
    s->vox[m] = (uint32_t)V;
    total += (int64_t)c;
  }
  s->vslot_base[s->n_maps] = total;
  s->avg_list = s->n_total / std::max<int64_t>(1, (int64_t)vb[(size_t)s->n_maps]);
  if (total >= (int64_t)0xFFFFFFFFll)
    return set_error(VGICP_ERR_INVALID_ARG, "more than 2^32-1 lookup slots in one batch");
  cudaError_t e = device_malloc(&s->d_vblock, sizeof(VSlot) * (size_t)total, nullptr, false);
  if (e != cudaSuccess) {
    cudaGetLastError();
    s->d_vblock = nullptr;
    return set_error(VGICP_ERR_OOM, "lookup table allocation of " +
                                        std::to_string(sizeof(VSlot) * (size_t)total) +
                                        " bytes failed");
  }
  s->d_vslots = static_cast<VSlot*>(s->d_vblock);
  s->vcap_total = total;
  VGICP_CUDA_TRY(cudaMemcpy(s->d_vslot_base, s->vslot_base.data(),
                            sizeof(int64_t) * s->vslot_base.size(), cudaMemcpyHostToDevice));
  return VGICP_OK;
}

int launch_build(MapSet* s, const float* points, const float* covs, cudaStream_t st) {
  const int64_t n = s->n_total;
  // was_built: the tables hold only the previous build's voxels (a build that
  // stops on an error leaves `built` cleared, so the next one starts over)
  const bool was_built = s->built;
  s->built = false;
  if (!was_built) {
    init_slots_kernel<<<grid_for(s->cap_total, kThreads), kThreads, 0, st>>>(
        s->d_slots, s->cap_total, s->d_status);
    count_launches(1);
  }
  if (n == 0) {
    VGICP_CUDA_TRY(cudaMemsetAsync(s->d_num_voxels, 0, sizeof(uint32_t), st));
    VGICP_CUDA_TRY(cudaMemsetAsync(s->d_vbase, 0, sizeof(uint32_t) * (s->n_maps + 1), st));
    if (!s->d_vblock) {
      const int rc = size_lookup_tables(s, st);
      if (rc != VGICP_OK) return rc;
    }
    vslot_init_kernel<<<dim3(1, s->n_maps), kThreads, 0, st>>>(s->d_vslot_base, s->d_vbase,
                                                              s->d_vslots, s->d_vmask,
                                                              was_built ? 0 : 1);
    VGICP_CUDA_TRY(cudaGetLastError());
    count_launches(1);
    s->built = true;
    return VGICP_OK;
  }
  const float inv_r = (float)(1.0 / s->resolution);
  const int g = grid_for(n, kThreads);
  const int reset = was_built ? std::max(1, g / (kResetEvery - 1)) : 0;
  insert_kernel<<<g + reset, kThreads, 0, st>>>(
      points, n, s->d_point_off, s->n_maps, s->d_slot_base, s->d_cap_mask, inv_r, s->resolution,
      s->max_probe, s->d_slots, s->d_pt_slot, s->d_status + 1, reset, s->d_num_voxels,
      s->d_lslot_of, s->d_vslots);
  // voxel ids in order of first appearance: first points marked in d_flag, the
  // words' popcounts scanned in d_vfill (both dead afterwards)
  int rc = VGICP_OK;
  {
    const int64_t n_words = n / 32 + 1;
    uint32_t* bitmap = s->d_flag;
    uint32_t* wscan = s->d_vfill;
    uint32_t* vmask = was_built ? s->d_vmask : nullptr;  // the first build sizes the tables below
    first_bits_kernel<<<grid_for(32 * n_words, kThreads), kThreads, 0, st>>>(s->d_pt_slot,
                                                                           s->d_slots, n, bitmap);
    if (n_words <= kNumberWords) {
      number_kernel<<<1, kNumberThreads, 0, st>>>(bitmap, n_words, wscan, s->n_maps, n,
                                                  s->d_point_off, s->d_vbase, s->d_num_voxels,
                                                  s->d_vslot_base, vmask, s->d_status,
                                                  s->d_dropped);
    } else {
      popc_words_kernel<<<grid_for(n_words, kThreads), kThreads, 0, st>>>(bitmap, n_words, wscan);
      rc = launch_exclusive_scan(wscan, wscan, n_words, nullptr, s->d_scan_tmp, nullptr, st);
      if (rc != VGICP_OK) return rc;
      vbase_kernel<<<(s->n_maps + 1 + 127) / 128, 128, 0, st>>>(
          s->n_maps, n, s->d_point_off, bitmap, wscan, s->d_vbase, s->d_num_voxels,
          s->d_vslot_base, vmask, s->d_status, s->d_dropped);
      count_launches(1);
    }
    assign_ids_kernel<<<g, kThreads, 0, st>>>(bitmap, wscan, n, s->d_pt_slot, s->d_slots,
                                              s->d_vcount, s->d_vkeys);
    VGICP_CUDA_TRY(cudaGetLastError());
    count_launches(3);
  }
  if (!s->d_vblock) {
    rc = size_lookup_tables(s, st);
    if (rc != VGICP_OK) return rc;
  }
  // Morton order of the voxels (chunks of a map), the list offsets in that order,
  // the lists, then the per-voxel sums (which also write the grouped clouds).
  // d_vfill (the numbering's word scan) is dead after the id assignment.
  uint32_t* vorder = s->d_voff;
  // the lists' (base << 32 | fill) words, by voxel: in the record storage, which
  // finalize fills only after the scatter (8 of its 48 B per voxel)
  unsigned long long* bfill = reinterpret_cast<unsigned long long*>(s->d_recs);
  // a cluster per chunk while that leaves two SMs or more to a chunk (figures at the
  // kernel)
  const uint32_t* chunk_points = nullptr;
  if (*std::max_element(s->vox.begin(), s->vox.end()) > kOwnCount) {
    chunk_points_kernel<<<(unsigned)s->n_chunks, kThreads, 0, st>>>(
        s->d_chunks, s->d_vbase, s->d_vcount, s->d_chunk_points);
    count_launches(1);
    chunk_points = s->d_chunk_points;
  }
  rc = 2 * s->n_chunks <= device_sm_count()
           ? launch_sort<8, 256>(s, chunk_points, vorder, bfill, st)
           : launch_sort<1, 1024>(s, chunk_points, vorder, bfill, st);
  if (rc != VGICP_OK) return rc;
  VGICP_CUDA_TRY(cudaGetLastError());
  scatter_kernel<<<g, kThreads, 0, st>>>(n, s->d_pt_slot, s->d_slots, bfill, s->d_plist,
                                         s->d_point_off, s->n_maps, s->d_dropped);
  if (!was_built) {  // empty the whole lookup region and set the masks
    int64_t max_cap = 16;
    for (int32_t m = 0; m < s->n_maps; ++m)
      max_cap = std::max<int64_t>(max_cap, s->vslot_base[m + 1] - s->vslot_base[m]);
    const unsigned gx = (unsigned)std::min<int64_t>(64, (max_cap + kThreads - 1) / kThreads);
    vslot_init_kernel<<<dim3(gx, s->n_maps), kThreads, 0, st>>>(s->d_vslot_base, s->d_vbase,
                                                               s->d_vslots, s->d_vmask, 1);
    count_launches(1);
  }
  // sums, records, grouped clouds and the lookup tables
  // large sets of short lists (the first build's average) keep the kernel that sorts
  // them a thread per voxel (figures at finalize_long_kernel)
  const auto finalize =
      s->avg_list > 10 || n < 500000 ? finalize_long_kernel : finalize_kernel;
  finalize<<<g, kFinThreads, 0, st>>>(
      n, s->d_num_voxels, points, covs, vorder, s->d_vcount, s->d_goff, s->d_plist, s->d_recs,
      s->d_gpts, s->d_gcovs, s->d_vkeys, s->n_maps, s->d_vbase, s->d_vslot_base, s->d_vmask,
      s->max_probe, s->d_vslots, s->d_lslot_of, s->d_status);
  VGICP_CUDA_TRY(cudaGetLastError());
  count_launches(4);  // insert, sort, scatter, finalize
  s->built = true;
  return VGICP_OK;
}

}  // namespace vgicp
