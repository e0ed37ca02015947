// Occupancy blocks for the 27-neighbour linearization: the voxels of a target map
// regrouped by blocks of 4 x 4 x 4, built by the call that uses them.
//
// A source point's 3 x 3 x 3 neighbourhood lies in 1 to 8 blocks (3.4 on average), so
// the occupied neighbours come from a few block masks instead of 27 hash probes, and
// the Gaussians of a block are contiguous.  The probes took 8.4 of the kernel's 12.9 ms
// on 48 large-map submaps (96M source points).
//
// Per map: a hash table of blocks (key, 64-bit occupancy, first record) and the
// records (mu', L).  Both are sized from the voxel count of the map's first build; a
// map rebuilt with many more voxels may not fit, which its flag reports: its work
// items are then left to the kernel that probes voxel by voxel.
//
//   insert  per voxel: its block, claimed or found; its bit in the mask
//   place   per block: a range of records
//   fill    per voxel: its Gaussian to the block's first record + rank in the mask
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "vgicp_device.cuh"
#include "vgicp_internal.h"

namespace vgicp {
namespace {

constexpr int kThreads = 256;
__device__ __forceinline__ void leave_to_probes(const BlockMap& M) {
  M.state[0] = 1u;
  *M.any = 1u;
}
// Whether the map has been left to the probes (by this kernel perhaps, and meanwhile).
__device__ __forceinline__ bool is_left(const BlockMap& M) {
  return *(const volatile uint32_t*)M.state != 0u;
}

// n more blocks: past three quarters full, absent blocks take long to rule out.
__device__ __forceinline__ void count_blocks(const BlockMap& M, uint32_t n) {
  if (atomicAdd(M.state + 2, n) + n > M.mask / 4u * 3u) leave_to_probes(M);
}

// Blocks are counted per CTA and 32 at a time: one by one, the kernel took 340 us for a map
// of 200,000 isolated voxels, and takes 236 so.
constexpr uint32_t kCountStep = 32;
__global__ void __launch_bounds__(kThreads) block_insert_kernel(const BlockMap* __restrict__ maps) {
  const BlockMap M = maps[blockIdx.y];
  __shared__ uint32_t n_new;
  if (threadIdx.x == 0) n_new = 0u;
  __syncthreads();
  const uint32_t v0 = M.vbase[0], V = M.vbase[1] - v0;
  if (V > M.rec_cap) {  // does not fit
    if (blockIdx.x == 0 && threadIdx.x == 0) leave_to_probes(M);
    return;
  }
  const unsigned long long fm = (1ull << kKeyBits) - 1ull;
  for (uint32_t i = blockIdx.x * kThreads + threadIdx.x; i < V; i += gridDim.x * kThreads) {
    const unsigned long long k = M.vkeys[v0 + i];
    const int kx = (int)((k >> (2 * kKeyBits)) & fm) - kKeyBias;
    const int ky = (int)((k >> kKeyBits) & fm) - kKeyBias;
    const int kz = (int)(k & fm) - kKeyBias;
    uint32_t found = kNoSlot;
    if (M.lslot_of[v0 + i] != kNoSlot) {
      const unsigned long long key = block_key(kx >> 2, ky >> 2, kz >> 2);
      uint32_t h = hash_key(kx >> 2, ky >> 2, kz >> 2) & M.mask;
      for (int p = 0; p < kBlockProbes; ++p) {
        const unsigned long long cur = atomicCAS(&M.table[h].key, 0ull, key);
        if (cur == 0ull || cur == key) {
          found = h;
          if (cur == 0ull && (atomicAdd(&n_new, 1u) + 1u) % kCountStep == 0u)
            count_blocks(M, kCountStep);
          break;
        }
        // a map of scattered voxels, a block or nearly one to each, fills its table; then
        // no voxel looks through 256 slots (a check before every voxel, here and in the
        // kernels below, cost maps that fit 2 % of a call of 0.9 ms)
        if ((p & 7) == 7 && is_left(M)) break;
        h = (h + 1) & M.mask;
      }
      if (found != kNoSlot)
        atomicOr(&M.table[found].bits,
                 1ull << ((kz & 3) * 16 + (ky & 3) * 4 + (kx & 3)));
      else
        leave_to_probes(M);
    }
    M.block_of[i] = found;
  }
  __syncthreads();
  if (threadIdx.x == 0 && n_new % kCountStep != 0u) count_blocks(M, n_new % kCountStep);
}

__global__ void __launch_bounds__(kThreads) block_place_kernel(const BlockMap* __restrict__ maps) {
  const BlockMap M = maps[blockIdx.y];
  __shared__ uint32_t warp_sum[kThreads / 32];
  __shared__ uint32_t base;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (uint32_t s0 = blockIdx.x * kThreads; s0 <= M.mask; s0 += gridDim.x * kThreads) {
    const uint32_t s = s0 + threadIdx.x;
    const uint32_t cnt = s <= M.mask ? (uint32_t)__popcll(M.table[s].bits) : 0u;
    uint32_t inc = cnt;
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
      base = t > 0u ? atomicAdd(M.state + 1, t) : 0u;
    }
    __syncthreads();
    // (at most rec_cap records in all: one per voxel, and V <= rec_cap)
    if (cnt > 0u) M.table[s].first = base + warp_sum[w] + inc - cnt;
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kThreads) block_fill_kernel(const BlockMap* __restrict__ maps) {
  const BlockMap M = maps[blockIdx.y];
  const uint32_t v0 = M.vbase[0], V = M.vbase[1] - v0;
  if (V > M.rec_cap) return;
  const unsigned long long fm = (1ull << kKeyBits) - 1ull;
  for (uint32_t i = blockIdx.x * kThreads + threadIdx.x; i < V; i += gridDim.x * kThreads) {
    const uint32_t s = M.block_of[i];
    if (s == kNoSlot) continue;
    const unsigned long long k = M.vkeys[v0 + i];
    const int bit = (int)(k & fm & 3ull) * 16 + (int)((k >> kKeyBits) & 3ull) * 4 +
                    (int)((k >> (2 * kKeyBits)) & 3ull);  // (the key bias is a multiple of 4)
    const BlockSlot b = M.table[s];
    const uint32_t r = b.first + (uint32_t)__popcll(b.bits & ((1ull << bit) - 1ull));
    const VSlot* t = M.vslots + M.lslot_of[v0 + i];
    M.recs[3 * r + 0] = make_float4(t->mu[0], t->mu[1], t->mu[2], 0.f);
    M.recs[3 * r + 1] = make_float4(t->cov[0], t->cov[1], t->cov[2], t->cov[3]);
    M.recs[3 * r + 2] = make_float4(t->cov[4], t->cov[5], 0.f, 0.f);
  }
}

}  // namespace

uint32_t block_capacity(int64_t voxels) {
  uint64_t c = 64;
  while (c < (uint64_t)voxels / 2) c <<= 1;
  return (uint32_t)c;
}

int launch_blocks(const BlockMap* d_maps, int32_t n_maps, int64_t max_voxels, cudaStream_t st) {
  // CTAs per map: 512 voxels each (two random reads of each voxel to hide)
  const unsigned gx =
      (unsigned)std::min<int64_t>(1024, std::max<int64_t>(1, max_voxels / (2 * kThreads)));
  const dim3 grid(gx, (unsigned)n_maps);
  block_insert_kernel<<<grid, kThreads, 0, st>>>(d_maps);
  block_place_kernel<<<grid, kThreads, 0, st>>>(d_maps);
  block_fill_kernel<<<grid, kThreads, 0, st>>>(d_maps);
  VGICP_CUDA_TRY(cudaGetLastError());
  count_launches(3);
  return VGICP_OK;
}

}  // namespace vgicp
