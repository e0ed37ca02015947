// Point covariances from k nearest neighbours (arXiv 2202.00242 Sec. III-C: each
// input point is modelled as a Gaussian whose covariance comes from its
// neighbouring points; GICP-style regularisation).
//
// For a batch of clouds given by offsets (neighbours are searched within each
// cloud only):
//   prep      per cloud, an empty cell table and the grid cell size h: the caller's,
//             or sqrt(A / n * k) from the cloud's bounding box (A = the sum of the
//             box's face areas), a cell holding about k points on a surface
//   insert    per point: exact cell key floor(x / h) (binary64 semantics),
//             open-addressing insert into the cloud's cell table, count
//   alloc, scatter   places for the cells' members; the points in cell order
//             (float4: x, y, z, point index), so a cell's members are contiguous
//   search    per point: the cells at Chebyshev ring distance s = 0, 1, ... from
//             its own, until the k-th best candidate lies within s h (any point
//             beyond lies farther than s h).  The order is (d^2, index) with
//             d^2 = ((dx dx + dy dy) + dz dz) in binary64 from the exact
//             float-to-double differences.  Candidates are selected by float32 d^2
//             (within 2^-21 of the binary64 value); values closer than that bound
//             allows are decided in binary64.
//   covariance  mean of the k neighbours and their scatter about it, in float32
//             relative to the query point, the eigenvector v of the smallest
//             eigenvalue by cyclic Jacobi (float32, on the trace-normalised matrix), and
//             C = V diag(1, 1, eps) V^T = I - (1 - eps) v v^T.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "vgicp.h"
#include "vgicp_device.cuh"
#include "vgicp_internal.h"

namespace vgicp {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxProbe = 256;

struct __align__(16) CellSlot {
  unsigned long long key;
  uint32_t start;  // one past the cell's last member in the cell-ordered arrays
  uint32_t count;
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

// Order-preserving bits of a float (for atomicMin / atomicMax), and back.
__device__ __forceinline__ uint32_t ordered_bits(float v) {
  const uint32_t b = __float_as_uint(v);
  return b ^ ((b >> 31) ? 0xFFFFFFFFu : 0x80000000u);
}
__device__ __forceinline__ float from_ordered(uint32_t b) {
  return __uint_as_float(b ^ ((b >> 31) ? 0x80000000u : 0xFFFFFFFFu));
}

// Points per cell the automatic cell size aims at, as a multiple of k, were the
// cloud spread evenly over half the faces of its bounding box.  Smaller cells mean
// fewer candidates and more queries that need a second ring: 64 submaps (3.3M
// points, k = 10), first / second search kernel at 0.7: 992 / 606 us, 0.8: 984 /
// 332, 1.0: 1022 / 178, 1.3: 1146 / 80, 1.7: 1364 / 149; with k = 20 (20 submaps,
// 0.95M points, the whole call) 1.0: 1347 us, 1.3: 1887 (cells with more than 512
// candidates around them).
constexpr double kCellFill = 1.0;

// Per-cloud set-up, gridDim.y CTAs per cloud: empties the cloud's cell table
// and, for the automatic cell size, takes the bounding box; the cloud's last CTA
// turns it into h and float32(1 / h).
//   bbox: 6 words per cloud (min xyz, max xyz as ordered bits, set by the host to
//         those of +inf / -inf); done: CTAs of the cloud that have finished.
constexpr int kPrepParts = 1024;  // at most
__global__ void prep_kernel(const float* __restrict__ pts, const int64_t* __restrict__ off,
                            int32_t k, double cell, const int64_t* __restrict__ slot_base,
                            const uint32_t* __restrict__ cap_mask, CellSlot* slots,
                            uint32_t* bbox, uint32_t* done, double* __restrict__ h_out,
                            float* __restrict__ inv_out, float* __restrict__ reach2_out) {
  const int c = blockIdx.x;
  const int64_t a = off[c], b = off[c + 1];
  const int64_t step = (int64_t)gridDim.y * blockDim.x;
  const int64_t t0 = (int64_t)blockIdx.y * blockDim.x + threadIdx.x;
  uint4* tab = reinterpret_cast<uint4*>(slots + slot_base[c]);
  const int64_t cap = (int64_t)cap_mask[c] + 1;
  for (int64_t s = t0; s < cap; s += step) tab[s] = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0u, 0u);
  if (cell > 0.0) {
    if (blockIdx.y == 0 && threadIdx.x == 0) {
      h_out[c] = cell;
      inv_out[c] = (float)(1.0 / cell);
      reach2_out[c] = __double2float_rd(cell * cell);
    }
    return;
  }
  float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (int64_t i = a + t0; i < b; i += step)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float v = pts[3 * i + d];
      lo[d] = fminf(lo[d], v);
      hi[d] = fmaxf(hi[d], v);
    }
  __shared__ float part[6][kThreads / 32];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo[d] = fminf(lo[d], __shfl_xor_sync(0xFFFFFFFFu, lo[d], o));
      hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xFFFFFFFFu, hi[d], o));
    }
    if ((threadIdx.x & 31) == 0) {
      part[d][threadIdx.x >> 5] = lo[d];
      part[3 + d][threadIdx.x >> 5] = hi[d];
    }
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    float l = part[d][0], u = part[3 + d][0];
    for (int w = 1; w < kThreads / 32; ++w) {
      l = fminf(l, part[d][w]);
      u = fmaxf(u, part[3 + d][w]);
    }
    atomicMin(bbox + 6 * c + d, ordered_bits(l));
    atomicMax(bbox + 6 * c + 3 + d, ordered_bits(u));
  }
  __threadfence();
  if (atomicAdd(done + c, 1u) + 1u != gridDim.y) return;
  __threadfence();
  double e[3], far = 0.0;
  for (int d = 0; d < 3; ++d) {
    const double l = (double)from_ordered(__ldcg(bbox + 6 * c + d));
    const double u = (double)from_ordered(__ldcg(bbox + 6 * c + 3 + d));
    e[d] = b > a ? u - l : 1.0;
    if (b > a) far = fmax(far, fmax(fabs(l), fabs(u)));
  }
  const double area = fmax(e[0] * e[1] + e[1] * e[2] + e[0] * e[2], 1e-12);
  const double per = area / (double)(b > a ? b - a : 1) * k;
  // the cell of 2 k points bounds what coordinates are accepted (|x / h| below
  // 2^20); the search itself prefers smaller cells, which must not refuse any
  // cloud that those accept
  const double h_max = fmax(sqrt(per * 2.0), 1e-3);
  const double h_min = far * (1.000001 / 1048576.0);
  const double h = fmin(h_max, fmax(fmax(sqrt(per * kCellFill), 1e-3), h_min));
  h_out[c] = h;
  inv_out[c] = (float)(1.0 / h);
  reach2_out[c] = __double2float_rd(h * h);
}

__device__ __forceinline__ void cell_key(const float* p, double h, float inv, int& kx, int& ky,
                                         int& kz) {
  kx = axis_key_target(p[0], inv, h);
  ky = axis_key_target(p[1], inv, h);
  kz = axis_key_target(p[2], inv, h);
}

__global__ void cell_insert_kernel(const float* __restrict__ pts, int64_t n,
                                   const int64_t* __restrict__ off, int32_t n_clouds,
                                   const double* __restrict__ hc, const float* __restrict__ invc,
                                   const int64_t* __restrict__ slot_base,
                                   const uint32_t* __restrict__ cap_mask, CellSlot* slots,
                                   uint32_t* __restrict__ pt_slot, int32_t* status) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int c = cloud_of(off, n_clouds, i);
    int kx, ky, kz;
    cell_key(pts + 3 * i, hc[c], invc[c], kx, ky, kz);
    if (!key_in_range(kx) || !key_in_range(ky) || !key_in_range(kz)) {
      pt_slot[i] = kNoSlot;
      set_status(status, VGICP_ERR_KEY_RANGE);
      continue;
    }
    const unsigned long long key = pack_key(kx, ky, kz);
    const uint32_t mask = cap_mask[c];
    CellSlot* t = slots + slot_base[c];
    uint32_t h = hash_key(kx, ky, kz) & mask;
    uint32_t found = kNoSlot;
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
      h = (h + 1) & mask;
    }
    if (found == kNoSlot) {
      pt_slot[i] = kNoSlot;
      set_status(status, VGICP_ERR_HASH_FULL);
      continue;
    }
    atomicAdd(&t[found].count, 1u);
    pt_slot[i] = (uint32_t)(slot_base[c] + found);
  }
}

// Places of the cells' members: each CTA takes kAllocPer slots per thread, sums
// their counts and reserves one range for them all.  (Which cells come first does
// not matter: a query's result does not depend on the order it sees candidates in.)
constexpr int kAllocPer = 4;
__global__ void __launch_bounds__(kThreads) cell_alloc_kernel(CellSlot* slots, int64_t cap_total,
                                                              uint32_t* cursor) {
  __shared__ uint32_t warp_sum[kThreads / 32];
  __shared__ uint32_t base;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t s0 = (int64_t)blockIdx.x * (kThreads * kAllocPer) + threadIdx.x;
  uint32_t cnt[kAllocPer], sum = 0u;
#pragma unroll
  for (int j = 0; j < kAllocPer; ++j) {
    const int64_t s = s0 + (int64_t)j * kThreads;
    cnt[j] = s < cap_total ? slots[s].count : 0u;
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
    for (int i = 0; i < kThreads / 32; ++i) {
      const uint32_t x = warp_sum[i];
      warp_sum[i] = t;
      t += x;
    }
    base = t > 0u ? atomicAdd(cursor, t) : 0u;
  }
  __syncthreads();
  uint32_t run = base + warp_sum[w] + inc - sum;
#pragma unroll
  for (int j = 0; j < kAllocPer; ++j) {
    if (cnt[j] > 0u) slots[s0 + (int64_t)j * kThreads].start = run;
    run += cnt[j];
  }
}

// The points in cell order: (x, y, z, point index), and the cell of each.  The
// cell's start doubles as its fill counter and ends at the cell's end.
__global__ void cell_scatter_kernel(const float* __restrict__ pts, int64_t n,
                                    const uint32_t* __restrict__ pt_slot, CellSlot* slots,
                                    float4* __restrict__ members,
                                    uint32_t* __restrict__ member_slot) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t s = pt_slot[i];
    if (s == kNoSlot) continue;
    const uint32_t pos = atomicAdd(&slots[s].start, 1u);
    members[pos] = make_float4(pts[3 * i], pts[3 * i + 1], pts[3 * i + 2],
                               __uint_as_float((uint32_t)i));
    member_slot[pos] = s;
  }
}

// Candidate order: (d^2, index), lexicographic.  Non-negative binary64 values
// order like their bit patterns read as unsigned integers, so the comparison
// runs on the integer pipe (binary64 arithmetic is scarce on this GPU).
__device__ __forceinline__ bool before(unsigned long long d, uint32_t j, unsigned long long e,
                                       uint32_t l) {
  return d < e || (d == e && j < l);
}

// Smallest-eigenvalue eigenvector of a symmetric 3x3 matrix (upper triangle a)
// by cyclic Jacobi rotations (float32).
__device__ void smallest_eigvec(const float a_in[6], float v_out[3]) {
  float A[3][3] = {{a_in[0], a_in[1], a_in[2]}, {a_in[1], a_in[3], a_in[4]},
                   {a_in[2], a_in[4], a_in[5]}};
  float V[3][3] = {{1.f, 0.f, 0.f}, {0.f, 1.f, 0.f}, {0.f, 0.f, 1.f}};
  for (int sweep = 0; sweep < 12; ++sweep) {
    const float off = fabsf(A[0][1]) + fabsf(A[0][2]) + fabsf(A[1][2]);
    if (off < 1e-12f * (fabsf(A[0][0]) + fabsf(A[1][1]) + fabsf(A[2][2])) || off == 0.f) break;
#pragma unroll
    for (int pq = 0; pq < 3; ++pq) {
      const int p = pq == 2 ? 1 : 0, q = pq == 0 ? 1 : 2;
      const float apq = A[p][q];
      if (apq == 0.f) continue;
      const float theta = (A[q][q] - A[p][p]) / (2.f * apq);
      const float t = copysignf(1.f, theta) / (fabsf(theta) + sqrtf(theta * theta + 1.f));
      const float c = rsqrtf(t * t + 1.f), s = t * c;
#pragma unroll
      for (int r = 0; r < 3; ++r) {  // A <- A J
        const float arp = A[r][p], arq = A[r][q];
        A[r][p] = c * arp - s * arq;
        A[r][q] = s * arp + c * arq;
      }
#pragma unroll
      for (int r = 0; r < 3; ++r) {  // A <- J^T A
        const float apr = A[p][r], aqr = A[q][r];
        A[p][r] = c * apr - s * aqr;
        A[q][r] = s * apr + c * aqr;
      }
#pragma unroll
      for (int r = 0; r < 3; ++r) {  // V <- V J
        const float vrp = V[r][p], vrq = V[r][q];
        V[r][p] = c * vrp - s * vrq;
        V[r][q] = s * vrp + c * vrq;
      }
    }
  }
  int m = 0;
  if (A[1][1] < A[0][0]) m = 1;
  if (A[2][2] < (m == 1 ? A[1][1] : A[0][0])) m = 2;
  float n2 = 0.f;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    v_out[r] = m == 0 ? V[r][0] : m == 1 ? V[r][1] : V[r][2];
    n2 += v_out[r] * v_out[r];
  }
  const float s = rsqrtf(n2);
#pragma unroll
  for (int r = 0; r < 3; ++r) v_out[r] *= s;
}

// ---------------------------------------------------------------------------
// The search, in three kernels.
//
// select: one warp takes 32 consecutive members (cell order) and works through
// their cells one after the other; the queries of one cell share their candidates,
// the members of the 3x3x3 block of cells around it:
//   look up   one neighbour cell per lane (27 probes in flight together);
//   load      the cells' members into the warp's tile in shared memory;
//   keep      lane = (query, part of the candidates); each lane keeps the CAP = K + 2
//             smallest float32 d^2 of its part in sorted registers, the low 9 bits
//             of each replaced by the candidate's number (a min and a max per
//             value, no branch), and the parts of a query are merged by shuffles.
// A query is finished when its k-th value lies within the reach of the block and
// the last kept one is larger than the k-th by two steps of the shortened value:
// then the kept ones hold every candidate that can be among the k nearest.  The
// lanes then take one query each, put its list in order (float32 d^2, each value
// further from the next than the error bound, so the order is the binary64 one)
// and sum the scatter matrix.  Everything else is left to the next kernel:
// queries that need cells further out, cells with more than 512 candidates around
// them, and near-ties.
//
// rest: one warp per query left over.  Ring after ring until the k-th value is
// within reach (or the whole table, once a ring has more cells than the table has
// slots); the candidates at or below the k-th value are collected and ranked by
// binary64 (d^2, index).
//
// eigenvectors: one thread per point turns its scatter matrix, left in the point's
// own place of the output, into the covariance.
//
// What bounds them: instruction issue (in select about 20 min / max instructions
// per candidate and 32 / parts queries, and the merges), then the latency of
// look-up and load at the start of each cell.  A thread per query with a sorted
// insertion per candidate, as this was before, took 9.31 ms for 3.3M points in 64
// submaps and 247 us for one scan of 20,000 (a warp executes the insertion whenever
// any lane needs it, and 27 dependent look-ups one after the other).
// ---------------------------------------------------------------------------

// Float32 squared distances are within 2^-21 of the binary64 ones (the
// differences and the fused sum each round once); thresholds and comparisons
// allow 2^-18.  Below kF2Tiny that bound may fail (underflow): binary64 decides.
constexpr float kF2Up = 1.0000038146972656f;  // 1 + 2^-18
constexpr float kF2Tiny = 1e-30f;
constexpr uint32_t kInfBits = 0x7F800000u;
constexpr int kTile = 192;     // candidates per tile
constexpr int kTilePad = 64;   // NaN entries behind them (a pass reads up to 32 past the last)
constexpr uint32_t kTag = 511u;  // candidate number in a kept value's low bits

__device__ __forceinline__ uint32_t f2_bits(const float4 q, float px, float py, float pz) {
  const float fx = q.x - px, fy = q.y - py, fz = q.z - pz;
  return __float_as_uint(fmaf(fx, fx, fmaf(fy, fy, fz * fz)));
}

// a: the smallest values so far, ascending (bits of non-negative floats, which
// order like the floats; a NaN orders last and is never kept).  Two new values at
// a time: three operations per kept value instead of four.
template <int N>
__device__ __forceinline__ void keep_smallest(uint32_t (&a)[N], uint32_t x, uint32_t y) {
  const uint32_t lo = min(x, y), hi = max(x, y);
#pragma unroll
  for (int j = N - 1; j > 1; --j) a[j] = min(min(max(lo, a[j - 1]), max(hi, a[j - 2])), a[j]);
  a[1] = min(min(max(lo, a[0]), hi), a[1]);
  a[0] = min(lo, a[0]);
}

// a <- the N smallest of this lane's a and that of lane ^ delta: the element-wise
// minimum of one list and the other reversed holds them (rising, then falling);
// a bitonic merge over the next power of two (zeros in front) sorts it.
template <int N>
__device__ __forceinline__ void merge_smallest(uint32_t (&a)[N], int delta) {
  constexpr int P = N <= 16 ? 16 : 32;
  uint32_t r[P];
#pragma unroll
  for (int j = 0; j < P; ++j) r[j] = 0u;
#pragma unroll
  for (int j = 0; j < N; ++j) r[N - 1 - j] = __shfl_xor_sync(0xFFFFFFFFu, a[j], delta);
#pragma unroll
  for (int j = 0; j < N; ++j) r[j] = min(r[j], a[j]);
#pragma unroll
  for (int st = P / 2; st > 0; st >>= 1)
#pragma unroll
    for (int j = 0; j < P; ++j)
      if (!(j & st)) {
        const uint32_t lo = min(r[j], r[j | st]), hi = max(r[j], r[j | st]);
        r[j] = lo;
        r[j | st] = hi;
      }
#pragma unroll
  for (int j = 0; j < N; ++j) a[j] = r[P - N + j];
}

// The k-th value (k <= N) of a list in registers.
template <int N>
__device__ __forceinline__ uint32_t value_at(const uint32_t (&a)[N], int k) {
  uint32_t v = a[N - 1];
#pragma unroll
  for (int j = 0; j < N; ++j)
    if (j == k - 1) v = a[j];
  return v;
}

// Members [start, start + cnt) of a cell of a cloud's table (cnt = 0: no such cell).
__device__ __forceinline__ void find_cell(const CellSlot* __restrict__ t, uint32_t mask, int kx,
                                          int ky, int kz, uint32_t& start, uint32_t& cnt) {
  if (!key_in_range(kx) || !key_in_range(ky) || !key_in_range(kz)) return;
  const unsigned long long want = pack_key(kx, ky, kz);
  uint32_t h = hash_key(kx, ky, kz) & mask;
  for (int p = 0; p < kMaxProbe; ++p) {
    const uint4 s = __ldg(reinterpret_cast<const uint4*>(t + h));
    const unsigned long long cur = (unsigned long long)s.x | ((unsigned long long)s.y << 32);
    if (cur == want) {
      cnt = s.w;
      start = s.z - s.w;
      return;
    }
    if (cur == kEmptyKey) return;
    h = (h + 1) & mask;
  }
}

// The members of 32 cells (each lane's start and cnt) one after the other.
struct Cells {
  uint32_t inc;    // members up to this lane's cell, inclusive
  uint32_t shift;  // member = shift of its cell + candidate number
  uint32_t total;
  __device__ __forceinline__ Cells(uint32_t start, uint32_t cnt) {
    const int lane = threadIdx.x & 31;
    inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += y;
    }
    total = __shfl_sync(0xFFFFFFFFu, inc, 31);
    shift = start - (inc - cnt);
  }
  // member of candidate c (every lane calls it; meaningless for c >= total)
  __device__ __forceinline__ uint32_t member(uint32_t c) const {
    int cell = 0;  // cells whose members end at or before c
#pragma unroll
    for (int st = 16; st > 0; st >>= 1)
      if (__shfl_sync(0xFFFFFFFFu, inc, cell + st - 1) <= c) cell += st;
    return __shfl_sync(0xFFFFFFFFu, shift, cell) + c;
  }
  // Candidates c0 .. c0 + m - 1 into the tile, x, y, z and the member's place; the
  // entries behind them, `pad` at least, are NaN (never near anything).
  __device__ __forceinline__ void load(uint32_t c0, uint32_t m, uint32_t pad, float4* tile,
                                       const float4* __restrict__ members) const {
    const int lane = threadIdx.x & 31;
    __syncwarp();  // the tile's previous readers are done
    for (uint32_t t = 0; t < m + pad; t += 32) {
      const uint32_t pos = member(c0 + t + lane);
      const float nan = __uint_as_float(0x7FFFFFFFu);
      float4 v = make_float4(nan, nan, nan, nan);
      if (t + lane < m) {
        v = members[pos];
        v.w = __uint_as_float(pos);
      }
      tile[t + lane] = v;
    }
    __syncwarp();
  }
};

// Scatter of the points v(0) .. v(cnt - 1) about their mean, relative to (px, py,
// pz), written to the point's place in the output.
template <int N, typename F>
__device__ __forceinline__ void write_scatter(int cnt, float px, float py, float pz, F&& v,
                                              float* __restrict__ out) {
  float m0 = 0.f, m1 = 0.f, m2 = 0.f;
#pragma unroll
  for (int j = 0; j < N; ++j)
    if (j < cnt) {
      const float4 q = v(j);
      m0 += q.x - px;
      m1 += q.y - py;
      m2 += q.z - pz;
    }
  const float idn = cnt > 0 ? 1.0f / (float)cnt : 0.f;
  m0 *= idn;
  m1 *= idn;
  m2 *= idn;
  float S[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int j = 0; j < N; ++j)
    if (j < cnt) {
      const float4 q = v(j);
      const float e0 = (q.x - px) - m0, e1 = (q.y - py) - m1, e2 = (q.z - pz) - m2;
      S[0] = fmaf(e0, e0, S[0]);
      S[1] = fmaf(e0, e1, S[1]);
      S[2] = fmaf(e0, e2, S[2]);
      S[3] = fmaf(e1, e1, S[3]);
      S[4] = fmaf(e1, e2, S[4]);
      S[5] = fmaf(e2, e2, S[5]);
    }
  float2* o = reinterpret_cast<float2*>(out);
  o[0] = make_float2(S[0], S[1]);
  o[1] = make_float2(S[2], S[3]);
  o[2] = make_float2(S[4], S[5]);
}

// What the search kernels read.
struct Grid {
  const int64_t* off;
  int32_t n_clouds;
  const double* h;
  const float* reach2;          // h^2, rounded down
  const int64_t* slot_base;
  const uint32_t* cap_mask;
  const CellSlot* slots;
  const float4* members;
  const uint32_t* member_slot;
  const uint32_t* n_members;
  uint32_t* rest;               // members left to the second kernel (null: all)
  uint32_t* n_rest;
};

// K: neighbours at most; W: warps per CTA.
template <int K, int W>
__global__ void __launch_bounds__(32 * W) knn_select_kernel(const Grid G, int32_t k, int32_t per_warp,
                                                            int32_t* __restrict__ nbr_out,
                                                            float* __restrict__ covs_out) {
  constexpr int CAP = K + 2 <= 32 ? K + 2 : 32;   // values kept
  constexpr int P = CAP <= 16 ? 16 : 32;
  constexpr uint32_t kSlotBits = (uint32_t)P - 1u;  // list slot in a sort key's low bits
  __shared__ float4 tile_s[W][kTile + kTilePad];
  __shared__ uint32_t list_s[W][CAP * 32];          // entry j of query q at 32 j + q
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float4* tile = tile_s[w];
  uint32_t* list = list_s[w];
  const int64_t nm = *G.n_members;
  const int64_t p0 = ((int64_t)blockIdx.x * W + w) * per_warp;
  if (p0 >= nm) return;
  const bool mine = lane < per_warp && p0 + lane < nm;
  const float4 me = G.members[mine ? p0 + lane : p0];
  const uint32_t my_slot = mine ? G.member_slot[p0 + lane] : kNoSlot;
  const int64_t i = __float_as_uint(me.w);
  const int my_cloud = cloud_of(G.off, G.n_clouds, i);
  const unsigned long long my_key = mine ? G.slots[my_slot].key : 0ull;
  const uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, my_slot, 1);
  uint32_t heads = __ballot_sync(0xFFFFFFFFu, mine && (lane == 0 || prev != my_slot));
  const int n_mine = __popc(__ballot_sync(0xFFFFFFFFu, mine));
  uint32_t finished = 0u;  // bit q: query q's list is complete

  while (heads) {  // the queries [b, e) share a cell
    const int b = __ffs(heads) - 1;
    heads &= heads - 1u;
    const int e = heads ? __ffs(heads) - 1 : n_mine;
    const int lg = e - b <= 4 ? 2 : e - b <= 8 ? 3 : e - b <= 16 ? 4 : 5;
    const int ql = lane & ((1 << lg) - 1);
    const int q = (b + ql) & 31, part = lane >> lg, parts = 32 >> lg;
    const bool act = b + ql < e;
    const float px = __shfl_sync(0xFFFFFFFFu, me.x, q), py = __shfl_sync(0xFFFFFFFFu, me.y, q),
                pz = __shfl_sync(0xFFFFFFFFu, me.z, q);
    const int c = __shfl_sync(0xFFFFFFFFu, my_cloud, b);
    const unsigned long long key = __shfl_sync(0xFFFFFFFFu, my_key, b);
    const unsigned long long fm = (1ull << kKeyBits) - 1ull;
    uint32_t start = 0u, cnt = 0u;
    if (lane < 27)
      find_cell(G.slots + G.slot_base[c], G.cap_mask[c],
                (int)((key >> (2 * kKeyBits)) & fm) - kKeyBias + lane % 3 - 1,
                (int)((key >> kKeyBits) & fm) - kKeyBias + lane / 3 % 3 - 1,
                (int)(key & fm) - kKeyBias + lane / 9 - 1, start, cnt);
    const Cells cells(start, cnt);
    if (cells.total > kTag + 1u) continue;  // left to the second kernel
    uint32_t a[CAP];
#pragma unroll
    for (int j = 0; j < CAP; ++j) a[j] = kInfBits;
    for (uint32_t c0 = 0; c0 < cells.total; c0 += kTile) {
      const uint32_t m = min((uint32_t)kTile, cells.total - c0);
      cells.load(c0, m, 8u, tile, G.members);
      auto tagged = [&](uint32_t t) { return (f2_bits(tile[t], px, py, pz) & ~kTag) | ((c0 + t) & kTag); };
      for (uint32_t t = part; t < m; t += 2 * parts)  // the last pair may read NaN entries
        keep_smallest<CAP>(a, tagged(t), tagged(t + parts));
    }
    for (int d = 1 << lg; d < 32; d <<= 1) merge_smallest<CAP>(a, d);
    // complete: the k-th value is within the block's reach (every point outside it
    // lies farther than h), or the block holds the whole cloud; and the values
    // left out are at least 2^-14 (or 512 denormal steps) above it
    const uint32_t ak = value_at<CAP>(a, k);
    const bool near = __uint_as_float(ak | kTag) * kF2Up < G.reach2[c] ||
                      (int64_t)cells.total >= G.off[c + 1] - G.off[c];
    const bool done = act && near && ak < kInfBits && (a[CAP - 1] >> 9) > (ak >> 9) + 1u;
    uint32_t place[CAP];  // the kept candidates' members
#pragma unroll
    for (int j = 0; j < CAP; ++j) place[j] = a[j] & kTag;
    if (cells.total > kTile) {
#pragma unroll
      for (int j = 0; j < CAP; ++j) place[j] = cells.member(place[j]);
    } else {
#pragma unroll
      for (int j = 0; j < CAP; ++j) place[j] = __float_as_uint(tile[place[j] & 255u].w);
    }
#pragma unroll
    for (int j = 0; j < CAP; ++j)
      if (act && (j & (parts - 1)) == part) list[j * 32 + q] = a[j] < kInfBits ? place[j] : kNoSlot;
    const uint32_t ok = __ballot_sync(0xFFFFFFFFu, done && part == 0);  // bit ql
    finished |= (lg == 5 ? ok : ok & ((1u << (1 << lg)) - 1u)) << b;
    __syncwarp();
  }

  // ---- order the lists and sum the scatter: one query per lane ----
  bool good = mine && ((finished >> lane) & 1u);
  const float px = me.x, py = me.y, pz = me.z;
  uint32_t ord[P];  // f2 with the list slot in its low bits
  int n = 0;
#pragma unroll
  for (int j = 0; j < CAP; ++j) {
    const uint32_t pos = good ? list[j * 32 + lane] : kNoSlot;
    ord[j] = ~kSlotBits | (uint32_t)j;
    if (pos != kNoSlot) {
      ord[j] = (f2_bits(G.members[pos], px, py, pz) & ~kSlotBits) | (uint32_t)j;
      ++n;
    }
  }
  // the kept values were sorted but for their low 9 bits: within a step of those any
  // order is possible.  Two passes of exchanges restore nearly every list.
  auto order2 = [&](int x, int y) {
    const uint32_t lo = min(ord[x], ord[y]), hi = max(ord[x], ord[y]);
    ord[x] = lo;
    ord[y] = hi;
  };
#pragma unroll
  for (int x = 0; x + 1 < CAP; x += 2) order2(x, x + 1);
#pragma unroll
  for (int x = 1; x + 1 < CAP; x += 2) order2(x, x + 1);
  // Accepted: each of the first k below the one after it, and the k-th below every
  // later one, by more than the error bound.
  uint32_t later = ~0u;  // the smallest after the k-th
#pragma unroll
  for (int x = 0; x < CAP; ++x)
    if (x >= k) later = min(later, ord[x]);
#pragma unroll
  for (int x = 0; x + 1 < CAP; ++x) {
    const float lo = __uint_as_float(ord[x] | kSlotBits);
    const float hi = __uint_as_float((x + 1 < k ? ord[x + 1] : later) & ~kSlotBits);
    good = good && (x >= k || x + 1 >= n || (hi > lo * kF2Up && hi > kF2Tiny));
  }
  // the others go to the second kernel's list
  const uint32_t left = __ballot_sync(0xFFFFFFFFu, mine && !good);
  if (left) {
    uint32_t at = 0u;
    if (lane == 0) at = atomicAdd(G.n_rest, (uint32_t)__popc(left));
    at = __shfl_sync(0xFFFFFFFFu, at, 0);
    if (mine && !good) G.rest[at + __popc(left & ((1u << lane) - 1u))] = (uint32_t)(p0 + lane);
  }
  if (!good) return;
  const int cnt = min(n, k);
  if (nbr_out) {
    const int64_t base = G.off[my_cloud];
#pragma unroll
    for (int j = 0; j < K; ++j)
      if (j < k)
        nbr_out[(int64_t)k * i + j] =
            j < cnt ? (int32_t)((int64_t)__float_as_uint(
                                    G.members[list[(ord[j] & kSlotBits) * 32 + lane]].w) - base)
                    : -1;
  }
  write_scatter<K>(cnt, px, py, pz,
                   [&](int j) { return G.members[list[(ord[j] & kSlotBits) * 32 + lane]]; },
                   covs_out + 6 * i);
}

// One warp per query left over by the first kernel.
constexpr int kRestWarps = 4;
constexpr int kRestList = 64;
template <int K>
__global__ void __launch_bounds__(32 * kRestWarps) knn_rest_kernel(const Grid G, int32_t k,
                                                                   int32_t* __restrict__ nbr_out,
                                                                   float* __restrict__ covs_out) {
  __shared__ float4 tile_s[kRestWarps][kTile + kTilePad];
  __shared__ float4 list_s[kRestWarps][kRestList];               // x, y, z, point index
  __shared__ unsigned long long dist_s[kRestWarps][kRestList];   // binary64 d^2
  __shared__ float4 near_s[kRestWarps][K];                       // the nearest, in order
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float4 *tile = tile_s[w], *list = list_s[w], *nearest = near_s[w];
  unsigned long long* dist = dist_s[w];
  const uint32_t n_rest = G.rest ? *G.n_rest : *G.n_members;
  for (uint32_t r = blockIdx.x * kRestWarps + w; r < n_rest; r += gridDim.x * kRestWarps) {
    const uint32_t p = G.rest ? G.rest[r] : r;
    const float4 me = G.members[p];
    const float px = me.x, py = me.y, pz = me.z;
    const int64_t i = __float_as_uint(me.w);
    const int c = cloud_of(G.off, G.n_clouds, i);
    const int64_t base = G.off[c], nc = G.off[c + 1] - base;
    const CellSlot* t = G.slots + G.slot_base[c];
    const uint32_t mask = G.cap_mask[c];
    const int64_t cap = (int64_t)mask + 1;
    const double h = G.h[c];
    const unsigned long long key = G.slots[G.member_slot[p]].key, fm = (1ull << kKeyBits) - 1ull;
    const int cx = (int)((key >> (2 * kKeyBits)) & fm) - kKeyBias;
    const int cy = (int)((key >> kKeyBits) & fm) - kKeyBias;
    const int cz = (int)(key & fm) - kKeyBias;
    auto visit = [&](uint32_t start, uint32_t cnt, auto&& f) -> int64_t {
      if (!__any_sync(0xFFFFFFFFu, cnt != 0u)) return 0;
      const Cells cells(start, cnt);
      for (uint32_t c0 = 0; c0 < cells.total; c0 += kTile) {
        const uint32_t m = min((uint32_t)kTile, cells.total - c0);
        cells.load(c0, m, 32u, tile, G.members);
        f(m);
      }
      return cells.total;
    };
    // the cells with Chebyshev distance in [from, to]
    auto rings = [&](int from, int to, auto&& f) -> int64_t {
      int64_t got = 0;
      const int side = 2 * to + 1;
      const int64_t cube = (int64_t)side * side * side;
      for (int64_t c0 = 0; c0 < cube; c0 += 32) {
        uint32_t start = 0u, cnt = 0u;
        const uint32_t cc = (uint32_t)(c0 + lane);
        if (c0 + lane < cube) {
          const int dx = (int)(cc % side) - to, dy = (int)(cc / side % side) - to,
                    dz = (int)(cc / side / side) - to;
          if (max(abs(dx), max(abs(dy), abs(dz))) >= from)
            find_cell(t, mask, cx + dx, cy + dy, cz + dz, start, cnt);
        }
        got += visit(start, cnt, f);
      }
      return got;
    };
    auto whole = [&](auto&& f) -> int64_t {  // every cell of the cloud's table
      int64_t got = 0;
      for (int64_t s0 = 0; s0 < cap; s0 += 32) {
        uint32_t start = 0u, cnt = 0u;
        if (s0 + lane < cap) {
          const uint4 s = __ldg(reinterpret_cast<const uint4*>(t + s0 + lane));
          cnt = s.w;
          start = s.z - s.w;
        }
        got += visit(start, cnt, f);
      }
      return got;
    };

    // how far to look, and the k-th float32 value
    uint32_t a[K];
    auto reset = [&]() {
#pragma unroll
      for (int j = 0; j < K; ++j) a[j] = kInfBits;
    };
    auto keep = [&](uint32_t m) {
      for (uint32_t x = lane; x < m; x += 64)
        keep_smallest<K>(a, f2_bits(tile[x], px, py, pz), f2_bits(tile[x + 32], px, py, pz));
    };
    auto merge = [&]() {
      for (int d = 1; d < 32; d <<= 1) merge_smallest<K>(a, d);
    };
    reset();
    int64_t seen = 0;
    int s = 1;
    bool all_cells = false;
    for (;; ++s) {
      const int64_t side = 2 * s + 1;
      if (side * side * side > cap) {  // fewer slots than cells: the whole table instead
        reset();
        whole(keep);
        merge();
        all_cells = true;
        break;
      }
      seen += rings(s == 1 ? 0 : s, s, keep);
      merge();
      // every point not yet visited lies farther than s h
      const float reach2 = __double2float_rd((double)s * h * ((double)s * h));
      if (seen >= nc || __uint_as_float(value_at<K>(a, k)) * kF2Up < reach2) break;
      if (lane != 0) reset();  // the merged list stays with lane 0
    }
    auto again = [&](auto&& f) {
      if (all_cells) whole(f);
      else rings(0, s, f);
    };
    auto d2_of = [&](const float4 m) {
      const double ex = __dsub_rn((double)m.x, (double)px), ey = __dsub_rn((double)m.y, (double)py),
                   ez = __dsub_rn((double)m.z, (double)pz);
      return (unsigned long long)__double_as_longlong(
          __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez)));
    };
    auto with_index = [&](float4 v) {  // the tile holds the member's place: its point index
      v.w = G.members[__float_as_uint(v.w)].w;
      return v;
    };
    // every candidate that can be among the k nearest (2^-15 or 256 denormal
    // steps above the k-th; all, if there are fewer than k)
    const uint32_t ak = value_at<K>(a, k);
    const uint32_t lim = ak >= kInfBits ? kInfBits : min(ak + 256u, kInfBits);
    uint32_t found = 0u;
    again([&](uint32_t m) {
      for (uint32_t x0 = 0; x0 < m; x0 += 32) {
        const float4 v = tile[x0 + lane];
        const bool hit = f2_bits(v, px, py, pz) <= lim;
        const uint32_t hits = __ballot_sync(0xFFFFFFFFu, hit);
        const uint32_t pos = found + __popc(hits & ((1u << lane) - 1u));
        if (hit && pos < kRestList) {
          list[pos] = with_index(v);
          dist[pos] = d2_of(v);
        }
        found += __popc(hits);
      }
    });
    __syncwarp();
    const int cnt = (int)min(found, (uint32_t)k);
    if (found <= kRestList) {
      for (uint32_t x = lane; x < found; x += 32) {  // rank in the order (d^2, index)
        const unsigned long long d = dist[x];
        const uint32_t id = __float_as_uint(list[x].w);
        int rank = 0;
        for (uint32_t y = 0; y < found; ++y)
          rank += before(dist[y], __float_as_uint(list[y].w), d, id) ? 1 : 0;
        if (rank < k) nearest[rank] = list[x];
      }
    } else {
      // many ties: the next one in the order (d^2, index), k times
      unsigned long long last_d = 0ull;
      uint32_t last_j = 0u;
      for (int j = 0; j < cnt; ++j) {
        unsigned long long best_d = ~0ull;
        uint32_t best_j = 0xFFFFFFFFu;
        float4 best = me;
        again([&](uint32_t m) {
          for (uint32_t x = lane; x < m; x += 32) {
            const float4 v = tile[x];
            if (f2_bits(v, px, py, pz) > lim) continue;
            const float4 u = with_index(v);
            const unsigned long long d = d2_of(v);
            const uint32_t id = __float_as_uint(u.w);
            if ((j == 0 || before(last_d, last_j, d, id)) && before(d, id, best_d, best_j)) {
              best_d = d;
              best_j = id;
              best = u;
            }
          }
        });
        __syncwarp();
        unsigned long long d = best_d;
        uint32_t id = best_j;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const unsigned long long od = __shfl_xor_sync(0xFFFFFFFFu, d, o);
          const uint32_t oj = __shfl_xor_sync(0xFFFFFFFFu, id, o);
          if (before(od, oj, d, id)) {
            d = od;
            id = oj;
          }
        }
        last_d = d;
        last_j = id;
        if (best_d == d && best_j == id) nearest[j] = best;
      }
    }
    __syncwarp();
    if (nbr_out)
      for (int j = lane; j < k; j += 32)
        nbr_out[(int64_t)k * i + j] =
            j < cnt ? (int32_t)((int64_t)__float_as_uint(nearest[j].w) - base) : -1;
    if (lane == 0)
      write_scatter<K>(cnt, px, py, pz, [&](int j) { return nearest[j]; }, covs_out + 6 * i);
    __syncwarp();
  }
}

// Scatter matrix -> regularised covariance, in place.
__global__ void __launch_bounds__(kThreads) knn_covariance_kernel(int64_t n, float eps,
                                                                  float* __restrict__ covs) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  float2* o = reinterpret_cast<float2*>(covs + 6 * i);
  const float2 s0 = o[0], s1 = o[1], s2 = o[2];
  const float S[6] = {s0.x, s0.y, s1.x, s1.y, s2.x, s2.y};
  const float tr = S[0] + S[3] + S[5];
  float v[3] = {0.f, 0.f, 1.f};
  if (tr > 0.f) {
    const float itr = 1.0f / tr;
    float a6[6];
#pragma unroll
    for (int r = 0; r < 6; ++r) a6[r] = S[r] * itr;
    smallest_eigvec(a6, v);
  }
  const float w = 1.0f - eps;
  o[0] = make_float2(1.0f - w * v[0] * v[0], -w * v[0] * v[1]);
  o[1] = make_float2(-w * v[0] * v[2], 1.0f - w * v[1] * v[1]);
  o[2] = make_float2(-w * v[1] * v[2], 1.0f - w * v[2] * v[2]);
}

template <int K, int W>
void launch_search(Grid G, int64_t n, int32_t k, int32_t* nbr_out, float* covs_out,
                   cudaStream_t st) {
  count_launches(1);
  // Queries per warp.  A warp takes its cells one after the other, so a cloud that
  // does not fill the GPU with 32 queries per warp is spread over more of them;
  // the price is more cells cut in two.  All kernels of the call, 8 / 16 / 32 per
  // warp: 20,000 points 69 / 72 / 81 us, 80,000 points 88 / 87 / 92 us, 160,000
  // points 153 / 141 / 140 us, 640,000 points 419 / 358 / 333 us.
  const int64_t sms = device_sm_count();
  const int per_warp = n < 160 * sms ? 8 : n < 660 * sms ? 16 : 32;
  const int64_t per = (int64_t)per_warp * W;
  // (with 32 neighbours the first kernel, which keeps 32 values, could finish no query:
  // 20,000 points 326 -> 283 us a call without it, 640,000 points 6,173 -> 5,576)
  if (k < 32) {
    knn_select_kernel<K, W><<<(unsigned)((n + per - 1) / per), 32 * W, 0, st>>>(
        G, k, per_warp, nbr_out, covs_out);
    count_launches(1);
  } else {
    G.rest = nullptr;
  }
  // the number left over is on the device: a grid that fills the GPU, or one warp
  // per 8 points of a small cloud
  const int64_t blocks = std::min<int64_t>((n + 8 * kRestWarps - 1) / (8 * kRestWarps),
                                           (int64_t)device_sm_count() * 8);
  knn_rest_kernel<K><<<(unsigned)blocks, 32 * kRestWarps, 0, st>>>(G, k, nbr_out, covs_out);
}

int grid_of(int64_t n) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + kThreads - 1) / kThreads, 0x7FFFFFFF));
}

}  // namespace
}  // namespace vgicp

extern "C" {

int vgicp_estimate_covariances(const float* points, const int64_t* offsets, int32_t n_clouds,
                               int32_t k, double eps, double cell, int32_t* nbr_out,
                               float* covs_out, vgicp_stream_t stream) {
  using namespace vgicp;
  if (n_clouds <= 0 || !offsets) return set_error(VGICP_ERR_INVALID_ARG, "n_clouds must be >= 1");
  if (k < 1 || k > 32) return set_error(VGICP_ERR_INVALID_ARG, "k must be in [1, 32]");
  if (!(eps > 0.0) || eps > 1.0) return set_error(VGICP_ERR_INVALID_ARG, "eps must be in (0, 1]");
  if (!(cell >= 0.0) || !std::isfinite(cell))
    return set_error(VGICP_ERR_INVALID_ARG, "cell must be 0 (automatic) or positive");
  if (offsets[0] != 0) return set_error(VGICP_ERR_INVALID_ARG, "offsets[0] must be 0");
  for (int32_t c = 0; c < n_clouds; ++c)
    if (offsets[c + 1] < offsets[c])
      return set_error(VGICP_ERR_INVALID_ARG, "offsets must be non-decreasing");
  const int64_t n = offsets[n_clouds];
  if (n >= (int64_t)0xFFFFFFFFll) return set_error(VGICP_ERR_INVALID_ARG, "more than 2^32-1 points");
  if (n == 0) return VGICP_OK;
  int rc = check_cloud(points, covs_out, n, "cloud");
  if (rc) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  // per-cloud cell tables: capacity next_pow2(2 n_c)
  std::vector<int64_t> base((size_t)n_clouds);
  std::vector<uint32_t> mask((size_t)n_clouds);
  int64_t cap_total = 0;
  for (int32_t c = 0; c < n_clouds; ++c) {
    uint64_t cap = 16;
    while (cap < 2ull * (uint64_t)std::max<int64_t>(offsets[c + 1] - offsets[c], 1)) cap <<= 1;
    base[(size_t)c] = cap_total;
    mask[(size_t)c] = (uint32_t)(cap - 1);
    cap_total += (int64_t)cap;
  }
  if (cap_total >= (int64_t)0xFFFFFFFFll)
    return set_error(VGICP_ERR_INVALID_ARG, "more than 2^32-1 cell slots");
  // one buffer; its front is filled by the host in one copy: offsets, tables,
  // empty boxes, and the zeroed counters
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = (off + std::max<size_t>(bytes, 1) + 255) & ~size_t(255);
    return o;
  };
  const size_t o_off = take(sizeof(int64_t) * (n_clouds + 1));
  const size_t o_base = take(sizeof(int64_t) * n_clouds);
  const size_t o_mask = take(sizeof(uint32_t) * n_clouds);
  const size_t o_bbox = take(sizeof(uint32_t) * 6 * n_clouds);
  const size_t o_done = take(sizeof(uint32_t) * n_clouds);
  const size_t o_cursor = take(sizeof(uint32_t));
  const size_t o_nrest = take(sizeof(uint32_t));
  const size_t o_status = take(sizeof(int32_t));
  const size_t upload = off;
  const size_t o_h = take(sizeof(double) * n_clouds);
  const size_t o_inv = take(sizeof(float) * n_clouds);
  const size_t o_reach = take(sizeof(float) * n_clouds);
  const size_t o_rest = take(sizeof(uint32_t) * n);
  const size_t o_slots = take(sizeof(CellSlot) * cap_total);
  const size_t o_ptslot = take(sizeof(uint32_t) * n);
  const size_t o_members = take(sizeof(float4) * n);
  const size_t o_mslot = take(sizeof(uint32_t) * n);
  std::vector<char> host(upload, 0);
  std::memcpy(host.data() + o_off, offsets, sizeof(int64_t) * (n_clouds + 1));
  std::memcpy(host.data() + o_base, base.data(), sizeof(int64_t) * n_clouds);
  std::memcpy(host.data() + o_mask, mask.data(), sizeof(uint32_t) * n_clouds);
  uint32_t* boxes = reinterpret_cast<uint32_t*>(host.data() + o_bbox);
  for (int64_t j = 0; j < 6 * (int64_t)n_clouds; ++j)
    boxes[j] = j % 6 < 3 ? 0xFF800000u : 0x007FFFFFu;  // ordered bits of +inf, of -inf
  char* d = nullptr;
  VGICP_CUDA_TRY(device_malloc(reinterpret_cast<void**>(&d), off, st, true));
  auto P = [&](size_t o) { return d + o; };
  const int64_t* d_off = reinterpret_cast<const int64_t*>(P(o_off));
  const int64_t* d_base = reinterpret_cast<const int64_t*>(P(o_base));
  const uint32_t* d_mask = reinterpret_cast<const uint32_t*>(P(o_mask));
  uint32_t* d_bbox = reinterpret_cast<uint32_t*>(P(o_bbox));
  uint32_t* d_done = reinterpret_cast<uint32_t*>(P(o_done));
  uint32_t* d_cursor = reinterpret_cast<uint32_t*>(P(o_cursor));
  int32_t* d_status = reinterpret_cast<int32_t*>(P(o_status));
  double* d_h = reinterpret_cast<double*>(P(o_h));
  float* d_inv = reinterpret_cast<float*>(P(o_inv));
  float* d_reach = reinterpret_cast<float*>(P(o_reach));
  CellSlot* d_slots = reinterpret_cast<CellSlot*>(P(o_slots));
  uint32_t* d_ptslot = reinterpret_cast<uint32_t*>(P(o_ptslot));
  float4* d_members = reinterpret_cast<float4*>(P(o_members));
  uint32_t* d_mslot = reinterpret_cast<uint32_t*>(P(o_mslot));
  // (a copy from pageable memory returns once the source is staged)
  cudaError_t e = cudaMemcpyAsync(d, host.data(), upload, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) rc = check_cuda(e, "estimate_covariances setup");
  if (rc == VGICP_OK) {
    const int g = grid_of(n);
    // CTAs per cloud: one per 512 points of an average cloud
    const int parts = (int)std::max<int64_t>(1, std::min<int64_t>(kPrepParts, n / n_clouds / 512));
    prep_kernel<<<dim3(n_clouds, parts), kThreads, 0, st>>>(points, d_off, k, cell, d_base, d_mask,
                                                           d_slots, d_bbox, d_done, d_h, d_inv, d_reach);
    cell_insert_kernel<<<g, kThreads, 0, st>>>(points, n, d_off, n_clouds, d_h, d_inv, d_base,
                                               d_mask, d_slots, d_ptslot, d_status);
    cell_alloc_kernel<<<grid_of((cap_total + kAllocPer - 1) / kAllocPer), kThreads, 0, st>>>(
        d_slots, cap_total, d_cursor);
    cell_scatter_kernel<<<g, kThreads, 0, st>>>(points, n, d_ptslot, d_slots, d_members, d_mslot);
    const Grid G{d_off,   n_clouds,  d_h,     d_reach, d_base,
                 d_mask,  d_slots,   d_members, d_mslot, d_cursor,
                 reinterpret_cast<uint32_t*>(P(o_rest)), reinterpret_cast<uint32_t*>(P(o_nrest))};
    if (k <= 10) launch_search<10, 4>(G, n, k, nbr_out, covs_out, st);
    else if (k <= 20) launch_search<20, 4>(G, n, k, nbr_out, covs_out, st);
    else launch_search<32, 4>(G, n, k, nbr_out, covs_out, st);
    knn_covariance_kernel<<<g, kThreads, 0, st>>>(n, (float)eps, covs_out);
    count_launches(5);
    e = cudaGetLastError();
    if (e != cudaSuccess) rc = check_cuda(e, "estimate_covariances kernels");
  }
  int32_t status = 0;
  if (rc == VGICP_OK) {
    e = cudaMemcpyAsync(&status, d_status, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) rc = check_cuda(e, "estimate_covariances status");
  }
  e = cudaFreeAsync(d, st);
  if (rc == VGICP_OK && e != cudaSuccess) rc = check_cuda(e, "cudaFreeAsync");
  if (rc == VGICP_OK && status == VGICP_ERR_KEY_RANGE)
    rc = set_error(status, "a point's cell key is outside [-2^20, 2^20) (cell too small for "
                           "the coordinates, or not finite)");
  else if (rc == VGICP_OK && status == VGICP_ERR_HASH_FULL)
    rc = set_error(status, "cell table probe limit exceeded");
  return rc;
}

}  // extern "C"
