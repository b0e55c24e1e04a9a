// scatter_eval.cu — MI evaluation of poses that share nothing (a single pose, the simplices of a
// Nelder-Mead phase, scattered candidates on the device), with the points of every pose spread over
// the whole GPU.
//
// The table kernels (eval.cu) give a pose to one CTA, which sweeps all its points: 64 us for 120k
// points whether there is one pose or 152 of them.  Here a pose's voxels are dense sums in global
// memory (16 bytes per voxel: n << 40 | S1, and S2; 8 without z sums), so any warp can take any 32
// points of any pose: consecutive scan points in one voxel are merged in the warp, the rest are two
// 64-bit adds in L2.  The add that finds a voxel empty lists it; only the listed voxels are read,
// turned into symbols and cleared again, so the sums stay zero between calls and no pass covers the
// whole grid.
//
//   sums_kernel    points -> sums and lists of occupied voxels
//   voxels_kernel  listed voxels -> feature symbols, joint histogram and occupied box per pose
// compose_kernel (eval.cu) then gives MI and argmax, and resets the histogram, box and list counter that
// it has read: a call is these three kernels.  (With a kernel to clear and one for the argmax a one-pose
// call with its read-back took 64 us, now 57; 16 simplices x 25 iterations 3.05, now 2.78 ms.)  Both are
// bound by the latency of their L2 atomics and scattered accesses.  Against the table kernels, with
// those two kernels still, per call with device inputs and outputs: 120k points at 0.5 m 105 -> 46 us
// for one pose, 110 -> 70 us for 16; at 0.25 m 153 -> 54 and 161 -> 90 us; 259k points on the
// 6.4M-voxel grid 315 -> 76 us and (10 poses) 344 -> 147 us.  Every sum is exact in 64 bits (at most
// kScatterMaxPoints points), so no pose needs the exact path.
#include <algorithm>
#include <climits>

#include "align_internal.h"
#include "device_common.cuh"

namespace mialign {

namespace {

constexpr uint32_t kFullMask = 0xFFFFFFFFu;
constexpr int kShiftN = 40;  // n above S1: S1 <= 2^22 points x 8,004 mm < 2^35
constexpr int kSumThreads = 512, kVoxelThreads = 512;

// One thread per point and pose; blockIdx.y walks the poses.
template <bool kVar>
__global__ void __launch_bounds__(kSumThreads) sums_kernel(const __grid_constant__ ScatterArgs a) {
  const int lane = threadIdx.x & 31;
  // one add to a pose's list per block (a list's counter takes turns: an add per warp bound the
  // kernel, 2 us per pose of 120k points)
  __shared__ uint32_t block_n, block_at;
  const int64_t p = blockIdx.x * (int64_t)kSumThreads + threadIdx.x;
  const int64_t q = min(p, a.n - 1);
  const float x = __ldg(a.xyz + 3 * q), y = __ldg(a.xyz + 3 * q + 1), z = __ldg(a.xyz + 3 * q + 2);
  const GridConst& gc = a.gc;
  uint32_t lane_lt;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lane_lt));
  for (int w = blockIdx.y; w < a.P; w += gridDim.y) {
    const float* pose = a.poses + 12 * (size_t)w;
    Pose12 P;
#pragma unroll
    for (int i = 0; i < 9; ++i) P.r[i] = __ldg(pose + i);
#pragma unroll
    for (int i = 0; i < 3; ++i) P.t[i] = __ldg(pose + 9 + i);
    int dz = 0;
    uint32_t key = p < a.n ? voxel_key(P, x, y, z, gc.inv_res, gc.X, gc.Y, gc.Z, gc.res_mm, &dz) : kEmptyKey;
    if (key == kEmptyKey) dz = 0;
    const uint32_t up = __shfl_up_sync(kFullMask, key, 1);
    const bool cut = lane == 0 || key != up;
    const uint32_t cuts = __ballot_sync(kFullMask, cut);
    // the run's last lane: before the next cut
    const uint32_t above = cuts & ~(lane_lt | 1u << lane);
    const int last = above ? __ffs(above) - 2 : 31;
    uint32_t s1 = (uint32_t)dz, s2 = (uint32_t)(dz * dz);  // inclusive sums over the warp; a run's by difference
    if (kVar) {
#pragma unroll
      for (int k = 1; k < 32; k <<= 1) {
        const uint32_t v1 = __shfl_up_sync(kFullMask, s1, k), v2 = __shfl_up_sync(kFullMask, s2, k);
        if (lane >= k) s1 += v1, s2 += v2;
      }
      const uint32_t e1 = __shfl_sync(kFullMask, s1, last), e2 = __shfl_sync(kFullMask, s2, last);
      s1 = e1 - s1 + (uint32_t)dz;
      s2 = e2 - s2 + (uint32_t)(dz * dz);  // at most 32 x 8,004^2 < 2^31
    }
    bool first = false;
    if (cut && key != kEmptyKey) {
      unsigned long long* acc = a.sums + ((size_t)w * a.V + key) * (kVar ? 2 : 1);
      const unsigned long long n = (unsigned long long)(last - lane + 1) << kShiftN;
      first = atomicAdd(acc, kVar ? n | s1 : n) == 0ull;
      if (kVar) atomicAdd(acc + 1, (unsigned long long)s2);
    }
    const uint32_t m = __ballot_sync(kFullMask, first);
    if (threadIdx.x == 0) block_n = 0u;
    __syncthreads();
    uint32_t at = 0u;
    if (lane == 0 && m != 0u) at = atomicAdd(&block_n, (uint32_t)__popc(m));
    at = __shfl_sync(kFullMask, at, 0) + __popc(m & lane_lt);
    __syncthreads();
    if (threadIdx.x == 0 && block_n != 0u) block_at = atomicAdd(a.list_n + w, block_n);
    __syncthreads();
    if (first) a.list[(size_t)w * a.list_cap + block_at + at] = key;
    __syncthreads();
  }
}

// Listed voxels of pose blockIdx.y, gridDim.x CTAs each: sums (cleared), symbols, box, histogram.
template <bool kVar>
__global__ void __launch_bounds__(kVoxelThreads) voxels_kernel(const __grid_constant__ ScatterArgs a) {
  __shared__ uint32_t hist[kMaxSymbols * kMaxSymbols];
  __shared__ int32_t box[6];
  __shared__ uint32_t ct[kMaxLevels];
  __shared__ int64_t vt[kMaxLevels];
  const GridConst& gc = a.gc;
  const int tid = threadIdx.x, pose = blockIdx.y, K = gc.K, KK = K * K;
  const uint32_t n_list = __ldg(a.list_n + pose);
  const uint32_t step = gridDim.x * kVoxelThreads;
  if (blockIdx.x == 0 && pose == 0 && tid == 0) {
    *a.best = 0ull;
    *a.redo_count = 0u;
  }
  if (blockIdx.x * kVoxelThreads >= n_list) return;
  for (int i = tid; i < KK; i += kVoxelThreads) hist[i] = 0u;
  for (int i = tid; i < kMaxLevels; i += kVoxelThreads) {
    ct[i] = gc.count_thresh[i];
    vt[i] = gc.var_thresh[i];
  }
  if (tid < 6) box[tid] = tid < 3 ? INT_MAX : INT_MIN;
  __syncthreads();
  int mn[3] = {INT_MAX, INT_MAX, INT_MAX}, mx[3] = {INT_MIN, INT_MIN, INT_MIN};
  for (uint32_t i = blockIdx.x * kVoxelThreads + tid; i < n_list; i += step) {
    const uint32_t key = __ldg(a.list + (size_t)pose * a.list_cap + i);
    const int sA = (int)__ldg(a.symA + key);
    unsigned long long* acc = a.sums + ((size_t)pose * a.V + key) * (kVar ? 2 : 1);
    unsigned long long v0, v1 = 0ull;
    if (kVar) {
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(acc);
      v0 = v.x;
      v1 = v.y;
      *reinterpret_cast<ulonglong2*>(acc) = make_ulonglong2(0ull, 0ull);
    } else {
      v0 = *acc;
      *acc = 0ull;
    }
    const uint64_t n = v0 >> kShiftN;
    const int64_t s1 = (int64_t)(v0 & ((1ull << kShiftN) - 1ull));
    const uint32_t r = gc.div_x ? (uint32_t)__umul64hi(gc.div_x, key) : key;  // key / X
    const uint32_t q = gc.div_y ? (uint32_t)__umul64hi(gc.div_y, r) : r;      // r / Y
    const int k[3] = {(int)(key - r * (uint32_t)gc.X), (int)(r - q * (uint32_t)gc.Y), (int)q};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      mn[j] = min(mn[j], k[j]);
      mx[j] = max(mx[j], k[j]);
    }
    int sB;
    if (n <= gc.nlim) {  // the sums fit 32 bits
      sB = feature_symbol_small(gc, (uint32_t)n, (int32_t)s1, (uint32_t)v1);
    } else {
      sB = feature_symbol(gc.feature, gc.Lc, gc.Lv, ct, vt, n, s1, v1);
      if (kVar) atomicAdd(a.wide_count, 1u);
    }
    if (k[0] >= gc.boxA[0] && k[0] <= gc.boxA[3] && k[1] >= gc.boxA[1] && k[1] <= gc.boxA[4] && k[2] >= gc.boxA[2] &&
        k[2] <= gc.boxA[5])
      atomicAdd(&hist[sA * K + sB], 1u);
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int lo = __reduce_min_sync(kFullMask, mn[j]), hi = __reduce_max_sync(kFullMask, mx[j]);
    if ((tid & 31) == 0 && lo != INT_MAX) {
      atomicMin(&box[j], lo);
      atomicMax(&box[3 + j], hi);
    }
  }
  __syncthreads();
  for (int i = tid; i < KK; i += kVoxelThreads)
    if (hist[i]) atomicAdd(a.out_c + (size_t)pose * KK + i, hist[i]);
  if (tid < 3) atomicMin(a.out_box + 6 * (size_t)pose + tid, box[tid]);
  else if (tid < 6) atomicMax(a.out_box + 6 * (size_t)pose + tid, box[tid]);
}

}  // namespace

size_t scatter_pose_bytes(const GridConst& gc, int64_t n) {
  const size_t V = (size_t)gc.X * gc.Y * gc.Z;
  return V * (gc.feature != 0 ? 16 : 8) + (size_t)std::min<int64_t>((int64_t)V, std::max<int64_t>(n, 1)) * 4;
}

cudaError_t launch_scatter(const ScatterArgs& a, int n_sm, cudaStream_t s, int32_t* launches) {
  cudaError_t e;
  const bool var = a.gc.feature != 0;
  if (a.n > 0) {
    const int64_t bx = (a.n + kSumThreads - 1) / kSumThreads;
    // poses in turn once the points alone fill the GPU a few times over
    const int64_t by = std::min<int64_t>(a.P, std::max<int64_t>(1, 32 * (int64_t)n_sm / bx));
    const dim3 gp((unsigned)bx, (unsigned)by);
    if (var) sums_kernel<true><<<gp, kSumThreads, 0, s>>>(a);
    else sums_kernel<false><<<gp, kSumThreads, 0, s>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    *launches += 1;
  }
  const dim3 gv((unsigned)std::max(1, std::min(16, 2 * n_sm / a.P)), (unsigned)a.P);
  if (var) voxels_kernel<true><<<gv, kVoxelThreads, 0, s>>>(a);
  else voxels_kernel<false><<<gv, kVoxelThreads, 0, s>>>(a);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  *launches += 1;
  return cudaSuccess;
}

}  // namespace mialign
