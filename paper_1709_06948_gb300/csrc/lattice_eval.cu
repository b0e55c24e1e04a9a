// lattice_eval.cu — MI evaluation of a pose lattice (every combination of some rotations and
// some t'_x, t'_y, t'_z values), sharing the voxel map between its poses.
//
// For a fixed pose the voxel index along an axis, k(u) = floor(fl(fl(u + t) * inv_res)), is a
// monotone step function of the rotated coordinate u.  For a set of translations t_1..t_m the
// sum s(u) = sum_i clamp(k_i(u) + 1, 0, D + 1) is monotone too, and equal sums mean equal
// terms: s names the cell of u in the common refinement of the m voxel grids.  A point
// therefore needs one cell index per axis and rotation; the voxels of every translation follow
// from the cells alone, bit for bit as the FP32 map gives them.
//
//   setup_kernel    thresholds of the axis maps: the smallest float of every voxel boundary, its
//                   cell, and the tables (y cell -> k_y per t'_y, x cell -> a float of that cell)
//   points_kernel   per (rotation, t'_x chunk, t'_z): the cells (s_x, s_y, k_z) of consecutive
//                   scan points, merged where they repeat (n, S1, S2), and the size of the bins
//                   (k_z, s_y); the scan as raw tiles, for poses that the exact path finishes
//   offsets_kernel  bin starts
//   scatter_kernel  those elements in bin order: rows (k_z, k_y) of voxels are contiguous for
//                   every t'_y
//   eval_kernel     a group = one (rotation, t'_z, t'_y) and up to 8 t'_x.  Rows in chunks that
//                   fit shared memory: the occupied x cells of a row as a bit mask, so that the
//                   popcount below a cell's bit is its place in (row, cell) order; sums
//                   (n, S1, S2) per occupied cell, then their running sums.  For each of the
//                   group's poses a voxel is a stretch of consecutive cells: its sums are the
//                   differences of two running sums, with no hash table and no per-pose atomics
//                   but the joint histogram's.
//
// Against the table kernels (eval.cu), which map every point under every pose (or pose pair)
// and insert its runs into a hash table, the per-pose work falls from every point to every
// occupied cell of the group (0.2 per point on the 120k-point LiDAR pair at 0.5 m) and every
// occupied voxel (0.06 per point).  Measured per evaluation of 4,096 poses (all kernels but compose),
// against the table kernels: 120k points at 0.5 m 1.27 -> 0.67 ms, at 0.25 m 2.59 -> 1.76 ms, 257k
// points at 1 m 1.77 -> 0.75 ms; 32,768 poses of 259k points at 0.2 m, joint feature, 55 -> 28.4 ms.
// The evaluation kernel (0.52 of the 0.67 ms) is bound by instruction issue and shared memory together
// (63% of its issue slots, 63% of the shared-memory pipe) and by the barriers between its short phases;
// points_kernel (73 us) by its instructions, scatter_kernel (55 us) by the latency of L2 atomics.
// Where most poses have a voxel past the 32-bit sums (2 m voxels and larger) the exact path binds: 120k
// points at 4 m 3.1 ms against 2.9 by tables, at 2 m 1.8 against 2.4.
#include <algorithm>
#include <climits>
#include <mutex>

#include "align_internal.h"
#include "device_common.cuh"

namespace mialign {

namespace {

constexpr uint32_t kFullMask = 0xFFFFFFFFu;
constexpr uint32_t kNoRow = 0xFFFFu;
constexpr int kRing = 320;          // voxels waiting per warp: up to 63, and those of 32 records x 8 poses

// Voxel index along an axis (the FP32 map of device_common.cuh), clamped to [-1, D].
__device__ __forceinline__ int axis_k(float u, float t, float inv_res, int D) {
  return max(-1, min(D, __float2int_rd(__fmul_rn(__fadd_rn(u, t), inv_res))));
}

// Float <-> integer of the same order (a bijection of the finite floats onto an interval).
__device__ __forceinline__ float ordered_float(int32_t o) {
  return __int_as_float(o >= 0 ? o : (int32_t)(0x80000000u - (uint32_t)o));
}
constexpr int32_t kOrderedMax = 0x7F7FFFFF;  // FLT_MAX

// Inverse of ordered_float.
__device__ __forceinline__ int32_t float_order(float f) {
  const int32_t b = __float_as_int(f);
  return b >= 0 ? b : (int32_t)(0x80000000u - (uint32_t)b);
}
// The smallest float u with k(u) >= k: searched around k res - t, whose rounding errors (of u, u + t
// and the product) are some spacings of the larger of u and t wide, else among all floats.
__device__ float axis_threshold(int k, float t, float inv_res, int D) {
  int32_t lo = -kOrderedMax, hi = kOrderedMax;  // k(hi) >= k: the largest float is past the grid
  const float at = __fsub_rn(__fdiv_rn((float)k, inv_res), t);
  const float wide = fmaxf(fabsf(at), fabsf(t)) * 4e-6f + 1e-30f;
  const float a = at - wide, b = at + wide;
  if (isfinite(a) && isfinite(b) && axis_k(a, t, inv_res, D) < k && axis_k(b, t, inv_res, D) >= k) {
    lo = float_order(a) + 1;
    hi = float_order(b);
  }
  while (lo < hi) {
    const int32_t mid = (int32_t)(((int64_t)lo + hi) >> 1);
    if (axis_k(ordered_float(mid), t, inv_res, D) >= k) hi = mid;
    else lo = mid + 1;
  }
  return ordered_float(lo);
}

__device__ __forceinline__ const float* pose_row(const LatticeArgs& a, int r, int iz, int iy, int ix) {
  return a.poses + 12 * (size_t)__ldg(a.pose_of + (((size_t)r * a.mz + iz) * a.my + iy) * a.mx + ix);
}

// Cell of u among the m translations t.
__device__ __forceinline__ uint32_t axis_cell(float u, const float* t, int m, float inv_res, int D) {
  int s = m;
#pragma unroll 8
  for (int i = 0; i < m; ++i) s += axis_k(u, t[i], inv_res, D);
  return (uint32_t)s;
}

__global__ void __launch_bounds__(256) setup_kernel(const __grid_constant__ LatticeArgs a) {
  __shared__ float ty[kLatticeMaxY], tx[kLatticeMaxX];
  const int tid = threadIdx.x;
  for (int i = tid; i < a.my; i += blockDim.x) ty[i] = __ldg(pose_row(a, 0, 0, i, 0) + 10);
  for (int i = tid; i < a.mxr; i += blockDim.x) tx[i] = __ldg(pose_row(a, 0, 0, 0, a.ix0 + i) + 9);
  const int64_t g0 = blockIdx.x * (int64_t)blockDim.x + tid, gs = (int64_t)gridDim.x * blockDim.x;
  // empty bins, histograms, boxes and counters
  const int64_t n_bins = (int64_t)a.n_rot * a.mz * a.ncx * a.bin_stride;
  for (int64_t i = g0; i < n_bins / 4; i += gs) reinterpret_cast<uint4*>(a.bins)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (a.first) {
    const int64_t n_c = (int64_t)a.P * a.gc.K * a.gc.K;  // out_c: a multiple of 4 words allocated
    for (int64_t i = g0; i < (n_c + 3) / 4; i += gs) reinterpret_cast<uint4*>(a.out_c)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int64_t i = g0; i < 6 * (int64_t)a.P; i += gs) a.out_box[i] = i % 6 < 3 ? INT_MAX : INT_MIN;
    for (int64_t i = g0; i < a.P; i += gs) a.redo_mark[i] = 0u;
    const float nan = __int_as_float(0x7fc00000);
    for (int64_t i = a.n + g0; i < a.tiles.n_out; i += gs) store_raw_point(a.tiles, i, nan, nan, nan);
  }
  if (g0 == 0) {
    *a.next_item = 0u;
    if (a.first) {
      *a.redo_count = 0u;
      *a.best = 0ull;
    }
  }
  __syncthreads();
  const GridConst& gc = a.gc;
  // y: boundaries of voxel rows per t'_y, and the row of every cell
  for (int64_t i = g0; i < (int64_t)a.my * (gc.Y + 1); i += gs) {
    const int iy = (int)(i / (gc.Y + 1)), k = (int)(i % (gc.Y + 1));
    const uint32_t s = axis_cell(axis_threshold(k, ty[iy], gc.inv_res, gc.Y), ty, a.my, gc.inv_res, gc.Y);
    const uint32_t e = k < gc.Y ? axis_cell(axis_threshold(k + 1, ty[iy], gc.inv_res, gc.Y), ty, a.my, gc.inv_res, gc.Y)
                                : (uint32_t)a.nsy;
    a.by[(size_t)iy * (gc.Y + 1) + k] = s;
    uint16_t* row = a.row_of + (size_t)iy * a.nsy;
    for (uint32_t q = s; q < e; ++q) row[q] = k < gc.Y ? (uint16_t)k : (uint16_t)kNoRow;
    if (k == 0)
      for (uint32_t q = 0; q < s; ++q) row[q] = (uint16_t)kNoRow;
  }
  // x: a float of every cell that starts at a voxel boundary (points lie in no other)
  for (int64_t i = g0; i < (int64_t)a.mxr * (gc.X + 1); i += gs) {
    const int ix = (int)(i / (gc.X + 1)), k = (int)(i % (gc.X + 1));
    const int c = ix / a.gx, x0 = c * a.gx;
    const float u = axis_threshold(k, tx[ix], gc.inv_res, gc.X);
    const uint32_t sx = axis_cell(u, tx + x0, min(a.gx, a.mxr - x0), gc.inv_res, gc.X);
    a.cell_u[(size_t)c * a.nsx + sx] = u;
    a.bx[(size_t)ix * (gc.X + 1) + k] = (uint16_t)sx;
  }
}

// Elements of one (rotation, t'_x chunk, t'_z) list: the cells of the scan's points in scan order,
// equal neighbours of a warp's 32 points merged.  A warp's elements are stored from its first
// point's place on, their number in `count`.  One thread per point; blockIdx.y is the rotation.
// Element: s_y | k_z << 16, s_x | n << 16, S1, S2 (sums of dz - res_mm / 2 and of its square).
__global__ void __launch_bounds__(256) points_kernel(const __grid_constant__ LatticeArgs a) {
  __shared__ float ty[kLatticeMaxY], tx[kLatticeMaxX], tz[kLatticeMaxZ];
  const int tid = threadIdx.x, lane = tid & 31, r = blockIdx.y;
  for (int i = tid; i < a.my; i += blockDim.x) ty[i] = __ldg(pose_row(a, 0, 0, i, 0) + 10);
  for (int i = tid; i < a.mxr; i += blockDim.x) tx[i] = __ldg(pose_row(a, 0, 0, 0, a.ix0 + i) + 9);
  for (int i = tid; i < a.mz; i += blockDim.x) tz[i] = __ldg(pose_row(a, 0, i, 0, 0) + 11);
  float R[9];
  const float* pr = pose_row(a, a.r0 + r, 0, 0, 0);
#pragma unroll
  for (int i = 0; i < 9; ++i) R[i] = __ldg(pr + i);
  __syncthreads();
  const GridConst& gc = a.gc;
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + tid;
  const int64_t p0 = p - lane;  // the warp's first point
  if (p0 >= a.n) return;
  const int64_t q = min(p, a.n - 1);
  float ux, uy, uz;
  const float px = __ldg(a.xyz + 3 * q), py = __ldg(a.xyz + 3 * q + 1), pz = __ldg(a.xyz + 3 * q + 2);
  if (a.first && r == 0 && p < a.n) store_raw_point(a.tiles, p, px, py, pz);
  rotate_point(R, px, py, pz, ux, uy, uz);
  // a non-finite point (or one that overflows) is outside the grid under every pose
  bool in_p = p < a.n && isfinite(ux) && isfinite(uy) && isfinite(uz);
  const uint32_t sy = axis_cell(uy, ty, a.my, gc.inv_res, gc.Y);
  in_p = in_p && sy > 0u && sy < (uint32_t)(a.my * (gc.Y + 1));
  uint32_t lane_lt;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lane_lt));
  for (int c = 0; c < a.ncx; ++c) {
    const int x0 = c * a.gx, m = min(a.gx, a.mxr - x0);
    const uint32_t sx = axis_cell(ux, tx + x0, m, gc.inv_res, gc.X);
    const bool in_c = in_p && sx > 0u && sx < (uint32_t)(m * (gc.X + 1));
    const uint32_t sxy = sx | sy << 16;
    for (int iz = 0; iz < a.mz; ++iz) {
      const float gz = __fadd_rn(uz, tz[iz]);
      const int kz = __float2int_rd(__fmul_rn(gz, gc.inv_res));
      const bool in = in_c && (uint32_t)kz < (uint32_t)gc.Z;
      const int key = in ? kz : -1;
      const int d = in ? __float2int_rn(__fmul_rn(gz, 1000.0f)) - kz * gc.res_mm - gc.res_mm / 2 : 0;
      const uint32_t up_xy = __shfl_up_sync(kFullMask, sxy, 1);
      const int up_key = __shfl_up_sync(kFullMask, key, 1);
      const bool cut = lane == 0 || key != up_key || sxy != up_xy;
      const uint32_t cuts = __ballot_sync(kFullMask, cut);
      const uint32_t heads = __ballot_sync(kFullMask, cut && in);
      // the run's last lane: before the next cut
      const uint32_t above = cuts & ~(lane_lt | 1u << lane);
      const int last = above ? __ffs(above) - 2 : 31;
      int s1 = d, s2 = d * d;  // inclusive sums over the warp; a run's by difference
#pragma unroll
      for (int k = 1; k < 32; k <<= 1) {
        const int v1 = __shfl_up_sync(kFullMask, s1, k), v2 = __shfl_up_sync(kFullMask, s2, k);
        if (lane >= k) s1 += v1, s2 += v2;  // the square sums wrap; their differences do not
      }
      const int e1 = __shfl_sync(kFullMask, s1, last), e2 = __shfl_sync(kFullMask, s2, last);
      const size_t list = ((size_t)r * a.mz + iz) * a.ncx + c;
      if (cut && in) {
        const uint4 e = make_uint4(sy | (uint32_t)kz << 16, sx | (uint32_t)(last - lane + 1) << 16,
                                   (uint32_t)(e1 - s1 + d), (uint32_t)e2 - (uint32_t)s2 + (uint32_t)(d * d));
        a.raw[list * a.n_pad + p0 + __popc(heads & lane_lt)] = e;
        // neighbouring points share bins: one add per bin and warp
        const uint32_t bin = (uint32_t)kz * (uint32_t)a.nsy + sy;
        const uint32_t same = __match_any_sync(heads, bin);
        if ((same & lane_lt) == 0u) atomicAdd(a.bins + list * a.bin_stride + bin + 1, (uint32_t)__popc(same));
      }
      if (lane == 0) a.count[list * (a.n_pad / 32) + p0 / 32] = (uint8_t)__popc(heads);
    }
  }
}

// Inclusive scan over a warp.
__device__ __forceinline__ uint32_t warp_scan(uint32_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t u = __shfl_up_sync(kFullMask, v, d);
    if (lane >= d) v += u;
  }
  return v;
}
// Exclusive scan over the block of one value per thread; tmp: a word per warp (not reused
// before another barrier).  Returns the value's prefix, and the sum in `total`.
template <int kNW>
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t* tmp, uint32_t& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t inc = warp_scan(v);
  if (lane == 31) tmp[w] = inc;
  __syncthreads();
  const uint32_t t = warp_scan(lane < kNW ? tmp[lane] : 0u);
  total = __shfl_sync(kFullMask, t, kNW - 1);
  const uint32_t before = __shfl_sync(kFullMask, t, (w + 31) & 31);
  return (w ? before : 0u) + inc - v;
}

// Bin starts of one list per block: exclusive prefix sums of its entries, in place.
__global__ void __launch_bounds__(1024) offsets_kernel(const __grid_constant__ LatticeArgs a) {
  __shared__ uint32_t tmp[2][32];
  uint32_t* b = a.bins + (size_t)blockIdx.x * a.bin_stride;
  const int64_t nb = (int64_t)a.gc.Z * a.nsy + 1;
  uint32_t carry = 0u;
  int t = 0;
  for (int64_t i0 = 0; i0 < nb; i0 += 4096, t ^= 1) {
    const int64_t i = i0 + 4 * (int64_t)threadIdx.x;  // bin_stride is a multiple of 4, zero-filled past nb
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (i < nb) v = *reinterpret_cast<const uint4*>(b + i);
    uint32_t total;
    uint32_t s = carry + block_scan<32>(v.x + v.y + v.z + v.w, tmp[t], total);
    if (i < nb) *reinterpret_cast<uint4*>(b + i) = make_uint4(s, s + v.x, s + v.x + v.y, s + v.x + v.y + v.z);
    carry += total;
  }
}

// Elements are stored with a stride of 8 within blocks of 256: the 32 elements that a warp reads
// together lie 8 apart in bin order.  Neighbours in bin order are neighbours in space; their adds to
// one mask word or record would take turns.
__device__ __forceinline__ uint32_t spread(uint32_t i) { return (i & ~255u) | (i & 7u) << 5 | ((i >> 3) & 31u); }
__device__ __forceinline__ uint32_t unspread(uint32_t i) { return (i & ~255u) | (i & 31u) << 3 | ((i >> 5) & 7u); }

// Elements into bin order.  Entry b + 1 of the bins holds the start of bin b and ends as its end,
// the start of bin b + 1: afterwards entry b is the start of bin b.
__global__ void __launch_bounds__(256) scatter_kernel(const __grid_constant__ LatticeArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t p0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane;
  if (p0 >= a.n) return;
  uint32_t lane_lt;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lane_lt));
  const int lists = a.mz * a.ncx;
  for (int i = 0; i < lists; ++i) {
    const size_t list = (size_t)blockIdx.y * lists + i;
    const bool have = lane < (int)__ldg(a.count + list * (a.n_pad / 32) + p0 / 32);
    const uint32_t mask = __ballot_sync(kFullMask, have);
    if (!have) continue;
    const uint4 e = __ldg(a.raw + list * a.n_pad + p0 + lane);
    // neighbouring elements share bins: one add per bin and warp
    const uint32_t bin = (e.x >> 16) * (uint32_t)a.nsy + (e.x & 0xFFFFu);
    const uint32_t same = __match_any_sync(mask, bin);
    uint32_t at = 0u;
    if ((same & lane_lt) == 0u) at = atomicAdd(a.bins + list * a.bin_stride + bin + 1, (uint32_t)__popc(same));
    at = __shfl_sync(mask, at, __ffs(same) - 1) + __popc(same & lane_lt);
    a.elems[list * a.n_pad + spread(at)] = e;
  }
}

// -----------------------------------------------------------------------------------
// Group evaluation
// -----------------------------------------------------------------------------------
// Shared memory: fixed part, then the chunk's arena (bit mask, places, records).
// Words of a pose's histogram of 16-bit counters: 4 past a multiple of 32, so that the same bin of
// different poses lies in different banks.
__host__ __device__ constexpr int hist_words(int K) { return (K * K + 1) / 2 / 32 * 32 + 36; }
// Rows planned at a time (one per thread).
__host__ __device__ constexpr int row_batch(int threads) { return threads < 512 ? threads : 512; }
struct EvalMem {
  uint32_t hist;     // byte offsets
  uint32_t row_of, by, cell_u, since, bx, rows, ends, ring, arena, arena_bytes;
};
template <int kNT>
__host__ __device__ inline EvalMem eval_mem(int K, int gx, int X, int Y, int nsy, int nsx, uint32_t total) {
  EvalMem m;
  uint32_t off = 2048;  // EvalCtl
  auto take = [&](uint32_t bytes) {
    const uint32_t o = off;
    off += (bytes + 15u) & ~15u;
    return o;
  };
  m.hist = take((uint32_t)(gx * hist_words(K)) * 4u);
  m.row_of = take((uint32_t)nsy * 2u);
  m.by = take((uint32_t)(Y + 1) * 2u);
  m.cell_u = take((uint32_t)nsx * 4u);
  m.since = take((uint32_t)nsx * 4u);
  m.bx = take((uint32_t)gx * (uint32_t)(X + 1) * 2u);
  m.rows = take((uint32_t)row_batch(kNT) * (2u + 4u + 4u));
  m.ends = take((uint32_t)row_batch(kNT) * 8u);
  m.ring = take((uint32_t)(kNT / 32) * kRing * 2u);
  m.arena = off;
  m.arena_bytes = total > off ? (total - off) & ~15u : 0u;
  if (m.arena_bytes > 8191u * 16u) m.arena_bytes = 8191u * 16u;  // 13-bit records in the ring
  return m;
}
// Arena bytes of a row's mask words (or summary words) and places, and of an occupied cell (with a mask
// word of its own when sparse).
__host__ __device__ constexpr uint32_t row_cost(uint32_t W, bool sparse) { return 6u * (sparse ? W / 32u + 1u : W); }
__host__ __device__ constexpr uint32_t cell_cost(bool sparse) { return sparse ? 22u : 16u; }
constexpr uint32_t kArenaSlack = 160;  // the last record and the padding of masks and places

struct EvalCtl {
  uint32_t tmp[3][32];
  uint32_t tmp2[32], tmp3[32];
  uint32_t vt32[64];    // variance thresholds below 2^32 (sym32), padded with 2^32 - 1
  uint32_t ct[64];      // count thresholds, padded with 2^32 - 1
  int32_t box[kLatticeGroup][6];
  float tx[kLatticeGroup];
  int32_t pose[kLatticeGroup];
  uint32_t wide[kLatticeGroup];
  uint32_t item, e0, e1, n_local, bound;
};
static_assert(sizeof(EvalCtl) <= 2048, "control block");

// Elements are streamed: they leave the small L1 to the tables.
__device__ __forceinline__ uint4 load_element(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ uint2 load_element_cell(const uint4* p) {
  uint2 v;
  asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}

__device__ __forceinline__ void copy_async4(uint32_t to, const uint32_t* from) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to), "l"(from) : "memory");
}

// Number of thresholds reached (a prefix of the ascending list), by descending powers of two.
__device__ __forceinline__ uint32_t count_level32(const uint32_t* ct, int top, uint32_t n) {
  uint32_t pos = 0u;
  for (uint32_t step = (uint32_t)top; step; step >>= 1)
    if (ct[pos + step - 1u] <= n) pos += step;
  return pos;
}

// kSparse: rows with few occupied cells.  A summary bit per mask word, and words only for the marked
// ones (see LatticeArgs::sparse).
template <int kNT, int kFeat, bool kSparse>
__global__ void __launch_bounds__(kNT, 1024 / kNT) lattice_eval_kernel(const __grid_constant__ LatticeArgs a) {
  constexpr int kNW = kNT / 32;
  constexpr bool kVar = kFeat != 0;
  constexpr int kRowBatch = row_batch(kNT);
  extern __shared__ __align__(128) uint8_t sm[];
  EvalCtl& C = *reinterpret_cast<EvalCtl*>(sm);
  const GridConst& gc = a.gc;
  const int K = gc.K, KK = K * K;
  const int hist_stride = hist_words(K);  // words of one pose's 16-bit counters
  const EvalMem mem = eval_mem<kNT>(K, a.gx, gc.X, gc.Y, a.nsy, a.nsx, a.smem_bytes);
  uint32_t* hist = reinterpret_cast<uint32_t*>(sm + mem.hist);
  uint16_t* row_of = reinterpret_cast<uint16_t*>(sm + mem.row_of);
  uint16_t* by = reinterpret_cast<uint16_t*>(sm + mem.by);
  float* cell_u = reinterpret_cast<float*>(sm + mem.cell_u);
  uint32_t* since = reinterpret_cast<uint32_t*>(sm + mem.since);
  uint16_t* bx = reinterpret_cast<uint16_t*>(sm + mem.bx);
  uint32_t* row_key = reinterpret_cast<uint32_t*>(sm + mem.rows);
  uint32_t* row_kk = row_key + kRowBatch;
  uint16_t* row_local = reinterpret_cast<uint16_t*>(row_kk + kRowBatch);
  const uint32_t* ends = reinterpret_cast<const uint32_t*>(sm + mem.ends);
  const uint32_t ends_at = (uint32_t)__cvta_generic_to_shared(sm + mem.ends);
  uint32_t* bits = reinterpret_cast<uint32_t*>(sm + mem.arena);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t lane_lt;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lane_lt));
  uint16_t* ring = reinterpret_cast<uint16_t*>(sm + mem.ring) + warp * kRing;
  const int all_hist = a.gx * hist_stride;
  const int X = gc.X, Y = gc.Y;
  const float inv_res = gc.inv_res;
  // largest power of two in the searches over Lv - 1 and Lc - 1 thresholds
  const int top_v = gc.Lv > 1 ? 1 << (31 - __clz(gc.Lv - 1)) : 0;
  const int top_c = gc.Lc > 1 ? 1 << (31 - __clz(gc.Lc - 1)) : 0;
  for (int i = tid; i < 64; i += kNT) {
    C.ct[i] = i < gc.Lc - 1 ? gc.count_thresh[i] : 0xFFFFFFFFu;
    C.vt32[i] = i < gc.Lv - 1 ? (uint32_t)min((int64_t)0xFFFFFFFFll, gc.var_thresh[i]) : 0xFFFFFFFFu;
  }

  int cur_c = -1, cur_iy = -1;
  uint32_t share = 256u;  // cells planned for, of 256 elements of a row
  uint32_t next = blockIdx.x;  // thread 0: the next item (the first ones are dealt out)
  for (;;) {
    if (tid == 0) C.item = next;
    for (int i = tid; i < all_hist; i += kNT) hist[i] = 0u;
    __syncthreads();
    const uint32_t item = C.item;
    if (item >= (uint32_t)a.n_items) break;
    if (tid == 0) next = gridDim.x + atomicAdd(a.next_item, 1u);  // needed only after this item
    // item -> (list = (rotation, t'_z, t'_x chunk), t'_y), whole or a part: groups that read one
    // list are adjacent
    const bool whole = item < (uint32_t)a.n_whole;
    const uint32_t n_split = whole ? 1u : (uint32_t)a.n_split;
    const uint32_t part = whole ? 0u : (item - (uint32_t)a.n_whole) % n_split;
    uint32_t q = whole ? item : (uint32_t)a.n_whole + (item - (uint32_t)a.n_whole) / n_split;
    const int iy = (int)(q % (uint32_t)a.my);
    const uint32_t list = q / (uint32_t)a.my;
    const int c = (int)(list % (uint32_t)a.ncx);
    q = list / (uint32_t)a.ncx;
    const int iz = (int)(q % (uint32_t)a.mz), r = (int)(q / (uint32_t)a.mz);
    const int x0 = c * a.gx, G = min(a.gx, a.mxr - x0);
    const uint32_t* off = a.bins + (size_t)list * a.bin_stride;
    const uint4* elems = a.elems + (size_t)list * a.n_pad;
    const uint32_t sx_end = (uint32_t)(G * (X + 1));
    const uint32_t W = sx_end / 32u + 1u;  // a word for every cell up to sx_end
    if (tid < G) {
      const int p = __ldg(a.pose_of + (((size_t)(a.r0 + r) * a.mz + iz) * a.my + iy) * a.mx + a.ix0 + x0 + tid);
      C.pose[tid] = p;
      C.tx[tid] = __ldg(a.poses + 12 * (size_t)p + 9);
      C.wide[tid] = 0u;
#pragma unroll
      for (int i = 0; i < 6; ++i) C.box[tid][i] = i < 3 ? INT_MAX : INT_MIN;
    }
    if (iy != cur_iy) {
      for (int i = tid; i < a.nsy; i += kNT) row_of[i] = __ldg(a.row_of + (size_t)iy * a.nsy + i);
      for (int i = tid; i <= Y; i += kNT) by[i] = (uint16_t)__ldg(a.by + (size_t)iy * (Y + 1) + i);
      cur_iy = iy;
    }
    if (c != cur_c) {
      for (int i = tid; i < (int)sx_end; i += kNT) {
        cell_u[i] = __ldg(a.cell_u + (size_t)c * a.nsx + i);
        since[i] = kFullMask;
      }
      for (int i = tid; i < G * (X + 1); i += kNT) bx[i] = __ldg(a.bx + (size_t)x0 * (X + 1) + i);
      __syncthreads();
      // per x cell, 4 bits per pose: cells since the pose's voxel began (15: outside its grid)
      for (int i = tid; i < G * (X + 1); i += kNT) {
        const int g = i / (X + 1);
        if (i - g * (X + 1) == X) continue;
        const uint32_t b = bx[i], e = bx[i + 1];
        for (uint32_t k = b; k < e; ++k) atomicAnd(since + k, ~(15u << 4 * g) | min(k - b, 14u) << 4 * g);
      }
      cur_c = c;
    }
    __syncthreads();

    // this part's rows: those whose first element lies in its share of the list
    const int n_rows = gc.Z * Y;
    int row = 0, row_end = n_rows;
    if (n_split > 1u) {
      const uint32_t n_list = __ldg(off + (size_t)gc.Z * a.nsy);
      // the first row that starts at or after j / n_split of the list, for j = part and part + 1
      const uint32_t target0 = (uint32_t)((uint64_t)n_list * part / n_split);
      const uint32_t target1 = (uint32_t)((uint64_t)n_list * (part + 1u) / n_split);
      auto start = [&](int lin) {
        if (lin >= n_rows) return kFullMask;
        const int kz = lin / Y;
        return __ldg(off + (size_t)kz * a.nsy + by[lin - kz * Y]);
      };
      const int stride = (n_rows + kNT - 1) / kNT;
      const uint32_t st = start(tid * stride);
      const int c0 = __syncthreads_count(st < target0), c1 = __syncthreads_count(st < target1);
      row = max(0, (c0 - 1) * stride);
      row_end = max(0, (c1 - 1) * stride);
      const int b0 = row, b1 = row_end;
      for (int i = 0; i < stride; i += kNT) {
        const bool on = i + tid < stride;
        const uint32_t s0 = on && c0 > 0 ? start(b0 + i + tid) : kFullMask;
        const uint32_t s1 = on && c1 > 0 ? start(b1 + i + tid) : kFullMask;
        row += __syncthreads_count(s0 < target0);
        row_end += __syncthreads_count(s1 < target1);
      }
      if (part == 0u) row = 0;
      if (part == n_split - 1u) row_end = n_rows;
    }
    // First and last elements of the next rows, one row per thread: copied to shared memory while the
    // chunk before is evaluated (held in registers they are spilled, and the spill waits for them).
    // A thread's copies are not ordered among themselves: those of the rows fetched before (a chunk
    // that is planned again) land first, or the plan could read them in place of the new ones.
    auto fetch_rows = [&]() {
      asm volatile("cp.async.wait_all;" ::: "memory");
      const int lin = row + tid;
      if (tid < kRowBatch && lin < row_end) {
        const int kz = lin / Y, ky = lin - kz * Y;
        const uint32_t* o = off + (size_t)kz * a.nsy;
        copy_async4(ends_at + 8u * tid, o + by[ky]);
        copy_async4(ends_at + 8u * tid + 4u, o + by[ky + 1]);
      }
    };
    fetch_rows();
    uint32_t voxels_max = 0u;  // bound of the counts in the 16-bit histograms

    // add the histograms to the poses' global ones
    auto flush = [&](bool clear) {
      for (int g = 0; g < G; ++g) {
        uint32_t* oc = a.out_c + (size_t)C.pose[g] * KK;
        const uint32_t* h = hist + g * hist_stride;
        for (int i = tid; 2 * i < KK; i += kNT) {
          const uint32_t v = h[i];
          if (v & 0xFFFFu) atomicAdd(oc + 2 * i, v & 0xFFFFu);
          if (v >> 16) atomicAdd(oc + 2 * i + 1, v >> 16);
        }
      }
      if (clear) {
        __syncthreads();
        for (int i = tid; i < all_hist; i += kNT) hist[i] = 0u;
      }
    };

    // The item's remaining rows are left out: its poses are finished by the exact path.
    auto give_up = [&]() {
      if (tid < G) C.wide[tid] = 1u;
    };

    while (row < row_end) {
      // ---- plan: as many of the next rows as fit the arena ----
      // cells of a row: at most its elements; `share` (of 256) of that bound as the last chunks had it
      uint32_t flag = 0u, cells = 0u;
      asm volatile("cp.async.wait_all;" ::: "memory");
      uint32_t o0 = 0u, o1 = 0u;
      const int lin = row + tid;
      const int n_here = min(kRowBatch, row_end - row);
      if (tid < n_here) {
        o0 = ends[2 * tid];
        o1 = ends[2 * tid + 1];
        flag = o1 > o0 ? 1u : 0u;
        cells = min(o1 - o0, sx_end);
      }
      uint32_t total;
      // cells < 2^21 in all (the host checks), the count of non-empty rows above it
      const uint32_t before = block_scan<kNW>(cells | flag << 21, C.tmp[0], total);
      const uint32_t cells_in = (before & 0x1FFFFFu) + cells, rows_in = (before >> 21) + flag;
      const bool fits = tid < n_here && ((cells_in * share + 255u) >> 8) * cell_cost(kSparse) +
                                                rows_in * row_cost(W, kSparse) + kArenaSlack <=
                                            mem.arena_bytes;
      const int taken = __syncthreads_count(fits);
      if (taken == 0) {  // never: the arena holds any one row (lattice_layout); else the exact path has its poses
        give_up();
        break;
      }
      if (tid < taken) {
        const uint32_t rl = before >> 21;
        row_local[tid] = flag ? (uint16_t)rl : (uint16_t)kNoRow;
        if (flag) {
          const int kz = lin / Y, ky = lin - kz * Y;
          const bool in_a = ky >= gc.boxA[1] && ky <= gc.boxA[4] && kz >= gc.boxA[2] && kz <= gc.boxA[5];
          row_key[rl] = (uint32_t)lin * (uint32_t)X | (in_a ? 0x80000000u : 0u);
          row_kk[rl] = (uint32_t)kz << 16 | (uint32_t)ky;
        }
        if (tid == 0) C.e0 = o0;
        if (tid == taken - 1) {
          C.e1 = o1;
          C.n_local = rl + flag;
          C.bound = cells_in;
        }
      }
      __syncthreads();
      const uint32_t n_local = C.n_local, e0 = C.e0, e1 = C.e1, bound = C.bound;
      const int row0 = row;
      row += taken;
      fetch_rows();
      if (n_local == 0u) {
        __syncthreads();  // C.e0.. are written again by the next plan
        continue;
      }
      constexpr uint32_t kB1 = 8, kB2 = 4;  // elements per thread and round of the two passes
      uint2 w1[kB1];
      auto load1 = [&](uint32_t eb) {  // past the end: y cell 0, which is in no row
#pragma unroll
        for (uint32_t j = 0; j < kB1; ++j)
          w1[j] = unspread(eb + j * kNT) - e0 < e1 - e0 ? load_element_cell(elems + eb + j * kNT) : make_uint2(0u, 0u);
      };
      const uint32_t eb0 = (e0 & ~255u) + tid, eb1 = (e1 + 255u) & ~255u;  // whole blocks
      load1(eb0);
      const uint32_t W1 = kSparse ? W / 32u + 1u : W;  // words (summary words) per row
      const uint32_t n_top4 = (n_local * W1 + 3u) / 4u;
      uint32_t* top = bits;  // summary bits, or the mask words themselves
      uint16_t* top_place = reinterpret_cast<uint16_t*>(bits + 4u * n_top4);
      for (uint32_t i = tid; i < n_top4; i += kNT) reinterpret_cast<uint4*>(top)[i] = make_uint4(0u, 0u, 0u, 0u);
      __syncthreads();
      // ---- occupied cells of every row ----
      // an element's row (false: outside the grid for every pose of the group)
      auto locate = [&](const uint2& w, uint32_t& rl) {
        const uint32_t k = row_of[w.x & 0xFFFFu];
        const uint32_t at = (w.x >> 16) * (uint32_t)Y + k - (uint32_t)row0;
        if (k >= (uint32_t)Y || at >= (uint32_t)taken) return false;
        rl = row_local[at];
        return true;
      };
      auto each_element = [&](auto&& f) {  // the elements' rows and cells; the first round is loaded
        for (uint32_t eb = eb0; eb < eb1;) {
#pragma unroll
          for (uint32_t j = 0; j < kB1; ++j) {
            uint32_t rl;
            if (locate(w1[j], rl)) f(rl, w1[j].y & 0xFFFFu);
          }
          eb += kB1 * kNT;
          if (eb < eb1) load1(eb);
        }
      };
      if (kSparse) {
        each_element([&](uint32_t rl, uint32_t sx) { atomicOr(top + rl * W1 + (sx >> 10), 1u << ((sx >> 5) & 31u)); });
        load1(eb0);
      } else {
        each_element([&](uint32_t rl, uint32_t sx) { atomicOr(top + rl * W1 + (sx >> 5), 1u << (sx & 31u)); });
      }
      __syncthreads();
      // ---- places: set bits before each word ----
      // each thread takes consecutive groups of four words; their counts stay in registers
      auto counts = [&](const uint32_t* v, uint32_t i) {  // four 8-bit counts
        const uint4 q = reinterpret_cast<const uint4*>(v)[i];
        return (q.x | q.y | q.z | q.w) == 0u
                   ? 0u
                   : (uint32_t)(__popc(q.x) | __popc(q.y) << 8 | __popc(q.z) << 16 | __popc(q.w) << 24);
      };
      auto places = [&](const uint32_t* v, uint16_t* to, uint32_t n4, uint32_t* tmp) {
        const uint32_t per = (n4 + kNT - 1) / kNT;
        const uint32_t wb = min((uint32_t)tid * per, n4), we = min(wb + per, n4);
        constexpr uint32_t kKeep = 4;
        uint32_t kept[kKeep], cnt = 0u, total;
#pragma unroll
        for (uint32_t j = 0; j < kKeep; ++j) {
          kept[j] = wb + j < we ? counts(v, wb + j) : 0u;
          cnt = __dp4a(kept[j], 0x01010101u, cnt);
        }
        for (uint32_t i = wb + kKeep; i < we; ++i) cnt = __dp4a(counts(v, i), 0x01010101u, cnt);
        uint32_t s_w = block_scan<kNW>(cnt, tmp, total);
        auto store = [&](uint32_t i, uint32_t k) {
          const uint32_t p1 = s_w + (k & 0xFFu), p2 = p1 + ((k >> 8) & 0xFFu), p3 = p2 + ((k >> 16) & 0xFFu);
          reinterpret_cast<uint2*>(to)[i] = make_uint2(s_w | p1 << 16, p2 | p3 << 16);
          s_w = p3 + (k >> 24);
        };
#pragma unroll
        for (uint32_t j = 0; j < kKeep; ++j)
          if (wb + j < we) store(wb + j, kept[j]);
        for (uint32_t i = wb + kKeep; i < we; ++i) store(i, counts(v, i));
        return total;
      };
      uint32_t* words = top;  // mask words and the set bits before each
      uint16_t* place = top_place;
      uint32_t used = 24u * n_top4 + (n_top4 & 1u) * 8u;  // arena bytes so far
      bool over = false;
      // a cell's mask word: its place among the words, and its bits (none set: not among them)
      auto word_at = [&](uint32_t rl, uint32_t sx, uint32_t& idx) {
        if (!kSparse) {
          idx = rl * W + (sx >> 5);
          return words[idx];
        }
        const uint32_t wi = rl * W1 + (sx >> 10), b = (sx >> 5) & 31u, m = top[wi];
        idx = top_place[wi] + __popc(m & ((1u << b) - 1u));
        return (m >> b) & 1u ? words[idx] : 0u;
      };
      uint4 w2[kB2];  // the first elements of the pass over sums, loaded meanwhile
      auto load2 = [&](uint32_t eb) {
#pragma unroll
        for (uint32_t j = 0; j < kB2; ++j)
          w2[j] = unspread(eb + j * kNT) - e0 < e1 - e0 ? load_element(elems + eb + j * kNT) : make_uint4(0u, 0u, 0u, 0u);
      };
      uint32_t M, n_words = 0u;
      if constexpr (kSparse) {
        n_words = places(top, top_place, n_top4, C.tmp2);
        const uint32_t n4 = n_words / 4u + 1u;  // one word past the last, for cells after it
        words = reinterpret_cast<uint32_t*>(sm + mem.arena + used);
        place = reinterpret_cast<uint16_t*>(words + 4u * n4);
        used += 24u * n4 + (n4 & 1u) * 8u;
        over = used + 16u > mem.arena_bytes;
        if (!over)
          for (uint32_t i = tid; i < n4; i += kNT) reinterpret_cast<uint4*>(words)[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        if (!over) {
          each_element([&](uint32_t rl, uint32_t sx) {
            uint32_t idx;
            word_at(rl, sx, idx);
            atomicOr(words + idx, 1u << (sx & 31u));
          });
          load2(eb0);
        }
        __syncthreads();
        M = 0u;
        if (!over) M = places(words, place, n4, C.tmp3);
      } else {
        load2(eb0);
        M = places(words, place, n_top4, C.tmp2);
      }
      // more than planned: fewer rows
      if (over || M > 8190u || used + 16u * (M + 1u) > mem.arena_bytes) {
        if (share == 256u) {  // never: the bound holds
          give_up();
          break;
        }
        const uint32_t need = over ? share + share / 2u : kSparse ? (16u * M + 6u * n_words) * 13u / bound : (M * 280u) / bound;
        share = min(256u, max(share + 1u, need + 8u));  // as these rows have it
        row = row0;
        fetch_rows();
        __syncthreads();
        continue;
      }
      uint4* rec = reinterpret_cast<uint4*>(sm + mem.arena + used);
      // (rows of one layer differ: falling slowly saves planning them twice)
      const uint32_t seen = kSparse ? (16u * M + 6u * n_words) * 13u / bound : (M * 290u) / bound;
      share = max(min(256u, seen + 8u), share - share / 8u);
      for (uint32_t i = tid; i <= M; i += kNT) rec[i] = make_uint4(0u, 0u, 0u, 0u);
      __syncthreads();
      // ---- sums per cell: records n, S1, S2, row << 16 | cell ----
      for (uint32_t eb = eb0; eb < eb1;) {
#pragma unroll
        for (uint32_t j = 0; j < kB2; ++j) {
          const uint4 w = w2[j];
          uint32_t rl, idx;
          if (!locate(make_uint2(w.x, w.y), rl)) continue;
          const uint32_t m = word_at(rl, w.y & 0xFFFFu, idx);
          const uint32_t at = place[idx] + __popc(m & ((1u << (w.y & 31u)) - 1u));
          // word j of a record at j ^ sw meanwhile: one word of 32 records in 32 banks, not in 8
          uint32_t* rc = reinterpret_cast<uint32_t*>(rec + at);
          const uint32_t sw = (at >> 3) & 3u;
          rc[3u ^ sw] = rl << 16 | (w.y & 0xFFFFu);
          atomicAdd(rc + sw, w.y >> 16);
          if (kVar) {
            atomicAdd(rc + (1u ^ sw), w.z);
            atomicAdd(rc + (2u ^ sw), w.w);
          }
        }
        eb += kB2 * kNT;
        if (eb < eb1) load2(eb);
      }
      __syncthreads();
      // ---- running sums (exclusive; record M holds the totals) ----
      {
        // each thread takes consecutive records, an odd number (bank conflicts)
        const uint32_t pr = (M + kNT) / kNT | 1u;
        const uint32_t rb = min((uint32_t)tid * pr, M + 1u), re = min(rb + pr, M + 1u);
        auto record = [&](uint32_t i) {  // in order
          const uint4 v = rec[i];
          const bool p = (i >> 3) & 1u, q = (i >> 4) & 1u;
          const uint4 u = make_uint4(p ? v.y : v.x, p ? v.x : v.y, p ? v.w : v.z, p ? v.z : v.w);
          return make_uint4(q ? u.z : u.x, q ? u.w : u.y, q ? u.x : u.z, q ? u.y : u.w);
        };
        uint32_t t0 = 0u, t1 = 0u, t2 = 0u;
        for (uint32_t i = rb; i < re; ++i) {
          const uint4 v = record(i);
          t0 += v.x;
          t1 += v.y;
          t2 += v.z;
        }
        const uint32_t i0 = warp_scan(t0), i1 = kVar ? warp_scan(t1) : 0u, i2 = kVar ? warp_scan(t2) : 0u;
        if (lane == 31) {
          C.tmp[0][warp] = i0;
          if (kVar) C.tmp[1][warp] = i1, C.tmp[2][warp] = i2;
        }
        __syncthreads();
        auto before_warp = [&](int j) { return __reduce_add_sync(kFullMask, lane < warp ? C.tmp[j][lane] : 0u); };
        uint32_t s0 = before_warp(0) + i0 - t0, s1 = 0u, s2 = 0u;
        if (kVar) s1 = before_warp(1) + i1 - t1, s2 = before_warp(2) + i2 - t2;
        for (uint32_t i = rb; i < re; ++i) {
          const uint4 v = record(i);
          rec[i] = make_uint4(s0, s1, s2, v.w);
          s0 += v.x;
          s1 += v.y;
          s2 += v.z;
        }
      }
      if (voxels_max + M > 65535u) {
        flush(true);
        voxels_max = 0u;
      }
      voxels_max += M;
      __syncthreads();

      // cells of row rl before cell s (s <= sx_end), counted from the chunk's first
      auto cells_before = [&](uint32_t rl, uint32_t s) {
        uint32_t idx;
        const uint32_t m = word_at(rl, s, idx);
        return (uint32_t)place[idx] + (uint32_t)__popc(m & ((1u << (s & 31u)) - 1u));
      };
      // ---- occupied box: rows with a cell inside the grid, their first and last cell ----
      // A lane per (row, pose): four rows and eight poses per warp.
      for (uint32_t rb = 4u * warp; rb < n_local; rb += 4u * kNW) {
        const uint32_t rl = rb + (lane >> 3);
        const int g = lane & 7;
        uint32_t s0 = kFullMask, s1 = 0u;
        int vy = 0, vz = 0;
        bool any = false;
        if (rl < n_local && g < G) {
          const uint32_t i0 = cells_before(rl, bx[g * (X + 1)]), i1 = cells_before(rl, bx[g * (X + 1) + X]);
          any = i0 < i1;
          if (any) {
            s0 = rec[i0].w & 0xFFFFu;
            s1 = rec[i1 - 1u].w & 0xFFFFu;
            vy = (int)(row_kk[rl] & 0xFFFFu);
            vz = (int)(row_kk[rl] >> 16);
          }
        }
        int y0 = any ? vy : INT_MAX, y1 = any ? vy : INT_MIN, z0 = any ? vz : INT_MAX, z1 = any ? vz : INT_MIN;
#pragma unroll
        for (int d = 8; d < 32; d <<= 1) {
          s0 = min(s0, __shfl_xor_sync(kFullMask, s0, d));
          s1 = max(s1, __shfl_xor_sync(kFullMask, s1, d));
          y0 = min(y0, __shfl_xor_sync(kFullMask, y0, d));
          y1 = max(y1, __shfl_xor_sync(kFullMask, y1, d));
          z0 = min(z0, __shfl_xor_sync(kFullMask, z0, d));
          z1 = max(z1, __shfl_xor_sync(kFullMask, z1, d));
        }
        if (lane < 8 && s0 != kFullMask) {  // k_x is monotone in the cell
          atomicMin(&C.box[g][0], axis_k(cell_u[s0], C.tx[g], inv_res, X));
          atomicMin(&C.box[g][1], y0);
          atomicMin(&C.box[g][2], z0);
          atomicMax(&C.box[g][3], axis_k(cell_u[s1], C.tx[g], inv_res, X));
          atomicMax(&C.box[g][4], y1);
          atomicMax(&C.box[g][5], z1);
        }
      }

      // ---- voxels of every pose: stretches of records with equal (row, k_x) ----
      uint32_t fill = 0u;
      struct Voxel {
        uint32_t g, n, s1, s2, sA;
        bool in_a;
      };
      auto fetch = [&](uint32_t w) {  // the voxel of pose w >> 13 that starts at record w & 0x1FFF
        Voxel v;
        const uint4 b = rec[w & 0x1FFFu];
        v.g = w >> 13;
        const uint32_t rl = b.w >> 16;
        const uint32_t rk = row_key[rl];
        const int kx = __float2int_rd(__fmul_rn(__fadd_rn(cell_u[b.w & 0xFFFFu], C.tx[v.g]), inv_res));
        v.sA = __ldg(a.symA + ((rk & 0x7FFFFFFFu) + (uint32_t)kx));
        v.in_a = (rk >> 31) && kx >= gc.boxA[0] && kx <= gc.boxA[3];
        // it ends where the pose's next voxel begins
        const uint4 e = rec[cells_before(rl, bx[v.g * (uint32_t)(X + 1) + (uint32_t)kx + 1u])];
        v.n = e.x - b.x;
        v.s1 = e.y - b.y;
        v.s2 = e.z - b.z;
        return v;
      };
      auto symbol = [&](const Voxel& v) {
        uint32_t lc = 0u, lv = 0u;
        const uint32_t n = v.n;
        if (kFeat != 1) lc = count_level32(C.ct, top_c, n);
        if (kVar) {
          const int32_t S1 = (int32_t)v.s1;
          const uint64_t spread = (uint64_t)n * v.s2 - (uint64_t)((int64_t)S1 * S1);
          if (gc.sym32) {  // n < 2^16 and every threshold < 2^32
            const uint32_t n2 = n * n;
            if (top_v <= 8) {
#pragma unroll
              for (uint32_t step = 8u; step; step >>= 1)
                if ((uint64_t)C.vt32[lv + step - 1u] * n2 <= spread) lv += step;
            } else {
              for (uint32_t step = 32u; step; step >>= 1)
                if ((uint64_t)C.vt32[lv + step - 1u] * n2 <= spread) lv += step;
            }
          } else {
            const uint64_t n2 = (uint64_t)n * n;
            for (uint32_t step = (uint32_t)top_v; step; step >>= 1) {
              const uint64_t th = lv + step < (uint32_t)gc.Lv ? (uint64_t)gc.var_thresh[lv + step - 1u] : ~0ull;
              if (__umul64hi(th, n2) == 0ull && th * n2 <= spread && lv + step < (uint32_t)gc.Lv) lv += step;
            }
          }
        }
        return 1u + (kFeat == 2 ? lc * (uint32_t)gc.Lv + lv : lc + lv);
      };
      auto count = [&](const Voxel& v, uint32_t sB) {
        if (kVar && v.n > gc.nlim3c) C.wide[v.g] = 1u;  // the 32-bit sums may have wrapped: exact path
        if (v.in_a) {
          const uint32_t h = v.sA * (uint32_t)K + sB;
          atomicAdd(hist + v.g * (uint32_t)hist_stride + (h >> 1), 1u << ((h & 1u) * 16u));
        }
      };
      auto voxel = [&](uint32_t w) {
        const Voxel v = fetch(w);
        count(v, symbol(v));
      };
      for (uint32_t b = 32u * warp; b < M; b += kNT) {
        const uint32_t i = b + lane;
        const uint32_t w = i < M ? rec[i].w : 0u;
        uint32_t pw = __shfl_up_sync(kFullMask, w, 1);
        if (lane == 0) pw = i > 0u ? rec[i - 1u].w : kFullMask;
        // cells since the record before (at most 15, as in another row): a pose's voxel starts here
        // if it began after that record, i.e. fewer cells ago
        const uint32_t gap = (w ^ pw) >> 16 ? 15u : min(15u, w - pw);
        const uint32_t sn = i < M ? since[w & 0xFFFFu] : kFullMask;
        const uint32_t gap4 = gap * 0x01010101u;
        const uint32_t even = (sn & 0x0F0F0F0Fu) + 0x10101010u - gap4;  // bit 4 of a byte: since >= gap
        const uint32_t odd = ((sn >> 4) & 0x0F0F0F0Fu) + 0x10101010u - gap4;
        const uint32_t starts = (~even & 0x10101010u) >> 4 | (~odd & 0x10101010u) >> 3;
        // places in the ring: prefix sums of the counts (0 to 8) by ballots of their bits
        const uint32_t cnt = __popc(starts);
        uint32_t at = fill;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t m = __ballot_sync(kFullMask, (cnt >> k) & 1u);
          at += (uint32_t)__popc(m & lane_lt) << k;
          fill += (uint32_t)__popc(m) << k;
        }
#pragma unroll
        for (uint32_t g = 0; g < kLatticeGroup; ++g)
          if (starts >> (8u * (g >> 1) + (g & 1u)) & 1u) ring[at++] = (uint16_t)(i | g << 13);
        __syncwarp();
        while (fill >= 64u) {  // two voxels per lane: their chains of loads overlap
          fill -= 64u;
          const Voxel v0 = fetch(ring[fill + lane]), v1 = fetch(ring[fill + 32u + lane]);
          const uint32_t b0 = symbol(v0), b1 = symbol(v1);
          count(v0, b0);
          count(v1, b1);
        }
        __syncwarp();
      }
      if ((uint32_t)lane < fill) voxel(ring[lane]);
      if ((uint32_t)lane + 32u < fill) voxel(ring[lane + 32]);
      __syncthreads();
    }
    flush(false);
    if (tid < 6 * G) {
      const int g = tid / 6, i = tid - 6 * g;
      const int v = C.box[g][i];
      int32_t* ob = a.out_box + 6 * (size_t)C.pose[g] + i;
      if (i < 3 && v != INT_MAX) atomicMin(ob, v);
      if (i >= 3 && v != INT_MIN) atomicMax(ob, v);
    }
    if (tid < G && C.wide[tid] && atomicExch(a.redo_mark + C.pose[tid], 1u) == 0u)
      a.redo_list[atomicAdd(a.redo_count, 1u)] = (uint32_t)(a.pose_base + C.pose[tid]);
    __syncthreads();  // the histograms are read before the next item clears them
  }
}

// Dynamic shared memory of a CTA, 1,024 threads per SM (228 KB, 1 KB reserved per CTA).
constexpr uint32_t kSmemPair = 113u * 1024u;

// Room for one row of the largest size, and for the planner's 21-bit counts.
bool arena_ok(const EvalMem& m, int W, int nsx, int threads, bool sparse) {
  const uint64_t row = (uint64_t)nsx * cell_cost(sparse) + row_cost((uint32_t)W, sparse);
  return row + kArenaSlack <= m.arena_bytes && (uint64_t)nsx * row_batch(threads) < (1u << 21);
}

template <int kNT>
cudaError_t launch_eval_nt(const LatticeArgs& a, int n_ctas, cudaStream_t s) {
  constexpr bool kS = kNT == 1024;  // sparse rows with one CTA per SM only (lattice_layout)
  auto* k = a.sparse ? (a.gc.feature == 0   ? lattice_eval_kernel<kNT, 0, kS>
                        : a.gc.feature == 1 ? lattice_eval_kernel<kNT, 1, kS>
                                            : lattice_eval_kernel<kNT, 2, kS>)
                     : (a.gc.feature == 0   ? lattice_eval_kernel<kNT, 0, false>
                        : a.gc.feature == 1 ? lattice_eval_kernel<kNT, 1, false>
                                            : lattice_eval_kernel<kNT, 2, false>);
  k<<<n_ctas, kNT, a.smem_bytes, s>>>(a);
  return cudaGetLastError();
}
template <int kNT>
cudaError_t setup_nt(int smem) {
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaSuccess;
  for (auto* k : {lattice_eval_kernel<kNT, 0, false>, lattice_eval_kernel<kNT, 1, false>, lattice_eval_kernel<kNT, 2, false>,
                  lattice_eval_kernel<kNT, 0, kNT == 1024>, lattice_eval_kernel<kNT, 1, kNT == 1024>,
                  lattice_eval_kernel<kNT, 2, kNT == 1024>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, attr, smem);
  return e;
}

}  // namespace

bool lattice_layout(LatticeArgs& a, int mx, size_t smem_optin) {
  const GridConst& gc = a.gc;
  if (a.my > kLatticeMaxY || a.mz > kLatticeMaxZ || mx < 1) return false;
  const int64_t nsy = (int64_t)a.my * (gc.Y + 1) + 1;
  // 16-bit cell, row and layer indices, 22-bit k_x keys; the row search takes n_rows <= threads^2
  if (nsy > 65535 || gc.Y >= 65535 || gc.Z >= 65535 || gc.X >= (1 << 20)) return false;
  if ((int64_t)gc.Z * gc.Y > (1 << 18) || (int64_t)gc.Z * nsy > (1 << 27)) return false;
  a.nsy = (int)nsy;
  a.n_pad = (a.n + 255) / 256 * 256;
  a.bin_stride = ((int64_t)gc.Z * nsy + 1 + 3) / 4 * 4;
  for (int group = kLatticeGroup; group >= 4; group /= 2) {  // wide grids: fewer cells with fewer t'_x
    a.mxr = std::min(mx, kLatticeMaxX);
    a.ncx = (a.mxr + group - 1) / group;
    a.gx = (a.mxr + a.ncx - 1) / a.ncx;
    a.ncx = (a.mxr + a.gx - 1) / a.gx;
    const int64_t nsx = (int64_t)a.gx * (gc.X + 1) + 1;
    if (nsx > 65535) continue;
    a.nsx = (int)nsx;
    const int W = (int)((nsx - 1) / 32 + 1);
    const EvalMem m2 = eval_mem<512>(gc.K, a.gx, gc.X, gc.Y, a.nsy, a.nsx, kSmemPair);
    if (arena_ok(m2, W, a.nsx, 512, false) && m2.arena_bytes >= 32u * 1024u && smem_optin >= kSmemPair) {
      a.threads = 512;
      a.sparse = 0;
      a.smem_bytes = kSmemPair;
      return true;
    }
    // One CTA per SM (large histograms, wide tables): nothing hides the fixed cost of a chunk, and rows
    // with few points against their mask words (at most half of the points' rows are counted) make
    // chunks small.  6.2 words per point (259k points, 400 x 400 x 40): 34.2 -> 28.4 ms.  With two CTAs
    // the third pass over the elements costs more than it saves: 6.9 words (120k, 320 x 320 x 32) 1.76
    // -> 1.85 ms, 5.9 (8k, 105 x 106 x 17) 0.18 -> 0.21, 2.1 (33k, 147 x 170 x 17) 0.44 -> 0.54.
    const int64_t rows = std::min<int64_t>((int64_t)gc.Z * gc.Y, a.n / 2);
    a.sparse = 4 * a.n < rows * W ? 1 : 0;
    const EvalMem m1 = eval_mem<1024>(gc.K, a.gx, gc.X, gc.Y, a.nsy, a.nsx, (uint32_t)smem_optin);
    if (arena_ok(m1, W, a.nsx, 1024, a.sparse != 0)) {
      a.threads = 1024;
      a.smem_bytes = (uint32_t)smem_optin;
      return true;
    }
  }
  return false;
}

cudaError_t lattice_setup() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0, smem = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (done[dev]) return cudaSuccess;
  if ((e = cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
  if ((e = setup_nt<512>(smem)) != cudaSuccess || (e = setup_nt<1024>(smem)) != cudaSuccess) return e;
  done[dev] = true;
  return cudaSuccess;
}

cudaError_t launch_lattice(LatticeArgs a, int32_t n_rot, int n_sm, cudaStream_t s, int32_t* launches) {
  cudaError_t e;
  const int32_t rot_round = a.n_rot, mx_round = a.mxr;
  a.first = 1;
  for (int32_t r0 = 0; r0 < n_rot; r0 += rot_round)
    for (int32_t ix0 = 0; ix0 < a.mx; ix0 += mx_round, a.first = 0) {
      a.r0 = r0;
      a.n_rot = std::min(rot_round, n_rot - r0);
      a.ix0 = ix0;
      a.mxr = std::min(mx_round, a.mx - ix0);
      a.ncx = (a.mxr + a.gx - 1) / a.gx;
      // Whole groups while every CTA gets one; the rest in parts, so that the last round of CTAs
      // costs little, each part with at least 4,096 points of the list (512 groups on 304 CTAs: 0.88
      // ms with two parts of every group, 0.79 ms so).
      const int32_t groups = a.n_rot * a.mz * a.my * a.ncx, slots = n_sm * (1024 / a.threads);
      a.n_whole = groups / slots * slots;
      if (a.n_whole > slots && groups - a.n_whole < slots / 2) a.n_whole -= slots;
      const int32_t rest = groups - a.n_whole;
      a.n_split = rest == 0 ? 1
                            : (int32_t)std::max<int64_t>(
                                  1, std::min<int64_t>({(3 * slots + rest - 1) / rest, a.n / 4096, 16}));
      a.n_items = a.n_whole + rest * a.n_split;
      setup_kernel<<<2 * n_sm, 256, 0, s>>>(a);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      if (a.n > 0) {
        const dim3 grid((unsigned)((a.n + 255) / 256), (unsigned)a.n_rot);
        points_kernel<<<grid, 256, 0, s>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        offsets_kernel<<<a.n_rot * a.mz * a.ncx, 1024, 0, s>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        scatter_kernel<<<grid, 256, 0, s>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
      }
      const int ctas = std::min(a.n_items, slots);
      e = a.threads == 512 ? launch_eval_nt<512>(a, ctas, s) : launch_eval_nt<1024>(a, ctas, s);
      if (e != cudaSuccess) return e;
      *launches += a.n > 0 ? 5 : 2;
    }
  return cudaSuccess;
}

}  // namespace mialign
