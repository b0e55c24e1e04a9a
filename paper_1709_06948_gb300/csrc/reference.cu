// reference.cu — Algorithm 1 initialisation for scan A (cold path, once per reference):
// voxelize A with the identity pose, its feature symbol per voxel, its occupied bbox,
// and per-symbol 3-D prefix sums used to count A's symbols over any overlap box.
#include <algorithm>
#include <climits>

#include "align_internal.h"
#include "device_common.cuh"

namespace mialign {

namespace {

__global__ void ref_accumulate_kernel(const GridConst gc, const float* __restrict__ xyz, int64_t n,
                                      const float* __restrict__ pose12, uint32_t* cnt, unsigned long long* s1,
                                      unsigned long long* s2) {
  Pose12 P;
#pragma unroll
  for (int i = 0; i < 9; ++i) P.r[i] = pose12[i];
#pragma unroll
  for (int i = 0; i < 3; ++i) P.t[i] = pose12[9 + i];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    int dz = 0;
    const uint32_t key =
        voxel_key(P, xyz[3 * i], xyz[3 * i + 1], xyz[3 * i + 2], gc.inv_res, gc.X, gc.Y, gc.Z, gc.res_mm, &dz);
    if (key == kEmptyKey) continue;
    atomicAdd(&cnt[key], 1u);
    atomicAdd(&s1[key], (unsigned long long)(long long)dz);
    atomicAdd(&s2[key], (unsigned long long)((long long)dz * dz));
  }
}

// Symbols of all voxels and the occupied box; the sums of the occupied ones are cleared again (they
// stay zero between references), and row_n counts them by (symbol, y).
__global__ void ref_symbols_kernel(const GridConst gc, uint32_t* __restrict__ cnt, unsigned long long* __restrict__ s1,
                                   unsigned long long* __restrict__ s2, uint8_t* symA, int32_t* box,
                                   uint32_t* __restrict__ row_n) {
  __shared__ uint32_t ct[kMaxLevels];
  __shared__ int64_t vt[kMaxLevels];
  for (int i = threadIdx.x; i < kMaxLevels; i += blockDim.x) {
    ct[i] = gc.count_thresh[i];
    vt[i] = gc.var_thresh[i];
  }
  __syncthreads();
  const int64_t V = (int64_t)gc.X * gc.Y * gc.Z;
  int mn[3] = {INT_MAX, INT_MAX, INT_MAX}, mx[3] = {INT_MIN, INT_MIN, INT_MIN};
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t n = cnt[v];
    if (n == 0) {
      symA[v] = 0;
      continue;
    }
    const int sym = feature_symbol(gc.feature, gc.Lc, gc.Lv, ct, vt, n, (int64_t)s1[v], s2[v]);
    cnt[v] = 0u;
    s1[v] = s2[v] = 0ull;
    symA[v] = (uint8_t)sym;
    const int kx = (int)(v % gc.X), ky = (int)((v / gc.X) % gc.Y), kz = (int)(v / ((int64_t)gc.X * gc.Y));
    const int k[3] = {kx, ky, kz};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      mn[i] = min(mn[i], k[i]);
      mx[i] = max(mx[i], k[i]);
    }
    if (row_n != nullptr) {  // one add per row and warp: neighbours share it
      const uint32_t row = (uint32_t)((sym - 1) * gc.Y + ky), same = __match_any_sync(__activemask(), row);
      if ((int)(threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&row_n[(size_t)row + 1], (uint32_t)__popc(same));
    }
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 3; ++i) {  // one update per warp
    const int lo = __reduce_min_sync(0xFFFFFFFFu, mn[i]), hi = __reduce_max_sync(0xFFFFFFFFu, mx[i]);
    if ((threadIdx.x & 31) == 0 && lo != INT_MAX) {
      atomicMin(&box[i], lo);
      atomicMax(&box[3 + i], hi);
    }
  }
}

// Exclusive prefix sums of n values in place, one block; *few: whether no symbol (Y values from entry 1
// on) counts more than `most` voxels.
__global__ void __launch_bounds__(1024) ref_rows_kernel(uint32_t* v, int64_t n, int Y, uint32_t most, int32_t* few) {
  __shared__ uint32_t tot[2][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t carry = 0u;
  int t = 0;
  for (int64_t i0 = 0; i0 < n; i0 += 1024, t ^= 1) {
    const int64_t i = i0 + threadIdx.x;
    const uint32_t x = i < n ? v[i] : 0u;
    uint32_t inc = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, inc, d);
      if (lane >= d) inc += u;
    }
    if (lane == 31) tot[t][w] = inc;
    __syncthreads();
    uint32_t all = tot[t][lane];  // every warp scans the warps' totals
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, all, d);
      if (lane >= d) all += u;
    }
    const uint32_t upto = __shfl_sync(0xFFFFFFFFu, all, (w + 31) & 31);
    const uint32_t before = carry + (w ? upto : 0u);
    all = __shfl_sync(0xFFFFFFFFu, all, 31);
    if (i < n) v[i] = before + inc - x;
    carry += all;
  }
  __syncthreads();  // entry 1 + a Y holds the start of symbol a's rows, the last entry that of the last row
  bool ok = true;
  const int64_t symbols = (n - 1) / Y;
  for (int64_t a = threadIdx.x; a < symbols; a += blockDim.x)
    ok = ok && (a + 1 < symbols ? v[1 + (a + 1) * Y] : carry) - v[1 + a * Y] <= most;
  ok = __syncthreads_and(ok);
  if (threadIdx.x == 0) *few = ok ? 1 : 0;
}

// The occupied voxels as x | z << 16, ordered by (symbol, y).  Entry r + 1 of row_n holds the start
// of row r and ends as its end: afterwards entry r is the start of row r.
__global__ void ref_list_kernel(const GridConst gc, const uint8_t* __restrict__ symA, uint32_t* row_n,
                                uint32_t* __restrict__ list, const int32_t* few) {
  if (*few == 0) return;
  const int64_t V = (int64_t)gc.X * gc.Y * gc.Z;
  for (int64_t v0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * 16; v0 < V;
       v0 += (int64_t)gridDim.x * blockDim.x * 16) {
    uint32_t q[4] = {0u, 0u, 0u, 0u};  // 16 symbols, the first in the lowest byte
    if (v0 + 16 <= V) {
      const uint4 w = *reinterpret_cast<const uint4*>(symA + v0);  // v0 is a multiple of 16
      q[0] = w.x, q[1] = w.y, q[2] = w.z, q[3] = w.w;
    } else {
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if (v0 + k < V) q[k / 4] |= (uint32_t)symA[v0 + k] << (8 * (k % 4));
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      for (uint32_t left = q[j]; left != 0u;) {
        const int k = (__ffs(left) - 1) / 8;
        const uint32_t sym = (left >> (8 * k)) & 0xFFu;
        left &= ~(0xFFu << (8 * k));
        const int64_t v = v0 + 4 * j + k;
        const uint32_t kx = (uint32_t)(v % gc.X), ky = (uint32_t)((v / gc.X) % gc.Y),
                       kz = (uint32_t)(v / ((int64_t)gc.X * gc.Y));
        list[atomicAdd(&row_n[(size_t)(sym - 1u) * gc.Y + ky + 1], 1u)] = kx | kz << 16;
      }
    }
  }
}

// sat[a-1][z][y][x] = #{ voxels (x', y', z') with x' < x, y' < y, z' < z and symA == a }.
//
// From the list of occupied voxels: a warp writes a strip of rows of one plane (a, z), starting from
// the counts per x of the strip's earlier rows and adding each row's voxels; a row without any is the
// row before.  Everything is written once and nothing but the list is read (the passes below write,
// read and write it again, and need it cleared): bound by the writes, 1.44 GB for 56 symbols on
// 400 x 400 x 40 voxels (0.25 to 0.3 ms, 5 TB/s; the whole reference of 87k points 1.69 -> 0.40 ms).
constexpr int64_t kSatMostBytes = 4096;  // sums' bytes per voxel of one symbol at least (launch_ref_sat_list)
constexpr int kSatRows = 31, kSatWarps = 4, kSatMaxX = 2048;  // rows per strip at most: a lane per row end

// kRegs: the running counts in registers (x = lane + 32 i, X <= 32 kRegs); 0: in shared memory.  Of a
// whole reference of 106k points and 56 symbols: 64 x 64 x 200 voxels 162 us with 5 registers, 184 with
// 13, 178 without; 160 x 160 x 16 125, 127, 126; 400 x 400 x 40 388 with 13, 390 without; 416 x 380 x 40,
// 15 symbols, 226 and 232.
template <int kRegs>
__global__ void __launch_bounds__(kSatWarps * 32) ref_sat_list_kernel(const GridConst gc,
                                                                      const uint32_t* __restrict__ row_n,
                                                                      const uint32_t* __restrict__ list,
                                                                      int32_t* __restrict__ sat, int strip_rows,
                                                                      const int32_t* few) {
  if (*few == 0) return;
  extern __shared__ int32_t cols[];  // per warp: X running counts (inclusive sums along x), X new counts
  int32_t reg[kRegs > 0 ? kRegs : 1];
  const int X = gc.X, Y = gc.Y, Z = gc.Z, X1 = X + 1, Y1 = Y + 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t* run = cols + (size_t)warp * 2 * X;
  int32_t* add = run + X;
  const int strips = (Y1 + strip_rows - 1) / strip_rows;
  const int64_t tasks = (int64_t)(gc.K - 1) * (Z + 1) * strips;
  for (int64_t task = blockIdx.x * (int64_t)kSatWarps + warp; task < tasks; task += (int64_t)gridDim.x * kSatWarps) {
    const int strip = (int)(task % strips);
    const int z = (int)((task / strips) % (Z + 1));
    const int a = (int)(task / ((int64_t)strips * (Z + 1)));
    const int y0 = strip * strip_rows, y1 = min(Y1, y0 + strip_rows);  // rows of the plane (row y: voxels below y)
    int32_t* out = sat + ((size_t)a * (Z + 1) + z) * Y1 * X1;
    const uint32_t* rows = row_n + (size_t)a * Y;
    for (int x = lane; x < X; x += 32) run[x] = add[x] = 0;
#pragma unroll
    for (int i = 0; i < kRegs; ++i) reg[i] = 0;
    __syncwarp();
    // add a listed voxel if it lies below z
    auto put = [&](uint32_t q) {
      const bool in = (int)(q >> 16) < z;
      if (in) atomicAdd(&add[q & 0xFFFFu], 1);
      return in;
    };
    constexpr uint32_t kNone = 0xFFFFFFFFu;  // z 65535: in no plane (Z < 65536 planes lie below)
    // running counts += inclusive sums of the new ones
    auto merge = [&]() {
      __syncwarp();
      int32_t carry = 0;
      auto step = [&](int x) {  // inclusive sum of the new counts up to x
        int32_t v = x < X ? add[x] : 0;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int32_t u = __shfl_up_sync(0xFFFFFFFFu, v, d);
          if (lane >= d) v += u;
        }
        if (x < X) add[x] = 0;
        v += carry;
        carry = __shfl_sync(0xFFFFFFFFu, v, 31);
        return v;
      };
      if constexpr (kRegs > 0) {
#pragma unroll
        for (int i = 0; i < kRegs; ++i)
          if (32 * i < X) reg[i] += step(32 * i + lane);
      } else {
        for (int x0 = 0; x0 < X; x0 += 32) {
          const int32_t v = step(x0 + lane);
          if (x0 + lane < X) run[x0 + lane] += v;
        }
      }
      __syncwarp();
    };
    // rows y0 - 1 .. y1 - 2 of voxels enter the planes' rows y0 .. y1 - 1; lane i holds the start of
    // voxel row y0 - 1 + i (their ends are the next starts)
    const int first = max(y0 - 1, 0);
    const uint32_t starts = __ldg(rows + min(first + lane, Y));
    const uint32_t before = __shfl_sync(0xFFFFFFFFu, starts, 0);
    bool any = false;
    if (z > 0)
      for (uint32_t i = __ldg(rows) + lane; i < before; i += 128) {  // four loads in flight
        uint32_t q[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) q[k] = i + 32 * k < before ? __ldg(list + i + 32 * k) : kNone;
#pragma unroll
        for (int k = 0; k < 4; ++k) any = put(q[k]) || any;
      }
    if (__any_sync(0xFFFFFFFFu, any)) merge();
    // a row's first 32 voxels are loaded while the row before is written
    auto head = [&](int j) {
      const uint32_t b = __shfl_sync(0xFFFFFFFFu, starts, j), e = __shfl_sync(0xFFFFFFFFu, starts, j + 1);
      return b + lane < e ? __ldg(list + b + lane) : kNone;
    };
    uint32_t next = head(0);
    for (int y = y0; y < y1; ++y) {
      const int j = y - 1 - first;  // the voxel row that enters here (-1: none, y = 0)
      if (z > 0 && j >= 0) {
        const uint32_t q = next;
        if (y + 1 < y1) next = head(j + 1);
        bool in = put(q);
        const uint32_t b = __shfl_sync(0xFFFFFFFFu, starts, j), e = __shfl_sync(0xFFFFFFFFu, starts, j + 1);
        for (uint32_t i = b + 32 + lane; i < e; i += 32) in = put(__ldg(list + i)) || in;
        if (__any_sync(0xFFFFFFFFu, in)) merge();
      }
      int32_t* o = out + (size_t)y * X1;
      if (lane == 0) o[0] = 0;
      if constexpr (kRegs > 0) {
#pragma unroll
        for (int i = 0; i < kRegs; ++i)
          if (32 * i + lane < X) o[32 * i + lane + 1] = reg[i];
      } else {
        for (int x = lane; x < X; x += 32) o[x + 1] = run[x];
      }
    }
    __syncwarp();
  }
}

// The same by passes over the whole array: for small arrays, for grids too wide for a warp's counts in
// shared memory (ref_sat_by_list) and for scans with too many voxels of one symbol (launch_ref_sat_list).
// Pass 0: running sums along x per (a, z, y) row (a warp per row: inclusive warp scans over
// 32-voxel chunks, coalesced) and the zero entries; pass 1 along y and pass 2 along z (a thread per
// column, rows read kChunk at a time so that the loads of a chunk are in flight together).
constexpr int kChunk = 8;

__global__ void ref_sat_x_kernel(const GridConst gc, const uint8_t* __restrict__ symA, int32_t* __restrict__ sat) {
  const int X = gc.X, Y = gc.Y, X1 = X + 1, Y1 = Y + 1, Z1 = gc.Z + 1;
  const int64_t rows = (int64_t)(gc.K - 1) * Z1 * Y1;
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t r = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += warps) {
    const int y = (int)(r % Y1) - 1;  // row y of layer z ends in the entries of y + 1 and z + 1
    const int z = (int)((r / Y1) % Z1) - 1;
    const int a = (int)(r / ((int64_t)Y1 * Z1)) + 1;
    int32_t* out = sat + (size_t)r * X1;
    if (y < 0 || z < 0) {
      for (int x = lane; x < X1; x += 32) out[x] = 0;
      continue;
    }
    const uint8_t* in = symA + ((size_t)z * Y + y) * X;
    if (lane == 0) out[0] = 0;
    int32_t carry = 0;
    for (int x0 = 0; x0 < X; x0 += 32) {
      const int x = x0 + lane;
      int32_t v = (x < X && in[x] == a) ? 1 : 0;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int32_t u = __shfl_up_sync(0xFFFFFFFFu, v, d);
        if (lane >= d) v += u;
      }
      if (x < X) out[x + 1] = carry + v;
      carry += __shfl_sync(0xFFFFFFFFu, v, 31);
    }
  }
}

// Running sums down a column of n entries `stride` apart (entry 0 stays as it is).
__device__ __forceinline__ void column_scan(int32_t* __restrict__ base, int n, size_t stride) {
  int32_t acc = 0;
  for (int i0 = 1; i0 < n; i0 += kChunk) {
    int32_t v[kChunk];
#pragma unroll
    for (int k = 0; k < kChunk; ++k) v[k] = (i0 + k < n) ? base[(size_t)(i0 + k) * stride] : 0;
#pragma unroll
    for (int k = 0; k < kChunk; ++k) {
      acc += v[k];
      if (i0 + k < n) base[(size_t)(i0 + k) * stride] = acc;
    }
  }
}

__global__ void ref_sat_y_kernel(const GridConst gc, int32_t* sat) {
  const int X1 = gc.X + 1, Y1 = gc.Y + 1, Z1 = gc.Z + 1;
  const int64_t cols = (int64_t)(gc.K - 1) * gc.Z * X1;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < cols; c += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(c % X1);
    const int z = (int)((c / X1) % gc.Z) + 1;
    const int a = (int)(c / ((int64_t)X1 * gc.Z));
    column_scan(sat + ((size_t)a * Z1 + z) * Y1 * X1 + x, Y1, (size_t)X1);
  }
}

__global__ void ref_sat_z_kernel(const GridConst gc, int32_t* sat) {
  const int X1 = gc.X + 1, Y1 = gc.Y + 1, Z1 = gc.Z + 1;
  const int64_t cols = (int64_t)(gc.K - 1) * Y1 * X1;
  const size_t plane = (size_t)Y1 * X1;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < cols; c += (int64_t)gridDim.x * blockDim.x) {
    const int64_t xy = c % ((int64_t)Y1 * X1);
    const int a = (int)(c / ((int64_t)Y1 * X1));
    column_scan(sat + (size_t)a * Z1 * plane + xy, Z1, plane);
  }
}

int blocks_for(int64_t work, int threads) {
  int64_t b = (work + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > 65535LL * 16) b = 65535LL * 16;
  return (int)b;
}

}  // namespace

cudaError_t launch_ref_accumulate(const GridConst& gc, const float* xyz, int64_t n, const float* pose12, uint32_t* cnt,
                                  unsigned long long* s1, unsigned long long* s2, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  ref_accumulate_kernel<<<blocks_for(n, 256), 256, 0, s>>>(gc, xyz, n, pose12, cnt, s1, s2);
  return cudaGetLastError();
}

cudaError_t launch_ref_symbols(const GridConst& gc, uint32_t* cnt, unsigned long long* s1, unsigned long long* s2,
                               uint8_t* symA, int32_t* box, uint32_t* row_n, cudaStream_t s) {
  const int64_t V = (int64_t)gc.X * gc.Y * gc.Z;
  // (a block copies the thresholds: several voxels per thread)
  ref_symbols_kernel<<<std::min(blocks_for(V, 256), 4096), 256, 0, s>>>(gc, cnt, s1, s2, symA, box, row_n);
  return cudaGetLastError();
}

// Small arrays stay with the passes: the list's strips are short chains of dependent loads (104k points
// on a 25 MB array, 150 x 160 x 16 voxels and 15 symbols, 109 against 117 us; 104k points on 108 MB, 250
// x 266 x 26, 206 against 143 us; on 92 MB, 56 symbols, 179 against 115 us).
bool ref_sat_by_list(const GridConst& gc) {
  const int64_t bytes = (int64_t)(gc.K - 1) * (gc.Z + 1) * (gc.Y + 1) * (gc.X + 1) * 4;
  return gc.X <= kSatMaxX && gc.Z < 65536 &&  // 64 KB of counts per block; 16-bit list entries
         bytes >= ((int64_t)32 << 20);
}

cudaError_t launch_ref_sat_list(const GridConst& gc, const uint8_t* symA, uint32_t* row_n, uint32_t* list,
                                int32_t* few, int32_t* sat, int n_sm, cudaStream_t s) {
  const int64_t V = (int64_t)gc.X * gc.Y * gc.Z;
  const int64_t n_sat = (int64_t)(gc.K - 1) * (gc.Z + 1) * (gc.Y + 1) * (gc.X + 1);
  // A strip adds up all of its symbol's voxels before it, 128 at a time: 4 ns per voxel of the symbol
  // with the most, while the passes take about 1 us per MB more than the list's writes.  1M points
  // spread evenly over 320 x 320 x 32 voxels, 15 symbols (196 MB): 3.2 ms by list, 0.48 by passes; 30k
  // points 0.29 and 0.37; a LiDAR scan of 106k 0.19 and 0.32.
  const int64_t most = n_sat * 4 / kSatMostBytes;
  ref_rows_kernel<<<1, 1024, 0, s>>>(row_n, (int64_t)(gc.K - 1) * gc.Y + 1, gc.Y,
                                   (uint32_t)std::min<int64_t>(most, UINT32_MAX), few);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  ref_list_kernel<<<blocks_for((V + 15) / 16, 256), 256, 0, s>>>(gc, symA, row_n, list, few);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const size_t smem = (size_t)kSatWarps * 2 * gc.X * 4;
  auto* k = gc.X <= 160 ? ref_sat_list_kernel<5> : gc.X <= 416 ? ref_sat_list_kernel<13> : ref_sat_list_kernel<0>;
  if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024)) != cudaSuccess) return e;
  // shorter strips while there are few: a strip's rows follow one another (latency), but each strip
  // adds up the rows before it first.  Strips of 31 rows throughout: 160 x 160 x 16 voxels 140 us, 320 x
  // 320 x 32 (15 symbols) 215, 1500 x 100 x 20 351; as here 126, 188, 214; 400 x 400 x 40 388 either way;
  // strips of 7 everywhere 122, 175, 214, 385, but 64 x 64 x 200 175 against 162.
  int rows = kSatRows;
  auto blocks_of = [&](int r) {
    return ((int64_t)(gc.K - 1) * (gc.Z + 1) * ((gc.Y + r) / r) + kSatWarps - 1) / kSatWarps;
  };
  while (rows > 7 && blocks_of(rows) < 16 * (int64_t)n_sm) rows /= 2;
  const int64_t blocks = blocks_of(rows);
  k<<<(unsigned)std::min<int64_t>(blocks, 64 * (int64_t)n_sm), kSatWarps * 32, smem, s>>>(gc, row_n, list, sat,
                                                                                           rows, few);
  return cudaGetLastError();
}

cudaError_t launch_ref_sat(const GridConst& gc, const uint8_t* symA, int32_t* sat, cudaStream_t s) {
  if (gc.K <= 1) return cudaSuccess;
  const int64_t rows = (int64_t)(gc.K - 1) * (gc.Z + 1) * (gc.Y + 1);
  ref_sat_x_kernel<<<blocks_for(rows * 32, 256), 256, 0, s>>>(gc, symA, sat);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int64_t cy = (int64_t)(gc.K - 1) * gc.Z * (gc.X + 1);
  ref_sat_y_kernel<<<blocks_for(cy, 128), 128, 0, s>>>(gc, sat);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int64_t cz = (int64_t)(gc.K - 1) * (gc.Y + 1) * (gc.X + 1);
  ref_sat_z_kernel<<<blocks_for(cz, 128), 128, 0, s>>>(gc, sat);
  return cudaGetLastError();
}

}  // namespace mialign
