// runtime_internal.h — host-side state shared by the library's C-ABI translation units
// (grids, device buffers, error reporting).  Not part of the public interface.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <atomic>
#include <cstdint>
#include <vector>

#include "align.h"
#include "align_internal.h"

namespace mialign {

// A growable device allocation (cudaMalloc; contents undefined after growth).
struct DevBuf {
  void* p = nullptr;
  size_t cap = 0;
  cudaError_t ensure(size_t bytes) {
    if (bytes <= cap && p != nullptr) return cudaSuccess;
    if (p) cudaFree(p);
    p = nullptr;
    cap = 0;
    size_t want = std::max<size_t>(bytes, 256);
    cudaError_t e = cudaMalloc(&p, want);
    if (e == cudaSuccess) cap = want;
    return e;
  }
  void release() {
    if (p) cudaFree(p);
    p = nullptr;
    cap = 0;
  }
  template <class T>
  T* as() const {
    return static_cast<T*>(p);
  }
};

// Device memory that a faster path takes where it can and does without where it cannot (voxel sums of
// scattered poses, lattice workspaces).  All objects of the process together hold at most `limit` of
// it (kOptionalShare of the device's memory; 0: not counted, a server's budget covers it), so that what
// other objects need is never taken by it; give_back returns an object's own when memory runs out.
constexpr size_t kOptionalShare = 8;
struct OptionalBuf : DevBuf {
  bool counted = false;
  bool ensure(size_t bytes, size_t limit) {
    if (bytes <= cap && p != nullptr) return true;
    const size_t want = std::max<size_t>(bytes, 256), had = counted ? cap : 0;
    if (limit != 0) {
      size_t h = held().load();
      do {
        if (h - had + want > limit) return false;
      } while (!held().compare_exchange_weak(h, h - had + want));
    } else if (counted) {
      held() -= had;
    }
    counted = limit != 0;
    if (DevBuf::ensure(want) == cudaSuccess) return true;
    (void)cudaGetLastError();
    if (counted) held() -= want;
    counted = false;
    return false;
  }
  void release() {
    if (counted) held() -= cap;
    counted = false;
    DevBuf::release();
  }

 private:
  static std::atomic<size_t>& held() {
    static std::atomic<size_t> bytes{0};
    return bytes;
  }
};

// A growable page-locked host allocation (asynchronous copies from and to it).
struct HostBuf {
  void* p = nullptr;
  size_t cap = 0;
  cudaError_t ensure(size_t bytes) {
    if (bytes <= cap && p != nullptr) return cudaSuccess;
    if (p) cudaFreeHost(p);
    p = nullptr;
    cap = 0;
    size_t want = std::max<size_t>(bytes, 256);
    cudaError_t e = cudaMallocHost(&p, want);
    if (e == cudaSuccess) cap = want;
    return e;
  }
  void release() {
    if (p) cudaFreeHost(p);
    p = nullptr;
    cap = 0;
  }
  template <class T>
  T* as() const {
    return static_cast<T*>(p);
  }
};

// Error reporting into the thread-local message of align_last_error.
align_status report_errorf(align_status st, const char* fmt, ...);
// The structure of a host pose batch: its distinct rotations (bitwise), each pose's rotation, and
// whether it is a lattice: every combination of the n_rot rotations and mx, my, mz values of
// t'_x, t'_y, t'_z (bitwise distinct), each once; then pose_of[((r mz + iz) my + iy) mx + ix].
struct PoseSet {
  int32_t n_rot = -1;  // -1: more than a quarter of the poses
  std::vector<float> rots;
  std::vector<int32_t> src;
  bool lattice = false;
  int32_t mx = 0, my = 0, mz = 0;
  double t_max = 0.0;  // largest |t'_x| of a lattice
  std::vector<int32_t> pose_of;
};
PoseSet pose_set(const float* poses12, int64_t P);
// Whether the first pose's rotation occurs as often as a lattice's would: false for poses that
// pose_set would find to be none, at a fraction of its time where no two rotations are alike.
bool may_be_lattice(const float* poses12, int64_t P);
align_status check_grid_device(align_grid* g);
// Pose pairs for the pair kernel: poses with the same rotation (tile copy) and bitwise equal
// t'_y, t'_z, two per unit (local indices; the second -1 for a single pose).  Returns the units.
int pair_units(const float* poses12, const PoseSet& set, int64_t P, std::vector<int32_t>& units);
constexpr size_t kScatterBudget = (size_t)1 << 30;  // sums and lists of poses spread over the GPU
// Beyond about this many poses a CTA per pose is faster (an L2 atomic per run, not a shared one): for
// 120k points in scan order they cross at 36 poses (0.25 m LiDAR grid), 42 (0.5 m), 56 (1 m), 22 on the
// 6.4M-voxel grid, where the budget holds 10 (as it holds 20 on the 0.25 m grid: 3.3M voxels).  Points in
// no order cross earlier: at 32 poses 148 against 219 us (0.5 m), 190 against 214 (1 m); on fewer voxels
// see enqueue_scatter.
constexpr int64_t kScatterMaxPoses = 32;
bool plan_lattice(const GridConst& gc, int n_sm, size_t smem_optin, int64_t n, int64_t n_rot, int32_t mx, int32_t my,
                  int32_t mz, double t_max, int min_groups, LatticeArgs& a);
// The same for the levels of a lattice search over n points (align_search_ex).
bool plan_search(const align_grid* g, int64_t n, const int32_t m[6], const double c[6], const double r[6],
                 LatticeArgs& a);
size_t lattice_carve(LatticeArgs& a, uint8_t* base);
// Whether pose pairs are the automatic choice for a grid with these learned key-partition
// counts (pairs, single poses).
bool pairs_fit(const align_grid* g, int32_t seed_pair, int32_t seed_single);
// One level of the coarse-to-fine lattice: FP64 poses around centre c (ranges r, m samples
// per axis; order rx, ry, rz, tx, ty, tz with tz fastest) and their rounded FP32 form.
void lattice_poses(const float origin[3], const double c[6], const double r[6], const int32_t m[6],
                   std::vector<double>& eta, std::vector<float>& poses);

// What a call reads back besides its MI: the kernels' error word and counters, the argmax and its
// packed key, in one device block, followed by the MI of calls with up to kHeadPoses poses, so that a
// call is one copy into page-locked memory and one synchronisation (six copies, each waited for,
// before: 113 -> 65 us for one pose of 120k points, 5.2 -> 3.0 ms for a Nelder-Mead of 75 phases).
struct GridHead {
  uint32_t err, max_passes, wide_count, wide_poses;
  int64_t argmax;
  unsigned long long best;
  uint32_t done, pad;  // compose_kernel's CTAs that have finished: 0 between launches
};
constexpr size_t kHeadBytes = (size_t)1 << 16;
constexpr int64_t kHeadPoses = (int64_t)((kHeadBytes - sizeof(GridHead)) / 4);
constexpr size_t kHistStage = (size_t)1 << 20;  // histograms up to this size are staged likewise

}  // namespace mialign

// A grid: its voxel map, the resident reference state of scan A, and the workspace of its
// own evaluations.
struct align_grid {
  mialign::GridConst gc{};
  float origin[3];
  float res_m;
  int64_t V = 0;
  cudaStream_t stream = nullptr;
  int device = 0;
  int n_sm = 0;
  int table_slots = 0;  // of the last launch (it depends on the table layout)
  size_t smem_optin = 0;
  bool has_ref = false;
  int32_t boxA[6];
  mialign::DevBuf symA, sat;
  // evaluation workspace
  mialign::DevBuf head;  // GridHead, then MI (GridHead's comment)
  mialign::HostBuf head_h, hist_h;
  mialign::GridHead* dev_head() const { return head.as<mialign::GridHead>(); }
  mialign::DevBuf xyz, poses, out_c, out_box, mi, hist, wide, dump;
  mialign::DevBuf pts4, pose_src, rots, redo_list, redo_count, ovf;
  // device-built lattice levels (align_search_ex): centres, rotation tables, read-backs
  mialign::DevBuf lat_c, lat_cand;
  // reference-build working buffers (align_set_reference)
  mialign::DevBuf ref_pts, ref_pose, ref_cnt, ref_s1, ref_s2, ref_box, ref_rows, ref_list;
  bool ref_clean = false;  // ref_cnt, ref_s1, ref_s2 hold zeros (the symbols kernel clears what it read)
  mialign::HostBuf ref_box_h;
  bool ref_pose_set = false;
  mialign::HostBuf lat_cand_h, lat_rec_h, lat_c_h;
  std::vector<cudaEvent_t> lat_ev;
  bool lat_pending = false;  // a search's copies may still be reading the pinned buffers
  int64_t n_points = 0;  // points staged in `xyz`
  // key partitions the next launch starts with, per kernel shape (its table size), and for
  // the pose-pair kernel (shape 0)
  int32_t passes_seed[mialign::kEvalShapes] = {1, 1, 1};
  int32_t passes_seed_pair[mialign::kEvalShapes] = {1, 1, 1};
  int32_t passes_seed_cluster = 1;  // the 2-CTA cluster kernel (shape 0)
  int32_t sweep_mode = -1;  // -1 automatic, else the sweep kind every launch takes (align_set_sweep)
  bool last_pairs = false;    // the last eval launch evaluated pose pairs
  bool last_lattice = false;  // ... or a pose lattice by groups
  int32_t lattice_on = 1;     // 0: pose lattices go through the table kernels (a server's workspace
                              // whose request was admitted without the groups' memory)
  int32_t scatter_on = 1;     // 0: poses that share nothing go through the table kernels (a server's
                              // workspace: its requests' estimates hold no dense sums)
  size_t optional_limit = 0;  // OptionalBuf::ensure
  bool optional_on = true;    // false while a call that ran out of memory is run again without them
  mialign::OptionalBuf lattice_ws;            // groups' workspace
  mialign::DevBuf lattice_order;              // a device-built level's pose order
  int32_t lattice_order_m[6] = {0, 0, 0, 0, 0, 0};
  // poses that share nothing; all but the list as the kernels leave it between calls (zero, no box)
  mialign::OptionalBuf scatter_sums, scatter_list;
  mialign::DevBuf scatter_n, scatter_c, scatter_box;
  bool last_cluster = false;  // ... or ran one pose per 2-CTA cluster
  mialign::DevBuf units;    // pose pairs of the last pair launch with host poses
  mialign::DevBuf spill;    // runs queued for the later key partitions (EvalArgs::spill)
  int32_t spill_on = 1;     // align_set_spill
  int32_t layout_min = 1;   // smallest table layout (value words) of this grid's z-sum launches:
                            // 3 once packed-layout poses went to the exact path for a wide voxel
  int32_t last_vw = 0;      // the layout of the last eval launch
  int64_t spill_runs = 0;   // runs per queue and CTA (0: half the padded points of B)
  int32_t spill_np_max = 8; // most key partitions the spill queues serve (a server's workspace: its request's)
  mialign::DevBuf lat_units;           // pose pairs of a device-built lattice level (by index)
  std::vector<int32_t> lattice_units;  // ... on the host
  int32_t lattice_units_m[6] = {0, 0, 0, 0, 0, 0};
  int64_t stats[6] = {0, 0, 0, 0, 0, 0};
  // event timing (align_profile): one (before eval, after eval, after argmax) triple per
  // launch, drained into the totals at the next synchronising call or profile read
  bool profiling = false;
  std::vector<std::array<cudaEvent_t, 3>> ev_pending, ev_pool;
  double prof[3] = {0.0, 0.0, 0.0};
};
