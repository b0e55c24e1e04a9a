// batch.cu — many scan pairs in one persistent launch (align_eval_batch).
//
// Every pair keeps its own grid (resident reference state of scan A) and pose batch; the
// launch evaluates all pairs' poses as one list, each pose carrying its pair's grid
// constants (EvalItem).  The launch sequence (clear, pack, eval + redo, compose, argmax)
// can be captured as a CUDA graph and replayed while the batch keeps its shape; inputs are
// copied into the batch's own buffers before each launch, so the graph's pointers stay
// valid.  Pairs whose poses are a lattice are evaluated by groups (lattice_eval.cu), one after
// another from one workspace; the others by the table kernels, whose shape is fixed, the default,
// or picked by timing the candidates on the batch itself (tuner below).
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "align.h"
#include "align_internal.h"
#include "runtime_internal.h"

using namespace mialign;

namespace {

#define BCU(call, what)                                                    \
  do {                                                                     \
    cudaError_t e_ = (call);                                               \
    if (e_ != cudaSuccess) return report_cuda_error(e_, (what));           \
  } while (0)

constexpr size_t kPrerotBudget = (size_t)8 << 30;  // bytes of pre-rotated tiles per batch

// Per-pair plan of one batch launch.
struct PairPlan {
  align_grid* g = nullptr;
  int64_t nB = 0, P = 0;
  int32_t n_tiles = 0;
  int64_t n_pad = 0;
  int n_copies = 1;           // tile copies to pack: rotations (pre-rotated), 1 (raw) or 0 (groups)
  bool prerot = false;
  std::vector<float> hposes;  // host fp32 poses (when given on the host)
  PoseSet set;                // their structure (rotations, lattice)
  bool by_groups = false;     // a lattice evaluated by groups (tiles and tables for the exact path only)
  LatticeArgs lat{};
  int64_t order_off = 0;      // its poses' order (in order)
  std::vector<int32_t> units; // pose pairs (pair kernel), two local pose indices per unit
  int32_t n_units = 0;        // 0: one pose per CTA step (eval_kernel)
  int64_t unit_off = 0;       // units before this pair's (in units)
  int64_t xyz_off = 0;        // floats
  int64_t pose_off = 0;       // poses (global pose index of pose 0)
  int64_t pts_off = 0;        // float4
  int64_t outc_off = 0;       // uint32
  int32_t passes0 = 1;        // the grid's key-partition seed for this launch's kind
  int32_t spill_np = 0;       // 2-8 key partitions: EvalArgs::spill_np (0: no queues)
  int64_t spill_cap = 0;      // ... and the runs per queue
};

// Workspace sizes of one launch; a change of any of them re-allocates and drops the graph.
struct Sizes {
  size_t xyz = 0, poses = 0, pts = 0, pose_src = 0, copies = 0, items = 0, starts = 0, outc = 0, box = 0,
         best = 0, mi = 0, argmax = 0, redo = 0, wide = 0, ipasses = 0, ovf = 0, units = 0, spill = 0, order = 0;
};

std::string env_cache_path() {
  const char* p = std::getenv("ALIGN_TUNE_CACHE");
  return p ? std::string(p) : std::string();
}

// Tuner cache: batch class -> choice (kernel shape * 2 + poses per CTA - 1).  Shared by all
// batches of the process.
constexpr int kChoices = 2 * kEvalShapes;
std::mutex g_tune_mu;
std::map<std::string, int> g_tune;
bool g_tune_loaded = false;

void tune_load_locked() {
  if (g_tune_loaded) return;
  g_tune_loaded = true;
  const std::string path = env_cache_path();
  if (path.empty()) return;
  FILE* f = std::fopen(path.c_str(), "r");
  if (!f) return;
  char key[512];
  int shape = 0;
  while (std::fscanf(f, "%511s %d", key, &shape) == 2)
    if (shape >= 0 && shape < kChoices) g_tune[key] = shape;
  std::fclose(f);
}

void tune_store_locked(const std::string& key, int shape) {
  g_tune[key] = shape;
  const std::string path = env_cache_path();
  if (path.empty()) return;
  FILE* f = std::fopen(path.c_str(), "a");
  if (!f) return;
  std::fprintf(f, "%s %d\n", key.c_str(), shape);
  std::fclose(f);
}

// floor(log2(v)) for v >= 1 (0 otherwise): the size classes of the tuner's cache key.
int bucket_log2(int64_t v) {
  int b = 0;
  while (v > 1) {
    v >>= 1;
    ++b;
  }
  return b;
}

}  // namespace

struct align_batch {
  cudaStream_t user_stream = nullptr;  // the caller's stream (ordering of device inputs)
  cudaStream_t stream = nullptr;       // the batch's own stream (capturable; the legacy
                                       // default stream cannot be captured)
  cudaEvent_t ev_in = nullptr;
  int device = 0;
  int n_sm = 0;
  size_t smem_optin = 0;
  std::string device_name;
  int shape_fixed = -1;
  DevBuf xyz, poses, pts, pose_src, copies, items, starts, outc, box, best, mi, argmax, redo_list, redo_count, wide,
      status, ipasses, ovf, units, spill, order;
  OptionalBuf lattice;
  size_t optional_limit = 0;  // OptionalBuf::ensure
  bool optional_on = true;    // false while a call that ran out of memory is run again without it
  // page-locked staging of the poses and their tile copies (asynchronous copies; a call's
  // copies are done when it returns, since every call synchronises its stream)
  mialign::HostBuf h_poses, h_src;
  bool staged = false;  // copies out of the staging buffers may still be queued
  std::vector<align_grid*> last_grids;  // grids of the last launch (per-item partition feedback)
  std::vector<char> last_pairs;         // whether each item of the last launch used pose pairs
  std::vector<int> last_vws;            // each item's table layout in the last launch
  int last_shape = 0;
  int pairs_fixed = -1;                 // poses per CTA set by the caller (1, 2), -1: default
  Sizes cap;
  // graph of the last launch sequence
  cudaGraphExec_t exec = nullptr;
  int32_t graph_launches = 0;           // kernels of its pairs
  std::vector<int64_t> sig;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  int64_t stats[9] = {0, 0, 0, 0, 0, 0, 0, 0, 1};
};

namespace {

void drop_graph(align_batch* b) {
  if (b->exec) cudaGraphExecDestroy(b->exec);
  b->exec = nullptr;
  b->sig.clear();
}

// Grow a buffer; any growth invalidates the captured graph.
align_status grow(align_batch* b, DevBuf& buf, size_t& cap, size_t bytes, const char* what, bool zero = false) {
  if (bytes <= cap && buf.p) return ALIGN_OK;
  drop_graph(b);
  const size_t want = std::max<size_t>(bytes, 256);
  BCU(buf.ensure(want), what);
  cap = want;
  if (zero) BCU(cudaMemsetAsync(buf.p, 0, want, b->stream), what);
  return ALIGN_OK;
}

struct Launch {
  const EvalKernels* ek = nullptr;
  int shape = 0;
  EvalArgs a{};  // all pairs (compose, argmax)
  // one single-pair eval + redo launch per pair: its arguments (the pair in the parameter
  // bank, its poses p_begin..P-1 of the batch) and its table layout
  std::vector<EvalArgs> evals;
  std::vector<LatticeArgs> lats;   // its lattice by groups instead,
  std::vector<int32_t> lat_rots;   // ... of this many rotations (0: by the table kernels)
  std::vector<int> vws;
  int n_ctas = 0;
  bool rotate = false;
  int n_items = 0;
  int n_copies = 0;
  int64_t max_out = 0;
};

// The launch sequence that a graph captures: clear, pack, eval + redo, compose, argmax.
// Adds the pairs' kernels to *launches.
align_status enqueue_launch(align_batch* b, const Launch& L, int32_t* launches) {
  cudaStream_t s = b->stream;
  BCU(cudaMemsetAsync(b->best.p, 0, (size_t)L.n_items * 8, s), "clear argmax keys");
  BCU(cudaMemsetAsync(b->ipasses.p, 0, (size_t)L.n_items * 4, s), "clear partition counts");
  BCU(cudaMemsetAsync(b->redo_count.p, 0, 4, s), "clear redo count");
  BCU(L.ek->launch_pack_batch(b->copies.as<PackCopy>(), L.n_copies, L.max_out, s), "launch pack");
  for (size_t k = 0; k < L.evals.size(); ++k) {
    // each pair's redo kernel finishes only that pair's poses
    if (k > 0) BCU(cudaMemsetAsync(b->redo_count.p, 0, 4, s), "clear redo count");
    if (L.lat_rots[k] > 0) {
      BCU(launch_lattice(L.lats[k], L.lat_rots[k], b->n_sm, s, launches), "launch lattice evaluation");
      BCU(L.ek->launch_redo(L.evals[k], b->n_sm, L.vws[k], s), "launch redo kernel");
      *launches += 1;
    } else {
      BCU(L.ek->launch_eval(L.evals[k], L.n_ctas, L.vws[k], L.rotate, s), "launch eval kernel");
      *launches += 2;
    }
  }
  BCU(L.ek->launch_compose(L.a, s), "launch compose kernel");
  BCU(L.ek->launch_argmax_finalize(L.a.items, L.n_items, s), "launch argmax");
  return ALIGN_OK;
}

align_status run_launch(align_batch* b, const Launch& L, bool use_graph, const std::vector<int64_t>& sig) {
  BCU(cudaEventRecord(b->ev0, b->stream), "record event");
  int32_t launches = 0;
  if (use_graph) {
    if (!b->exec || b->sig != sig) {
      drop_graph(b);
      cudaGraph_t graph = nullptr;
      BCU(cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal), "begin capture");
      b->graph_launches = 0;
      align_status st = enqueue_launch(b, L, &b->graph_launches);
      cudaError_t e = cudaStreamEndCapture(b->stream, &graph);
      if (st != ALIGN_OK) {
        if (graph) cudaGraphDestroy(graph);
        return st;
      }
      BCU(e, "end capture");
      e = cudaGraphInstantiate(&b->exec, graph, 0);
      cudaGraphDestroy(graph);
      BCU(e, "instantiate graph");
      b->sig = sig;
      b->stats[1] += 1;
    } else {
      b->stats[2] += 1;
    }
    BCU(cudaGraphLaunch(b->exec, b->stream), "launch graph");
    launches = b->graph_launches;
  } else {
    align_status st = enqueue_launch(b, L, &launches);
    if (st != ALIGN_OK) return st;
  }
  BCU(cudaEventRecord(b->ev1, b->stream), "record event");
  b->stats[0] += 1;
  b->stats[5] += 3 + launches;  // pack, the pairs' kernels, compose, argmax
  return ALIGN_OK;
}

// Read the kernels' status words (synchronises the stream).
align_status collect(align_batch* b) {
  uint32_t v[4] = {0, 0, 0, 0};
  std::vector<uint32_t> ip(b->last_grids.size(), 0);
  BCU(cudaMemcpyAsync(v, b->status.p, 16, cudaMemcpyDeviceToHost, b->stream), "read status");
  if (!ip.empty())
    BCU(cudaMemcpyAsync(ip.data(), b->ipasses.p, ip.size() * 4, cudaMemcpyDeviceToHost, b->stream),
        "read partition counts");
  BCU(cudaStreamSynchronize(b->stream), "synchronize");
  b->staged = false;
  // seed each grid's next launches with the partitions its poses needed (a power of two);
  // batches on other threads may share the grid (a server's workers): atomic max
  for (size_t i = 0; i < ip.size(); ++i) {
    align_grid* g = b->last_grids[i];
    int32_t* seed = b->last_pairs[i] ? &g->passes_seed_pair[b->last_shape] : &g->passes_seed[b->last_shape];
    if (ip[i] > (1u << 16) || (ip[i] & (ip[i] - 1)) != 0) continue;
    int32_t cur = __atomic_load_n(seed, __ATOMIC_RELAXED);
    while ((int32_t)ip[i] > cur &&
           !__atomic_compare_exchange_n(seed, &cur, (int32_t)ip[i], false, __ATOMIC_RELAXED, __ATOMIC_RELAXED)) {
    }
  }
  // packed-layout poses sent to the exact path by a wide voxel: the grids of the launch that
  // used the packed layout take the three-word layout from now on (one counter for the launch)
  if (v[3] > 0)
    for (size_t i = 0; i < b->last_grids.size() && i < b->last_vws.size(); ++i)
      if (b->last_vws[i] == 2) __atomic_store_n(&b->last_grids[i]->layout_min, 3, __ATOMIC_RELAXED);
  float ms = 0.0f;
  if (cudaEventElapsedTime(&ms, b->ev0, b->ev1) == cudaSuccess) b->stats[6] = (int64_t)std::llround(ms * 1000.0);
  // reset the error word, the partition maximum and the wide counters (per launch)
  BCU(cudaMemsetAsync(b->status.p, 0, 16, b->stream), "reset status");
  if (v[0] & kErrDzBound) return report_error(ALIGN_E_INTERNAL, "a z offset exceeded its proven bound");
  if (v[0] & kErrPassLimit) return report_error(ALIGN_E_INTERNAL, "key partitioning limit reached");
  return ALIGN_OK;
}

}  // namespace

extern "C" {

align_status align_batch_create(void* cuda_stream, align_batch** out) {
  if (!out) return report_error(ALIGN_E_INVALID, "out is NULL");
  *out = nullptr;
  int n_dev = 0;
  cudaError_t e = cudaGetDeviceCount(&n_dev);
  if (e != cudaSuccess || n_dev < 1) {
    (void)cudaGetLastError();
    return report_error(ALIGN_E_CUDA, "no usable CUDA device");
  }
  int dev = 0;
  BCU(cudaGetDevice(&dev), "cudaGetDevice");
  cudaDeviceProp prop;
  BCU(cudaGetDeviceProperties(&prop, dev), "cudaGetDeviceProperties");
  if (prop.major < 10) return report_errorf(ALIGN_E_CUDA, "this library is built for sm_103a (found sm_%d%d)",
                                            prop.major, prop.minor);
  for (int i = 0; i < kEvalShapes; ++i) BCU(eval_shape(i).setup(), "set up eval kernels");
  align_batch* b = new (std::nothrow) align_batch();
  if (!b) return report_error(ALIGN_E_OOM, "host allocation failed");
  b->user_stream = (cudaStream_t)cuda_stream;
  b->device = dev;
  b->n_sm = prop.multiProcessorCount;
  b->smem_optin = prop.sharedMemPerBlockOptin;
  b->optional_limit = prop.totalGlobalMem / kOptionalShare;
  b->device_name = prop.name;
  for (char& c : b->device_name)
    if (c == ' ') c = '_';
  if (cudaEventCreate(&b->ev0) != cudaSuccess || cudaEventCreate(&b->ev1) != cudaSuccess ||
      cudaEventCreateWithFlags(&b->ev_in, cudaEventDisableTiming) != cudaSuccess ||
      cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess) {
    (void)cudaGetLastError();
    if (b->ev0) cudaEventDestroy(b->ev0);
    if (b->ev1) cudaEventDestroy(b->ev1);
    if (b->ev_in) cudaEventDestroy(b->ev_in);
    delete b;
    return report_error(ALIGN_E_CUDA, "creating the batch's events and stream failed");
  }
  *out = b;
  return ALIGN_OK;
}

align_status align_batch_destroy(align_batch* b) {
  if (!b) return ALIGN_OK;
  cudaSetDevice(b->device);
  cudaStreamSynchronize(b->stream);
  drop_graph(b);
  for (DevBuf* d : {&b->xyz, &b->poses, &b->pts, &b->pose_src, &b->copies, &b->items, &b->starts, &b->outc, &b->box,
                    &b->best, &b->mi, &b->argmax, &b->redo_list, &b->redo_count, &b->wide, &b->status, &b->ipasses, &b->ovf,
                    &b->units, &b->spill, &b->order})
    d->release();
  b->lattice.release();
  b->h_poses.release();
  b->h_src.release();
  if (b->ev0) cudaEventDestroy(b->ev0);
  if (b->ev1) cudaEventDestroy(b->ev1);
  if (b->ev_in) cudaEventDestroy(b->ev_in);
  if (b->stream) cudaStreamDestroy(b->stream);
  delete b;
  return ALIGN_OK;
}

align_status align_batch_set_shape(align_batch* b, int32_t shape) {
  if (!b) return report_error(ALIGN_E_INVALID, "batch is NULL");
  if (shape < -1 || shape >= kEvalShapes) return report_error(ALIGN_E_INVALID, "shape out of range");
  b->shape_fixed = shape;
  return ALIGN_OK;
}

align_status align_batch_set_poses_per_cta(align_batch* b, int32_t poses_per_cta) {
  if (!b) return report_error(ALIGN_E_INVALID, "batch is NULL");
  if (poses_per_cta != -1 && poses_per_cta != 1 && poses_per_cta != 2)
    return report_error(ALIGN_E_INVALID, "poses_per_cta must be 1, 2 or -1");
  b->pairs_fixed = poses_per_cta;
  return ALIGN_OK;
}

align_status align_batch_stats(const align_batch* b, int64_t out[9]) {
  if (!b || !out) return report_error(ALIGN_E_INVALID, "NULL argument");
  for (int i = 0; i < 9; ++i) out[i] = b->stats[i];
  return ALIGN_OK;
}

}  // extern "C"

namespace {

// Plan, stage and launch one batch with kernel shape `shape`; outputs stay in the batch's
// buffers (copied out by the caller).
align_status eval_batch_shape(align_batch* b, std::vector<PairPlan>& plans, const align_pair* pairs,
                              const std::vector<int32_t>& which, int flags, int shape, bool pose_pairs) {
  const EvalKernels& ek = eval_shape(shape);
  const int n = (int)plans.size();
  const bool xyz_dev = (flags & ALIGN_XYZ_DEVICE) != 0;
  bool rotate = false, var = false;
  int maxK = 2;
  for (const PairPlan& pp : plans) {
    if (pp.hposes.empty()) rotate = true;  // device poses: every pair rotates in the kernel
    if (pp.g->gc.feature != ALIGN_FEAT_COUNT) var = true;
    maxK = std::max(maxK, (int)pp.g->gc.K);
  }
  // ---- layout ----
  const int tile = ek.tile_points();
  int64_t xyz_f = 0, poses_n = 0, pts_n = 0, outc_n = 0, max_out = 0;
  int n_copies = 0;
  // One pre-rotated copy per distinct rotation when every pair's rotations repeat (lattices)
  // and the copies fit the budget; otherwise every pair's tiles are raw and the kernel
  // rotates (one launch has one tile kind).
  size_t prerot_bytes = 0;
  for (PairPlan& pp : plans) {
    pp.n_tiles = (int32_t)std::max<int64_t>(ek.min_tiles(), (pp.nB + tile - 1) / tile);
    pp.n_pad = (int64_t)pp.n_tiles * tile;
    if (rotate || pp.by_groups) continue;
    const int groups = pp.set.n_rot;
    prerot_bytes += (size_t)std::max(groups, 1) * (size_t)pp.n_pad * 16;
    if (groups <= 0 || prerot_bytes > kPrerotBudget) rotate = true;
  }
  int64_t units_n = 0, order_n = 0;
  int64_t spill_words = 0;  // largest (queues x runs per queue) of a pair with spill queues
  for (PairPlan& pp : plans) {
    pp.prerot = !rotate && !pp.by_groups;
    pp.n_copies = pp.by_groups ? 0 : rotate ? 1 : pp.set.n_rot;
    // pose pairs: a pair's poses with the same rotation, t_y and t_z (pre-rotated tiles only);
    // a pair whose poses form no pair keeps the single-pose kernel
    pp.n_units = 0;
    pp.units.clear();
    // (and only while the grid's pairs have needed no more key partitions than its single
    // poses: a pair table holds two poses' voxels)
    // (a grid's align_set_sweep choice of single poses or pairs holds here too)
    const bool fits = pp.g->sweep_mode >= 0
                          ? pp.g->sweep_mode == 1
                          : pairs_fit(pp.g, __atomic_load_n(&pp.g->passes_seed_pair[shape], __ATOMIC_RELAXED),
                                      __atomic_load_n(&pp.g->passes_seed[shape], __ATOMIC_RELAXED));
    if (pose_pairs && fits && pp.prerot && pp.P >= 2) {
      const int nu = pair_units(pp.hposes.data(), pp.set, pp.P, pp.units);
      if (nu < pp.P) pp.n_units = nu;
      else pp.units.clear();
    }
    // the seed of the kind this pair runs; poses (or pose pairs) with key partitions sweep B
    // once and queue its runs by partition (as the single-pair path does)
    pp.passes0 = __atomic_load_n(pp.n_units > 0 ? &pp.g->passes_seed_pair[shape] : &pp.g->passes_seed[shape],
                                 __ATOMIC_RELAXED);
    pp.spill_np = 0;
    pp.spill_cap = 0;
    if (pp.g->spill_on && !pp.by_groups && pp.passes0 >= 2 && pp.passes0 <= 8) {
      pp.spill_np = std::min(8, 2 * pp.passes0);
      const int64_t runs = pp.g->spill_runs > 0 ? pp.g->spill_runs : pp.n_units > 0 ? pp.n_pad : pp.n_pad / 2;
      pp.spill_cap = (runs + 31) / 32 * 32;
      spill_words = std::max(spill_words, (int64_t)pp.spill_np * pp.spill_cap);
    }
    pp.unit_off = units_n;
    units_n += pp.n_units;
    pp.xyz_off = xyz_f;
    pp.pose_off = poses_n;
    pp.pts_off = pts_n;
    pp.outc_off = outc_n;
    pp.order_off = order_n;
    if (pp.by_groups) order_n += pp.P;
    xyz_f += pp.nB * 3;
    poses_n += pp.P;
    pts_n += std::max(1, pp.n_copies) * pp.n_pad;  // groups write raw tiles for the exact path
    outc_n += (pp.P * (int64_t)pp.g->gc.K * pp.g->gc.K + 3) / 4 * 4;  // cleared four words at a time
    n_copies += pp.n_copies;
    max_out = std::max(max_out, pp.n_pad);
  }
  if (poses_n >= INT32_MAX) return report_error(ALIGN_E_INVALID, "too many poses in one batch");
  if (n_copies > 65535) return report_error(ALIGN_E_INVALID, "too many tile copies in one batch");
  // per pair: its table layout and table size (one eval launch per pair)
  std::vector<int> vws, Ts;
  int T = 0;  // the largest table of the launches (sizes the 64-bit side sums)
  for (const PairPlan& pp : plans) {
    if (pp.by_groups) {  // the redo kernel's tables
      vws.push_back(pp.g->gc.feature != ALIGN_FEAT_COUNT ? 2 : 1);
      Ts.push_back(ek.table_slots_for(pp.g->gc.K, vws.back(), b->smem_optin, 1));
      T = std::max(T, Ts.back());
      continue;
    }
    int vw = eval_layout(pp.g->gc, var);  // at least the layout the grid has learned to need
    if (var) vw = std::max(vw, (int)__atomic_load_n(&pp.g->layout_min, __ATOMIC_RELAXED));
    vws.push_back(vw);
    Ts.push_back(ek.table_slots_for(pp.g->gc.K, vws.back(), b->smem_optin, pp.n_units > 0 ? 2 : 1));
    T = std::max(T, Ts.back());
  }
  const int n_ctas = b->n_sm * ek.ctas_per_sm;
  // ---- workspace ----
  align_status st;
#define GROW(buf, field, bytes, what, zero) \
  if ((st = grow(b, b->buf, b->cap.field, (bytes), (what), (zero))) != ALIGN_OK) return st;
  GROW(xyz, xyz, (size_t)xyz_f * 4, "allocate points", false);
  GROW(poses, poses, (size_t)poses_n * 48, "allocate poses", false);
  GROW(pts, pts, (size_t)pts_n * 16, "allocate tiles", false);
  GROW(pose_src, pose_src, (size_t)poses_n * 4, "allocate pose sources", false);
  GROW(copies, copies, (size_t)n_copies * sizeof(PackCopy), "allocate copy table", false);
  GROW(items, items, (size_t)n * sizeof(EvalItem), "allocate item table", false);
  GROW(starts, starts, (size_t)(n + 1) * 4, "allocate item starts", false);
  GROW(outc, outc, (size_t)outc_n * 4, "allocate histograms", false);
  GROW(box, box, (size_t)poses_n * 24, "allocate boxes", false);
  GROW(best, best, (size_t)n * 8, "allocate argmax keys", false);
  GROW(mi, mi, (size_t)poses_n * 4, "allocate MI", false);
  GROW(argmax, argmax, (size_t)n * 8, "allocate argmax", false);
  GROW(redo_list, redo, (size_t)poses_n * 4, "allocate redo list", false);
  GROW(ipasses, ipasses, (size_t)n * 4, "allocate partition counts", false);
  GROW(wide, wide, (size_t)n_ctas * 2 * T * 8, "allocate wide sums", true);
  GROW(ovf, ovf, (size_t)n_ctas * ek.ovf_cap() * 16, "allocate overflow lists", false);
  GROW(units, units, (size_t)std::max<int64_t>(1, units_n) * 8, "allocate pose pairs", false);
  GROW(spill, spill, (size_t)n_ctas * (size_t)std::max<int64_t>(1, spill_words) * 16, "allocate spill queues", false);
  GROW(order, order, (size_t)std::max<int64_t>(1, order_n) * 4, "allocate lattice order", false);
#undef GROW
  if (!b->status.p || !b->redo_count.p) {
    drop_graph(b);
    BCU(b->status.ensure(16), "allocate status words");
    BCU(b->redo_count.ensure(16), "allocate redo count");
    BCU(cudaMemsetAsync(b->status.p, 0, 16, b->stream), "clear status words");
  }
  // ---- stage inputs and tables (outside any graph) ----
  cudaStream_t s = b->stream;
  if (b->staged) BCU(cudaStreamSynchronize(b->stream), "synchronize");  // a call that stopped early
  b->staged = true;
  BCU(b->h_src.ensure((size_t)std::max<int64_t>(1, poses_n) * 4), "allocate pinned pose sources");
  if (!rotate) BCU(b->h_poses.ensure((size_t)std::max<int64_t>(1, poses_n) * 48), "allocate pinned poses");
  float* hp = b->h_poses.as<float>();
  int32_t* hsrc = b->h_src.as<int32_t>();
  std::memset(hsrc, 0, (size_t)poses_n * 4);
  std::vector<PackCopy> hcopies;
  std::vector<EvalItem> hitems((size_t)n);
  std::vector<int32_t> hstarts((size_t)n + 1);
  hcopies.reserve((size_t)n_copies);
  for (int i = 0; i < n; ++i) {
    PairPlan& pp = plans[(size_t)i];
    const align_pair& q = pairs[which[(size_t)i]];
    align_grid* g = pp.g;
    if (pp.nB > 0)
      BCU(cudaMemcpyAsync(b->xyz.as<float>() + pp.xyz_off, q.xyzB, (size_t)pp.nB * 12,
                          xyz_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s),
          "copy points");
    if (!pp.hposes.empty() && !rotate) {
      std::memcpy(&hp[(size_t)pp.pose_off * 12], pp.hposes.data(), (size_t)pp.P * 48);
    } else if (!pp.hposes.empty()) {
      BCU(cudaMemcpyAsync(b->poses.as<float>() + pp.pose_off * 12, pp.hposes.data(), (size_t)pp.P * 48,
                          cudaMemcpyHostToDevice, s),
          "copy poses");
    } else {
      BCU(cudaMemcpyAsync(b->poses.as<float>() + pp.pose_off * 12, q.poses12, (size_t)pp.P * 48,
                          cudaMemcpyDeviceToDevice, s),
          "copy poses");
    }
    if (pp.prerot)
      for (int64_t p = 0; p < pp.P; ++p) hsrc[(size_t)(pp.pose_off + p)] = pp.set.src[(size_t)p];
    for (int c = 0; c < pp.n_copies; ++c) {
      PackCopy pc{};
      pc.xyz = b->xyz.as<float>() + pp.xyz_off;
      pc.n = pp.nB;
      pc.n_out = pp.n_pad;
      pc.out = b->pts.as<float4>() + pp.pts_off + (int64_t)c * pp.n_pad;
      pc.rotate = pp.prerot ? 1 : 0;
      for (int k = 0; k < 9; ++k) pc.R[k] = pp.prerot ? pp.set.rots[(size_t)c * 9 + k] : 0.0f;
      hcopies.push_back(pc);
    }
    EvalItem& it = hitems[(size_t)i];
    it.gc = g->gc;
    it.symA = g->symA.as<uint8_t>();
    it.sat = g->sat.as<int32_t>();
    it.src = b->pts.as<float4>() + pp.pts_off;
    it.src_stride = (uint64_t)pp.n_pad;
    it.pose_src = pp.prerot ? b->pose_src.as<int32_t>() + pp.pose_off : nullptr;
    it.poses = b->poses.as<float>() + pp.pose_off * 12;
    it.n_tiles = pp.n_tiles;
    it.P = (int32_t)pp.P;
    it.pose_base = (int32_t)pp.pose_off;
    it.out_c = b->outc.as<uint32_t>() + pp.outc_off;
    it.out_box = b->box.as<int32_t>() + pp.pose_off * 6;
    it.mi = b->mi.as<float>() + pp.pose_off;
    it.hist = nullptr;
    it.best = b->best.as<unsigned long long>() + i;
    it.argmax = b->argmax.as<int64_t>() + i;
    it.dump = nullptr;
    it.passes0 = pp.passes0;
    if (pp.n_units > 0)  // a pageable source: staged before the copy call returns
      BCU(cudaMemcpyAsync(b->units.as<int32_t>() + 2 * pp.unit_off, pp.units.data(), pp.units.size() * 4,
                          cudaMemcpyHostToDevice, s),
          "copy pose pairs");
    it.item_passes = b->ipasses.as<uint32_t>() + i;
    if (pp.by_groups)  // likewise
      BCU(cudaMemcpyAsync(b->order.as<int32_t>() + pp.order_off, pp.set.pose_of.data(), (size_t)pp.P * 4,
                          cudaMemcpyHostToDevice, s),
          "copy lattice order");
    hstarts[(size_t)i] = (int32_t)pp.pose_off;
  }
  hstarts[(size_t)n] = (int32_t)poses_n;
  if (!rotate && poses_n > 0)
    BCU(cudaMemcpyAsync(b->poses.p, hp, (size_t)poses_n * 48, cudaMemcpyHostToDevice, s), "copy poses");
  if (poses_n > 0)
    BCU(cudaMemcpyAsync(b->pose_src.p, hsrc, (size_t)poses_n * 4, cudaMemcpyHostToDevice, s),
        "copy pose sources");
  BCU(cudaMemcpyAsync(b->copies.p, hcopies.data(), hcopies.size() * sizeof(PackCopy), cudaMemcpyHostToDevice, s),
      "copy copy table");
  BCU(cudaMemcpyAsync(b->items.p, hitems.data(), hitems.size() * sizeof(EvalItem), cudaMemcpyHostToDevice, s),
      "copy item table");
  BCU(cudaMemcpyAsync(b->starts.p, hstarts.data(), hstarts.size() * 4, cudaMemcpyHostToDevice, s),
      "copy item starts");
  // ---- launch ----
  Launch L;
  L.ek = &ek;
  L.shape = shape;
  L.n_ctas = n_ctas;
  L.rotate = rotate;
  L.vws = vws;
  L.n_items = n;
  L.n_copies = n_copies;
  L.max_out = max_out;
  EvalArgs& a = L.a;
  a.items = b->items.as<EvalItem>();
  a.item_start = b->starts.as<int32_t>();
  a.n_items = n;
  a.P = (int32_t)poses_n;
  a.K = maxK;
  a.table_slots = T;
  a.n_buckets = T / 4;
  a.passes0 = 1;  // every item brings its grid's own partition count
  uint32_t* status = b->status.as<uint32_t>();
  a.err = status;
  a.max_passes = status + 1;
  a.wide_count = status + 2;
  a.wide_poses = status + 3;
  a.wide = b->wide.as<unsigned long long>();
  a.redo_list = b->redo_list.as<uint32_t>();
  a.redo_count = b->redo_count.as<uint32_t>();
  a.ovf = b->ovf.as<uint4>();
  a.ovf_cap = ek.ovf_cap();
  for (int i = 0; i < n; ++i) {
    EvalArgs ai = a;
    ai.one = hitems[(size_t)i];
    ai.items = nullptr;  // a single item is read from the parameters
    ai.item_start = nullptr;
    ai.n_items = 1;
    ai.p_begin = (int32_t)plans[(size_t)i].pose_off;
    ai.P = (int32_t)(plans[(size_t)i].pose_off + plans[(size_t)i].P);
    ai.K = plans[(size_t)i].g->gc.K;
    ai.table_slots = Ts[(size_t)i];
    ai.n_buckets = Ts[(size_t)i] / 4;
    ai.units = plans[(size_t)i].n_units > 0 ? b->units.as<int32_t>() + 2 * plans[(size_t)i].unit_off : nullptr;
    ai.n_units = plans[(size_t)i].n_units;
    if (plans[(size_t)i].spill_np > 0) {
      ai.spill = b->spill.as<uint4>();
      ai.spill_cap = plans[(size_t)i].spill_cap;
      ai.spill_np = plans[(size_t)i].spill_np;
    }
    L.evals.push_back(ai);
    LatticeArgs la = plans[(size_t)i].lat;
    if (plans[(size_t)i].by_groups) {
      const EvalItem& it = hitems[(size_t)i];
      lattice_carve(la, b->lattice.as<uint8_t>());
      la.symA = it.symA;
      la.xyz = b->xyz.as<float>() + plans[(size_t)i].xyz_off;
      la.poses = it.poses;
      la.pose_of = b->order.as<int32_t>() + plans[(size_t)i].order_off;
      la.pose_base = it.pose_base;
      la.tiles = RawTiles{b->pts.as<float4>() + plans[(size_t)i].pts_off, plans[(size_t)i].n_pad, ek.threads, ek.ppt};
      la.out_c = it.out_c;
      la.out_box = it.out_box;
      la.best = it.best;
      la.redo_list = a.redo_list;
      la.redo_count = a.redo_count;
    }
    L.lats.push_back(la);
    L.lat_rots.push_back(plans[(size_t)i].by_groups ? plans[(size_t)i].set.n_rot : 0);
  }
  b->last_grids.clear();
  b->last_pairs.clear();
  b->last_vws = vws;
  for (size_t i = 0; i < plans.size(); ++i)
    if (plans[i].by_groups) b->last_vws[i] = 0;  // no table layout to learn from
  for (const PairPlan& pp : plans) {
    b->last_grids.push_back(pp.g);
    b->last_pairs.push_back(pp.n_units > 0 ? 1 : 0);
  }
  b->last_shape = shape;
  // a graph replays the kernels' parameters as captured, the pairs' items included
  uint64_t h = 1469598103934665603ull;
  const unsigned char* hb = reinterpret_cast<const unsigned char*>(hitems.data());
  for (size_t k = 0; k < hitems.size() * sizeof(EvalItem); ++k) h = (h ^ hb[k]) * 1099511628211ull;
  std::vector<int64_t> sig = {shape,   n,       rotate,     a.passes0, T, n_ctas,
                              poses_n, n_copies, max_out,   maxK,      (int64_t)(uintptr_t)b->pts.p,
                              (int64_t)(uintptr_t)b->items.p, (int64_t)h};
  for (size_t i = 0; i < vws.size(); ++i)
    sig.insert(sig.end(), {vws[i], Ts[i], plans[i].n_units, plans[i].spill_np, plans[i].spill_cap,
                           plans[i].by_groups ? plans[i].set.n_rot : 0, plans[i].set.mx, plans[i].set.my,
                           plans[i].set.mz, plans[i].nB});
  sig.push_back((int64_t)(uintptr_t)b->units.p);
  sig.push_back((int64_t)(uintptr_t)b->spill.p);
  sig.push_back((int64_t)(uintptr_t)b->order.p);
  sig.push_back((int64_t)(uintptr_t)b->lattice.p);
  st = run_launch(b, L, (flags & ALIGN_BATCH_GRAPH) != 0, sig);
  if (st != ALIGN_OK) return st;
  b->stats[3] = shape;
  b->stats[4] = T;
  b->stats[8] = units_n > 0 ? 2 : 1;
  return ALIGN_OK;
}

}  // namespace

namespace {

align_status eval_batch(align_batch* b, const align_pair* pairs, int32_t n_pairs, int flags) {
  BCU(cudaSetDevice(b->device), "cudaSetDevice");
  // work already queued on the caller's stream (device inputs) comes first
  BCU(cudaEventRecord(b->ev_in, b->user_stream), "record event");
  BCU(cudaStreamWaitEvent(b->stream, b->ev_in, 0), "wait event");
  const bool poses_dev = (flags & ALIGN_POSES_DEVICE) != 0;
  const bool out_dev = (flags & ALIGN_OUT_DEVICE) != 0;
  std::vector<PairPlan> plans;
  std::vector<int32_t> which;  // plan -> pair index
  for (int32_t i = 0; i < n_pairs; ++i) {
    const align_pair& q = pairs[i];
    if (!q.grid) return report_errorf(ALIGN_E_INVALID, "pair %d: grid is NULL", i);
    if (q.grid->device != b->device) return report_errorf(ALIGN_E_INVALID, "pair %d: grid on another device", i);
    if (!q.grid->has_ref) return report_errorf(ALIGN_E_NOREF, "pair %d: no reference scan set", i);
    if (q.nB < 0 || q.nB >= INT32_MAX) return report_errorf(ALIGN_E_INVALID, "pair %d: nB out of range", i);
    if (q.nB > 0 && !q.xyzB) return report_errorf(ALIGN_E_INVALID, "pair %d: xyzB is NULL", i);
    if (q.P < 0 || q.P >= INT32_MAX) return report_errorf(ALIGN_E_INVALID, "pair %d: P out of range", i);
    if (q.P > 0 && ((q.poses12 == nullptr) == (q.eta6 == nullptr)))
      return report_errorf(ALIGN_E_INVALID, "pair %d: give exactly one of poses12 and eta6", i);
    if (q.P > 0 && q.eta6 && poses_dev) return report_errorf(ALIGN_E_INVALID, "pair %d: eta6 must be host memory", i);
    if (q.P > 0 && !q.mi_out) return report_errorf(ALIGN_E_INVALID, "pair %d: mi_out is NULL", i);
    if (q.P == 0) continue;
    PairPlan pp;
    pp.g = q.grid;
    pp.nB = q.nB;
    pp.P = q.P;
    if (q.eta6) {
      pp.hposes.resize((size_t)q.P * 12);
      round_poses_host(q.grid->origin, q.eta6, q.P, pp.hposes.data());
    } else if (!poses_dev) {
      pp.hposes.assign(q.poses12, q.poses12 + (size_t)q.P * 12);
    }
    for (float v : pp.hposes)
      if (!std::isfinite(v)) return report_errorf(ALIGN_E_INVALID, "pair %d: a pose is not finite", i);
    plans.push_back(std::move(pp));
    which.push_back(i);
  }
  // pairs without poses: argmax -1
  for (int32_t i = 0; i < n_pairs; ++i) {
    if (pairs[i].P != 0 || !pairs[i].argmax_out) continue;
    const int64_t none = -1;
    if (out_dev)
      BCU(cudaMemcpyAsync(pairs[i].argmax_out, &none, 8, cudaMemcpyHostToDevice, b->stream), "write argmax");
    else
      *pairs[i].argmax_out = -1;
  }
  if (plans.empty()) {
    BCU(cudaStreamSynchronize(b->stream), "synchronize");
    return ALIGN_OK;
  }
  // Lattices by groups, unless the caller fixed the table kernels' shape or poses per CTA: those with
  // a group per SM (smaller ones share the table kernels' launches, two per pair).
  // (once a pair rotates in the kernel all table pairs do, and only lattices are looked for: 22 us of
  // hashing per pair of 500 poses without shared rotations otherwise)
  bool rotate = std::any_of(plans.begin(), plans.end(), [](const PairPlan& pp) { return pp.hposes.empty(); });
  for (PairPlan& pp : plans) {
    if (pp.hposes.empty() || (rotate && !may_be_lattice(pp.hposes.data(), pp.P))) continue;
    pp.set = pose_set(pp.hposes.data(), pp.P);
    pp.by_groups = b->shape_fixed < 0 && b->pairs_fixed < 0 && pp.set.lattice && pp.g->sweep_mode < 0 &&
                   plan_lattice(pp.g->gc, b->n_sm, b->smem_optin, pp.nB, pp.set.n_rot, pp.set.mx, pp.set.my, pp.set.mz,
                                pp.set.t_max, b->n_sm, pp.lat);
    rotate = rotate || (!pp.by_groups && pp.set.n_rot <= 0);
  }
  size_t lattice_bytes = 0;
  for (PairPlan& pp : plans)
    if (pp.by_groups) lattice_bytes = std::max(lattice_bytes, lattice_carve(pp.lat, nullptr));
  if (lattice_bytes > 0) {
    BCU(lattice_setup(), "set up lattice kernels");  // before any capture
    // without the memory for it the table kernels take the poses
    const void* const old = b->lattice.p;
    const bool ok = b->optional_on && b->lattice.ensure(lattice_bytes, b->optional_limit);
    if (b->lattice.p != old) drop_graph(b);
    if (!ok)
      for (PairPlan& pp : plans) pp.by_groups = false;
  }
  const bool tables = std::any_of(plans.begin(), plans.end(), [](const PairPlan& pp) { return !pp.by_groups; });
  // kernel shape and poses per CTA: fixed, tuned (cached per batch class) or the default
  // (shape 0, pose pairs)
  int shape = b->shape_fixed >= 0 ? b->shape_fixed : 0;
  bool pose_pairs = b->pairs_fixed != 1;
  if (tables && (b->shape_fixed < 0 || b->pairs_fixed < 0) && (flags & ALIGN_BATCH_TUNE)) {
    int64_t pts_tot = 0, poses_tot = 0;
    int maxK = 0;
    bool dev_poses = false;
    for (const PairPlan& pp : plans) {
      pts_tot += pp.nB;
      poses_tot += pp.P;
      maxK = std::max(maxK, (int)pp.g->gc.K);
      dev_poses = dev_poses || pp.hposes.empty();
    }
    char buf[256];
    std::snprintf(buf, sizeof(buf), "%s/pairs%d/pts%d/poses%d/K%d/devposes%d", b->device_name.c_str(),
                  bucket_log2((int64_t)plans.size()), bucket_log2(pts_tot / (int64_t)plans.size() + 1),
                  bucket_log2(poses_tot + 1), maxK, dev_poses ? 1 : 0);
    const std::string key = buf;
    bool known = false;
    {
      std::lock_guard<std::mutex> lock(g_tune_mu);
      tune_load_locked();
      auto it = g_tune.find(key);
      if (it != g_tune.end()) {
        shape = it->second / 2;
        pose_pairs = (it->second % 2) == 1;
        known = true;
      }
    }
    if (!known) {
      // time every candidate (kernel shape x poses per CTA) on this batch: one warm-up run,
      // then the sum of three timed runs (device time between events)
      double best_ms = 0.0;
      int best = -1;
      for (int c = 0; c < kChoices; ++c) {
        const int cs = c / 2;
        const bool cp = (c % 2) == 1;
        if (b->shape_fixed >= 0 && cs != b->shape_fixed) continue;
        if (b->pairs_fixed >= 1 && cp != (b->pairs_fixed == 2)) continue;
        double total = 0.0;
        for (int rep = 0; rep < 4; ++rep) {
          align_status st = eval_batch_shape(b, plans, pairs, which, flags & ~ALIGN_BATCH_GRAPH, cs, cp);
          if (st != ALIGN_OK) return st;
          st = collect(b);
          if (st != ALIGN_OK) return st;
          if (rep > 0) total += (double)b->stats[6] / 1000.0;
        }
        b->stats[7] += 1;
        if (best < 0 || total < best_ms) {
          best_ms = total;
          best = c;
        }
      }
      shape = best / 2;
      pose_pairs = (best % 2) == 1;
      std::lock_guard<std::mutex> lock(g_tune_mu);
      tune_store_locked(key, best);
    }
  }
  align_status st = eval_batch_shape(b, plans, pairs, which, flags, shape, pose_pairs);
  if (st != ALIGN_OK) return st;
  // outputs
  const cudaMemcpyKind kind = out_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  for (size_t k = 0; k < plans.size(); ++k) {
    const align_pair& q = pairs[which[k]];
    BCU(cudaMemcpyAsync(q.mi_out, b->mi.as<float>() + plans[k].pose_off, (size_t)plans[k].P * 4, kind, b->stream),
        "read MI");
    if (q.argmax_out)
      BCU(cudaMemcpyAsync(q.argmax_out, b->argmax.as<int64_t>() + k, 8, kind, b->stream), "read argmax");
  }
  return collect(b);
}

}  // namespace

extern "C" align_status align_eval_batch(align_batch* b, const align_pair* pairs, int32_t n_pairs, int flags) {
  if (!b) return report_error(ALIGN_E_INVALID, "batch is NULL");
  if (n_pairs < 0 || (n_pairs > 0 && !pairs)) return report_error(ALIGN_E_INVALID, "bad pair array");
  align_status st = eval_batch(b, pairs, n_pairs, flags);
  if (st != ALIGN_E_OOM || b->lattice.p == nullptr) return st;
  drop_graph(b);  // once more without the groups' workspace (no results have been returned yet)
  b->lattice.release();
  b->optional_on = false;
  st = eval_batch(b, pairs, n_pairs, flags);
  b->optional_on = true;
  return st;
}

