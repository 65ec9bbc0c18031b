// Host-side runtime structures of the Jacobi3D library (shared by the C-ABI
// translation units; not part of the public interface).
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <cstdarg>
#include <cstdint>
#include <mutex>
#include <shared_mutex>
#include <string>
#include <vector>

#include "../../include/jacobi.h"
#include "common.cuh"
#include "kernels.cuh"

namespace jgb {

// Thread-local message of the last failing call.
int set_error(int code, const char* fmt, ...);
#define JGB_CUDA(call)                                                                      \
  do {                                                                                      \
    cudaError_t e_ = (call);                                                                \
    if (e_ != cudaSuccess)                                                                  \
      return ::jgb::set_error(JACOBI_ECUDA, "%s failed: %s (%s:%d)", #call,                 \
                              cudaGetErrorString(e_), __FILE__, __LINE__);                 \
  } while (0)

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

struct BlockHost {
  int64_t grid;
  int64_t origin[3], extent[3];
  int64_t nbr[6];
  int64_t item_begin, item_end;  // items of this block in the full list
  int64_t rx, ry;                // padded row pitch and rows per plane
  int64_t pitch;                 // elements per z-plane
  size_t u_off[2];
  size_t recv_off[6][2];
  size_t stage_off[6];           // explicit-path staging (internal faces only)
};

struct GridHost {
  jacobi_dim3 dims;
  jacobi_split split;
  jacobi_init init;
  int64_t counts[3];
  int64_t block_begin, block_end;
  int64_t item_begin, item_end;
  int32_t max_rows = 0;  // most extended rows (ny + 2) * (nz + 2) of a block
  int64_t start_iter;    // global iteration at which the local count was 0
  int64_t frozen_local;  // local iteration held while inactive
  bool active;
};

// Decomposition + workspace layout of a set of grids.
struct Plan {
  int32_t dtype;
  size_t elem;
  std::vector<GridHost> grids;
  std::vector<BlockHost> blocks;
  std::vector<WorkItem> items;
  int64_t n_points = 0;
  int64_t halo_elems = 0;  // face elements moved per iteration (internal faces)
  uint32_t max_stage = 0;  // largest ring stage (bytes) of a plane-streamed block
  int64_t zchunk = 1;      // planes per z-chunk (the last chunk of a block may be shorter)
  int32_t cw_cap = 8;      // most consumer warps per streaming CTA (sets the row windows)
  int64_t n_units = 0;     // persistent-kernel units: (block, z-chunk) pairs
  int64_t cap_items = 0;   // item / unit table capacity in the workspace (the finest shape)
  int64_t cap_units = 0;
  // byte offsets into the workspace
  size_t off_blocks, off_geom, off_items, off_active, off_kind, off_grids, off_norms, off_inits, off_gids, off_partials,
      off_progress, off_err, off_stage_tab, off_punit_items, off_punit_ids, off_pdep_off, off_pdep_ids,
      off_active_blocks, off_it0, off_ticket;
  size_t res_bytes = 0;    // resident-path tables and packets of a handle whose grids fit (not part of `bytes`)
  size_t off_stage_begin = 0, off_stage_end = 0;  // the explicit-path staging buffers, contiguous
  int64_t halo_faces = 0;                         // internal faces (one message each per iteration)
  size_t bytes = 0;
};

// With target_items <= 0 (a handle) the z-chunk comes from a cost model of
// waves, per-item pipeline fill and halo re-reads; with target_items > 0 it is
// the longest chunk that still gives that many items.  The server plans each
// request alone (so its result does not depend on the mix) with
// kServeTargetItems and z-chunks of at least kServeMinChunk planes: a request
// running alone still spreads over the GPU, while the halo planes each chunk
// re-reads stay a bounded share.
constexpr int64_t kServeTargetItems = 304;
constexpr int kMaxBlockExtent = JACOBI_MAX_BLOCK_EXTENT;
constexpr int64_t kServeMinChunk = 16;
int plan_build(int64_t n_grids, const jacobi_dim3* grids, const jacobi_split* splits, jacobi_dtype dtype,
               const jacobi_init* inits, Plan* out, int64_t target_items = 0, int64_t min_chunk = 1);
// Rebuild the work items of a built plan for another shape (z-chunk zc_req,
// 0 = the cost model's; at most cw_cap consumer warps per streaming CTA).
int plan_items(Plan* P, int64_t zc_req, int cw_cap, int64_t target_items, int64_t min_chunk);

// Resident path: a plan's grid as resident_plan takes it, and the layout of its
// tables and packets (byte offsets).
struct ResLayout {
  size_t grids, ctl, packets, bytes;
};
ResGrid resident_grid(const GridHost& G, int32_t index);
ResLayout resident_layout(const ResPlan& rp, size_t n_grids);

// Device block table entries of a plan whose workspace starts at `ws`; block
// and neighbour ids are offset by `base`; grid_override >= 0 replaces every
// block's grid index.  stage_tab (nullable) receives the explicit-path staging
// buffers (6 per block).  local_halo aims every block's face stores at its own
// receive slots instead of its neighbours' (the halo-share measurement).
void fill_block_tables(const Plan& P, char* ws, int64_t base, int32_t grid_override, BlockDev* bd, BlockGeom* geo,
                       void** stage_tab, bool local_halo = false);

}  // namespace jgb

namespace jgb {

// Resident-path tables of one handle (resident.cu), rebuilt with the active lists
// in memory that it gets at its creation: behind a workspace of the library's own,
// or an allocation beside a caller's.
constexpr int32_t kResRefused = -2;
struct Resident {
  bool allowed = true;   // off when the environment asks for a given persistent kernel
  bool ok = false;       // the active grids fit
  int n_boxes = 0, smem = 0;
  int64_t min_iters = 0; // shortest call it takes
  double iter_ns = 0.0, launch_ns = 0.0;  // estimates (ResPlan)
  double points = 0.0;   // of the active grids
  int64_t launches = 0;  // so far, for jacobi_info
  bool unchecked = false;  // launched since the error word was last looked at
  int32_t debug = -1;    // jacobi_debug_resident
  char* mem = nullptr;   // Plan::res_bytes
  char* own = nullptr;   // mem, where it is an allocation of its own
  ResBox* d_boxes = nullptr;
  ResGrid* d_grids = nullptr;
  uint32_t* d_ctl = nullptr;
  uint4* d_packets = nullptr;
};

// Channels open on a device.  A resident launch needs all its SMs at once, while
// a channel's receive (or a send whose slot is taken) holds SMs until a message of
// another stream has come: if that message stands behind the launch, neither ends
// before the wait limit.  So no resident launch is issued while a channel is open:
// launches hold `m` shared, and channel_open, which takes it alone to count, waits
// for the device before it hands the channel out.
struct ChannelGate {
  std::shared_mutex m;
  int64_t open = 0;
};
ChannelGate& channel_gate(int dev);

// The steps that the resident kernel could take, one note per handle that has some
// under way on a device.  Resident launches that do not fit side by side take
// turns, while launches per iteration of several streams share the GPU: the steps
// that are under way together are resident or not by which ends them sooner
// (note_steps).  Times are estimates; a note holds for twice its own, or until its
// stream has been waited for through the handle.
struct StepCost {
  int boxes = 0;
  double iter_ns = 0.0;    // a resident iteration
  double launch_ns = 0.0;  // one by the path's other kernels, alone
  double share_ns = 0.0;   // and with others beside it that keep the GPU busy
};
struct StepNote {
  void* stream = nullptr;
  std::atomic<int64_t> until_ns{0};
  double per_iter_ns = 1.0;
  StepCost cost;
  bool listed = false;
};
// Note n iterations of `me` on stream s; true if they should be resident.
bool note_steps(int dev, StepNote* me, void* s, int64_t n, const StepCost& cost);
void drop_note(int dev, StepNote* me);

}  // namespace jgb

struct channel_s;

struct jacobi_s {
  jgb::Plan plan;
  int device = 0;
  char* ws = nullptr;
  bool own_ws = false;
  int32_t path = JACOBI_PATH_FUSED;
  int64_t iter = 0;  // global iterations completed

  // device tables (inside ws)
  jgb::BlockDev* d_blocks = nullptr;
  jgb::BlockGeom* d_geom = nullptr;
  jgb::WorkItem* d_items = nullptr;
  jgb::WorkItem* d_active = nullptr;
  jgb::WorkItem* d_kind = nullptr;
  jgb::GridDev* d_grids = nullptr;
  jgb::GridNorm* d_norms = nullptr;
  jgb::InitDev* d_inits = nullptr;
  int32_t* d_gids = nullptr;
  double* d_partials = nullptr;
  int64_t* d_progress = nullptr;
  uint32_t* d_err = nullptr;
  void** d_stage_tab = nullptr;
  int32_t* d_punit_items = nullptr;
  int32_t* d_punit_ids = nullptr;
  int32_t* d_pdep_off = nullptr;
  int32_t* d_pdep_ids = nullptr;
  int32_t* d_active_blocks = nullptr;  // blocks of the active grids (exchange kernels)
  int64_t* d_it0 = nullptr;            // start iteration of a replayed persistent graph
  unsigned long long* d_ticket = nullptr;  // work counter of the warp-specialised persistent kernel

  // host mirrors
  std::vector<jgb::WorkItem> active_items;
  // persistent kernel: active units (block, z-chunk) in item order, their item
  // ranges in active_items and their dependency lists (unit ids, CSR)
  std::vector<int32_t> active_units;        // unit ids
  std::vector<int32_t> active_unit_items;   // n_active_units + 1 offsets into active_items
  std::vector<int32_t> active_dep_off;      // n_active_units + 1 offsets into active_deps
  std::vector<int32_t> active_deps;
  std::vector<int32_t> active_grids;
  std::vector<int32_t> active_blocks;
  std::vector<jgb::WorkItem> kind_items;        // active items grouped by kind
  int32_t kind_off[jgb::kItemKinds + 1] = {};
  bool tables_dirty = true;
  jgb::GridDev* h_grids = nullptr;   // pinned, uploaded to d_grids
  jgb::GridNorm* h_norms = nullptr;  // pinned, read back from d_norms
  uint32_t* h_err = nullptr;        // pinned: copy of d_err; [1] set by a resident launch that gave up

  jgb::StepNote note;             // steps under way that the resident kernel could take
  jgb::Resident res;              // small problems: all iterations of a call on chip
  jgb::KindFork fork;             // side-by-side launch of the step's item kinds
  // CUDA graph of the fused path
  cudaGraphExec_t graph = nullptr;
  int64_t graph_iters = 0;
  int32_t graph_items = -1;
  // PERSISTENT path: the cooperative launch captured once per shape (without /
  // with the fused residual of the first iteration) and replayed; the start
  // iteration comes from d_it0
  struct PersistGraph {
    cudaGraphExec_t exec = nullptr;
    int64_t n_iters = 0;
    int32_t n_units = -1, stages = 0, ctas = 0, threads = 0, ws_cw = 0;
  } pgraph[2];
  bool persist_ws = true;         // warp-specialised persistent kernel where it applies
  bool pgraph_off = false;        // capture of the cooperative launch failed: launch directly

  uint64_t wait_ns = 1000000000ull;
  int32_t stages = 4;             // ring stages of the persistent kernel's plane streaming
  bool stages_fixed = false;      // set by JACOBI_STAGES or the autotuner (else large stages may take 5)
  int32_t fp64_emu = 1;           // FP64 pair sums on the integer pipe when safe
  int64_t drop_block = -1;        // fault injection (persistent path)
  bool local_halo = false;        // halo-share measurement: face stores stay in the block
  void* stage = nullptr;          // device staging for host transfers
  size_t stage_bytes = 0;
  // host-driven exchange forms (CHANNEL, MESSAGING, HOST_STAGED paths)
  void* h_halo = nullptr;                       // pinned copy of the staging region (HOST_STAGED)
  jgb::CopyDesc* d_desc = nullptr;              // posted receives of one exchange (MESSAGING)
  jgb::CopyDesc* h_desc = nullptr;              // pinned
  struct HaloMeta {                             // metadata message of one face (MESSAGING)
    const void* src;
    int64_t bytes;
    int32_t face;                               // the receiver's face the payload belongs to
  };
  std::vector<std::vector<HaloMeta>> mailbox;   // per receiving block
  std::vector<channel_s*> channels;
};
