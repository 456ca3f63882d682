// Batched execution: one short chain of launches services many maps.
//
// A batch is a list of operations, at most one per (map, phase), on maps of
// key dimension 1..4.  Phases run in the order insert/activate -> find ->
// erase (per map, the order the serving and batched workloads apply), each as
// one persistent kernel over ALL maps of that phase: claim, commit, find,
// erase-mark and erase-resolve.  Work is cut into tiles of blockDim.x keys that
// never straddle two operations, so a commit or erase-resolve tile still
// aggregates its heap atomic over one map.  The kernels read everything (maps,
// pointers, tile counts) from a descriptor table that the first launch copies
// from a pinned ring slot; a last one publishes the maps' control-block
// snapshots.  All are programmatic dependents of the one before, and a phase
// without work is not launched.  (As a CUDA graph of a table copy and six
// kernels the same work took 255 against 237 us for 24 maps, and 96 against
// 81 us when it held finds only: a graph runs its empty phases, copies the
// whole table and has no programmatic edges.)
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <vector>

#include "ash.h"
#include "ash_internal.h"
#include "ash_kernels.cuh"
#include "ash_trace.h"

namespace ash {

constexpr int kBatchMaxOps = 256;
constexpr int kBatchThreads = 256;
constexpr int kBatchRing = 4;
enum { kPhaseInsert = 0, kPhaseFind = 1, kPhaseErase = 2, kPhases = 3 };

struct BatchOp {
  TableView t;
  const int32_t* keys;
  int32_t* idx;    // insert/activate/find: outputs (claim scratch too); erase: slot scratch
  uint8_t* mask;
  ValueRow v;      // v.row_bytes == 0: no value copy
  int64_t n;
  int64_t tile0;   // first tile of this op within its phase
  int32_t key_dim;
  int32_t S;
};

struct BatchPhase {
  int32_t first;
  int32_t count;
  int64_t tiles;
};

// A control-block snapshot that a map asks for after the batch.
struct BatchSnap {
  Ctrl* ctrl;
  Snap* snap;
  uint32_t seq;
};

struct alignas(16) BatchTable {
  BatchPhase ph[kPhases];
  int32_t n_ops;
  int32_t n_snaps;
  BatchSnap snaps[kBatchMaxOps];
  BatchOp ops[kBatchMaxOps];  // last: only the part in use is copied
};

// 16-byte units of the table's part in use; the last may reach past it, so the
// table's size is a multiple of 16.
constexpr int upload_units(int n_ops) {
  return static_cast<int>((offsetof(BatchTable, ops) + sizeof(BatchOp) * n_ops + 15) / 16);
}
static_assert(upload_units(kBatchMaxOps) * 16 <= sizeof(BatchTable), "a full batch is uploaded within its table");

// Copies the table's part in use from pinned host memory (the SMs read it
// over the CPU-GPU link).
__global__ void __launch_bounds__(1024) batch_upload_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst,
                                                            int units) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < units; i += gridDim.x * blockDim.x) dst[i] = src[i];
}

// Loads the tile starts of one phase into shared memory and maps a tile to
// its operation (binary search over at most kBatchMaxOps entries).
__device__ __forceinline__ void load_tile_starts(const BatchTable* tb, int phase, int64_t* s_tile0) {
  asm volatile("griddepcontrol.wait;" ::: "memory");  // every batch kernel is a programmatic dependent
  const BatchPhase ph = tb->ph[phase];
  for (int i = threadIdx.x; i < ph.count; i += blockDim.x) s_tile0[i] = tb->ops[ph.first + i].tile0;
  __syncthreads();
}

__device__ __forceinline__ int op_of_tile(const int64_t* s_tile0, int count, int64_t tile) {
  int lo = 0, hi = count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (s_tile0[mid] <= tile) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// The kernels exist twice: for batches whose maps all have 4-slot buckets (the
// default), and for any bucket sizes.  The 16-slot code alone sets the
// register count of a kernel that holds it (WIDE).
#define ASH_DS_CASES(WIDE, FN, ...)                                 \
  if constexpr (!(WIDE)) {                                          \
    switch (op.key_dim) {                                           \
      case 1: FN<1, 4>(__VA_ARGS__); break;                         \
      case 2: FN<2, 4>(__VA_ARGS__); break;                         \
      case 3: FN<3, 4>(__VA_ARGS__); break;                         \
      default: FN<4, 4>(__VA_ARGS__); break;                        \
    }                                                               \
  } else {                                                          \
    switch (op.key_dim * 100 + op.S) {                              \
      case 104: FN<1, 4>(__VA_ARGS__); break;                       \
      case 108: FN<1, 8>(__VA_ARGS__); break;                       \
      case 116: FN<1, 16>(__VA_ARGS__); break;                      \
      case 204: FN<2, 4>(__VA_ARGS__); break;                       \
      case 208: FN<2, 8>(__VA_ARGS__); break;                       \
      case 216: FN<2, 16>(__VA_ARGS__); break;                      \
      case 304: FN<3, 4>(__VA_ARGS__); break;                       \
      case 308: FN<3, 8>(__VA_ARGS__); break;                       \
      case 316: FN<3, 16>(__VA_ARGS__); break;                      \
      case 404: FN<4, 4>(__VA_ARGS__); break;                       \
      case 408: FN<4, 8>(__VA_ARGS__); break;                       \
      default: FN<4, 16>(__VA_ARGS__); break;                       \
    }                                                               \
  }

// In the batched kernels the full per-key protocols are the main path, so
// they are inlined (the single-map kernels keep them out of line as their
// rare slow path).
template <int D, int S>
__device__ __forceinline__ void batch_claim_one(const BatchOp& op, int64_t pos) {
  // slot order (measured 7 % faster here than preferred-first placement);
  // the host clears the map's pref_placed flag
  op.idx[pos] = claim_key<D, S, const int32_t*, kClaimSlotMask, false>(op.t, op.keys, pos);
}

template <int D, int S>
__device__ __forceinline__ void batch_find_one(const BatchOp& op, int64_t pos) {
  int32_t k[1][D], r[1];
  const bool ok[1] = {true};
  load_input_key<D>(op.keys, pos, k[0]);
  find_keys<D, S, 1>(op.t, k, ok, r);
  op.idx[pos] = r[0];
  op.mask[pos] = r[0] >= 0 ? 1 : 0;
}

template <int D, int S>
__device__ __forceinline__ void batch_mark_one(const BatchOp& op, int64_t pos) {
  op.idx[pos] = erase_mark_one<D, S>(op.t, op.keys, pos);
}

template <bool WIDE>
__global__ void __launch_bounds__(kBatchThreads) batch_claim_kernel(const BatchTable* __restrict__ tb) {
  __shared__ int64_t s_tile0[kBatchMaxOps];
  load_tile_starts(tb, kPhaseInsert, s_tile0);
  const BatchPhase ph = tb->ph[kPhaseInsert];
  for (int64_t tile = blockIdx.x; tile < ph.tiles; tile += gridDim.x) {
    const BatchOp& op = tb->ops[ph.first + op_of_tile(s_tile0, ph.count, tile)];
    const int64_t pos = (tile - op.tile0) * blockDim.x + threadIdx.x;
    if (pos < op.n) { ASH_DS_CASES(WIDE, batch_claim_one, op, pos) }
  }
}

__global__ void __launch_bounds__(kBatchThreads) batch_commit_kernel(const BatchTable* __restrict__ tb) {
  __shared__ int64_t s_tile0[kBatchMaxOps];
  __shared__ TileShared sh;
  load_tile_starts(tb, kPhaseInsert, s_tile0);
  const BatchPhase ph = tb->ph[kPhaseInsert];
  int turn = 0;
  for (int64_t tile = blockIdx.x; tile < ph.tiles; tile += gridDim.x, turn ^= 1) {
    const BatchOp& op = tb->ops[ph.first + op_of_tile(s_tile0, ph.count, tile)];
    const int64_t base0 = (tile - op.tile0) * blockDim.x;
    const bool val = op.v.row_bytes > 0;  // uniform over the block
    switch (op.key_dim * 2 + (val ? 1 : 0)) {
      case 2: commit_tile<1, 1, false>(op.t, op.keys, op.n, base0, op.idx, op.mask, op.v, sh, turn); break;
      case 3: commit_tile<1, 1, true>(op.t, op.keys, op.n, base0, op.idx, op.mask, op.v, sh, turn); break;
      case 4: commit_tile<2, 1, false>(op.t, op.keys, op.n, base0, op.idx, op.mask, op.v, sh, turn); break;
      case 5: commit_tile<2, 1, true>(op.t, op.keys, op.n, base0, op.idx, op.mask, op.v, sh, turn); break;
      case 6: commit_tile<3, 1, false>(op.t, op.keys, op.n, base0, op.idx, op.mask, op.v, sh, turn); break;
      case 7: commit_tile<3, 1, true>(op.t, op.keys, op.n, base0, op.idx, op.mask, op.v, sh, turn); break;
      case 8: commit_tile<4, 1, false>(op.t, op.keys, op.n, base0, op.idx, op.mask, op.v, sh, turn); break;
      default: commit_tile<4, 1, true>(op.t, op.keys, op.n, base0, op.idx, op.mask, op.v, sh, turn); break;
    }
  }
}

template <bool WIDE>
__global__ void __launch_bounds__(kBatchThreads) batch_find_kernel(const BatchTable* __restrict__ tb) {
  __shared__ int64_t s_tile0[kBatchMaxOps];
  load_tile_starts(tb, kPhaseFind, s_tile0);
  const BatchPhase ph = tb->ph[kPhaseFind];
  for (int64_t tile = blockIdx.x; tile < ph.tiles; tile += gridDim.x) {
    const BatchOp& op = tb->ops[ph.first + op_of_tile(s_tile0, ph.count, tile)];
    const int64_t pos = (tile - op.tile0) * blockDim.x + threadIdx.x;
    if (pos < op.n) { ASH_DS_CASES(WIDE, batch_find_one, op, pos) }
  }
}

template <bool WIDE>
__global__ void __launch_bounds__(kBatchThreads) batch_erase_mark_kernel(const BatchTable* __restrict__ tb) {
  __shared__ int64_t s_tile0[kBatchMaxOps];
  load_tile_starts(tb, kPhaseErase, s_tile0);
  const BatchPhase ph = tb->ph[kPhaseErase];
  for (int64_t tile = blockIdx.x; tile < ph.tiles; tile += gridDim.x) {
    const BatchOp& op = tb->ops[ph.first + op_of_tile(s_tile0, ph.count, tile)];
    const int64_t pos = (tile - op.tile0) * blockDim.x + threadIdx.x;
    if (pos < op.n) { ASH_DS_CASES(WIDE, batch_mark_one, op, pos) }
  }
}

template <bool WIDE>
__global__ void __launch_bounds__(kBatchThreads) batch_erase_resolve_kernel(const BatchTable* __restrict__ tb) {
  __shared__ int64_t s_tile0[kBatchMaxOps];
  __shared__ TileShared sh;
  load_tile_starts(tb, kPhaseErase, s_tile0);
  const BatchPhase ph = tb->ph[kPhaseErase];
  int turn = 0;
  for (int64_t tile = blockIdx.x; tile < ph.tiles; tile += gridDim.x, turn ^= 1) {
    const BatchOp& op = tb->ops[ph.first + op_of_tile(s_tile0, ph.count, tile)];
    const int64_t base0 = (tile - op.tile0) * blockDim.x;
    if (!WIDE || op.S == 4) erase_resolve_tile<4>(op.t, op.n, base0, op.idx, op.mask, sh, turn);
    else if (op.S == 8) erase_resolve_tile<8>(op.t, op.n, base0, op.idx, op.mask, sh, turn);
    else erase_resolve_tile<16>(op.t, op.n, base0, op.idx, op.mask, sh, turn);
  }
}

// Publishes the snapshots of every map that asked for one, once its
// operations are done.
__global__ void __launch_bounds__(kBatchMaxOps) batch_snapshot_kernel(const BatchTable* __restrict__ tb) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int i = threadIdx.x;
  if (i < tb->n_snaps) publish_snapshot(tb->snaps[i].ctrl, tb->snaps[i].snap, tb->snaps[i].seq);
}

}  // namespace ash

using namespace ash;
using namespace ash::host;

struct ash_batch {
  int device = 0;
  int grid = 0;
  Allocator alloc;
  struct Slot {
    BatchTable* h = nullptr;  // pinned
    BatchTable* d = nullptr;
    cudaEvent_t done = nullptr;
    bool used = false;
    int32_t* scratch = nullptr;  // erase slot indices
    int64_t scratch_n = 0;
  } slot[kBatchRing];
  int next = 0;
  std::mutex mu;
};

namespace {

// How many kernels launch_batch launches.
int batch_launches(const BatchTable& tb) {
  return 1 + (tb.ph[kPhaseInsert].tiles > 0 ? 2 : 0) + (tb.ph[kPhaseFind].tiles > 0 ? 1 : 0) +
         (tb.ph[kPhaseErase].tiles > 0 ? 2 : 0) + (tb.n_snaps > 0 ? 1 : 0);
}

// The batch's kernels on st, empty phases left out.
template <bool WIDE>
void launch_batch(const ash_batch* b, const ash_batch::Slot& s, cudaStream_t st) {
  const BatchTable* tb = s.h;
  const BatchTable* d = s.d;
  auto grid = [&](int phase) {
    const int64_t tiles = tb->ph[phase].tiles;
    return static_cast<int>(tiles < b->grid ? tiles : b->grid);
  };
  const int units = upload_units(tb->n_ops);
  launch_dependent(batch_upload_kernel, (units + 1023) / 1024, 1024, st, reinterpret_cast<const uint4*>(s.h),
                   reinterpret_cast<uint4*>(s.d), units);
  if (tb->ph[kPhaseInsert].tiles > 0) {
    launch_dependent(batch_claim_kernel<WIDE>, grid(kPhaseInsert), kBatchThreads, st, d);
    launch_dependent(batch_commit_kernel, grid(kPhaseInsert), kBatchThreads, st, d);
  }
  if (tb->ph[kPhaseFind].tiles > 0)
    launch_dependent(batch_find_kernel<WIDE>, grid(kPhaseFind), kBatchThreads, st, d);
  if (tb->ph[kPhaseErase].tiles > 0) {
    launch_dependent(batch_erase_mark_kernel<WIDE>, grid(kPhaseErase), kBatchThreads, st, d);
    launch_dependent(batch_erase_resolve_kernel<WIDE>, grid(kPhaseErase), kBatchThreads, st, d);
  }
  if (tb->n_snaps > 0) launch_dependent(batch_snapshot_kernel, 1, kBatchMaxOps, st, d);
}

void* batch_alloc(ash_batch* b, size_t bytes, cudaStream_t st) {
  if (b->alloc.alloc) return b->alloc.alloc(bytes, b->device, reinterpret_cast<ash_stream>(st), b->alloc.ctx);
  void* p = nullptr;
  if (cudaMallocAsync(&p, bytes, st) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return p;
}

void batch_free(ash_batch* b, void* p, cudaStream_t st) {
  if (!p) return;
  if (b->alloc.free) b->alloc.free(p, b->device, reinterpret_cast<ash_stream>(st), b->alloc.ctx);
  else cudaFreeAsync(p, st);
}

int phase_of(int32_t op) {
  switch (op) {
    case ASH_OP_INSERT: case ASH_OP_ACTIVATE: return kPhaseInsert;
    case ASH_OP_FIND: return kPhaseFind;
    case ASH_OP_ERASE: return kPhaseErase;
    default: return -1;
  }
}

}  // namespace

extern "C" {

ash_status ash_batch_create(int device, ash_batch** out_host) {
  if (!out_host) return fail(ASH_ERR_INVALID, "out is NULL");
  *out_host = nullptr;
  int n_dev = 0;
  if (cudaGetDeviceCount(&n_dev) != cudaSuccess || device < 0 || device >= n_dev) {
    cudaGetLastError();
    return fail(ASH_ERR_INVALID, "no such CUDA device");
  }
  DeviceGuard g(device);
  ash_batch* b = new ash_batch();
  b->device = device;
  b->grid = sm_count(device) * 8;
  for (auto& s : b->slot) {
    if (cudaMallocHost(&s.h, sizeof(BatchTable)) != cudaSuccess || cudaMalloc(&s.d, sizeof(BatchTable)) != cudaSuccess ||
        cudaEventCreateWithFlags(&s.done, cudaEventDisableTiming) != cudaSuccess) {
      cudaGetLastError();
      ash_batch_destroy(b);
      return fail(ASH_ERR_OOM, "batch context allocation failed");
    }
    std::memset(s.h, 0, sizeof(BatchTable));
  }
  *out_host = b;
  return ASH_OK;
}

ash_status ash_batch_destroy(ash_batch* b) {
  if (!b) return ASH_OK;
  DeviceGuard g(b->device);
  for (auto& s : b->slot) {
    if (s.done) cudaEventSynchronize(s.done);
    if (s.h) cudaFreeHost(s.h);
    if (s.d) cudaFree(s.d);
    if (s.done) cudaEventDestroy(s.done);
    batch_free(b, s.scratch, nullptr);
  }
  cudaDeviceSynchronize();
  delete b;
  return ASH_OK;
}

ash_status ash_batch_run(ash_batch* b, const ash_batch_op* ops, int n_ops, ash_stream stream) {
  if (!b) return fail(ASH_ERR_INVALID, "batch is NULL");
  if (n_ops < 0 || n_ops > kBatchMaxOps) return fail(ASH_ERR_INVALID, "n_ops must be in [0, 256]");
  if (n_ops > 0 && !ops) return fail(ASH_ERR_INVALID, "ops is NULL");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  // ---- validate
  std::vector<std::pair<const ash_map*, int>> seen;
  int64_t erase_total = 0;
  for (int i = 0; i < n_ops; ++i) {
    const ash_batch_op& o = ops[i];
    const int ph = phase_of(o.op);
    if (ph < 0) return fail(ASH_ERR_INVALID, "unknown batch op code");
    ash_status s = check_keys(o.map, o.keys, o.n);
    if (s != ASH_OK) return s;
    if (o.map->device != b->device) return fail(ASH_ERR_INVALID, "map is on another device than the batch");
    if (o.map->key_dim > 4) return fail(ASH_ERR_INVALID, "batched maps support key_dim 1..4");
    if (o.n > 0 && !o.masks) return fail(ASH_ERR_INVALID, "masks is required");
    if (o.n > 0 && ph != kPhaseErase && !o.buf_indices) return fail(ASH_ERR_INVALID, "buf_indices is required");
    if (o.op == ASH_OP_INSERT && o.map->n_values > 0) {
      const int64_t rb = o.map->row_bytes[0];
      if (o.map->n_values != 1 || !(rb == 4 || rb == 8 || rb == 16) || !o.values ||
          vec_width(rb, o.map->vb[0], o.values) != rb)
        return fail(ASH_ERR_INVALID,
                    "batched insert needs one value buffer of 4, 8 or 16-byte rows with aligned values");
    }
    for (auto& p : seen)
      if (p.first == o.map && p.second == ph) return fail(ASH_ERR_INVALID, "two ops on one map in the same phase");
    seen.emplace_back(o.map, ph);
    if (ph == kPhaseErase) erase_total += o.n;
  }
  DeviceGuard g(b->device);
  std::lock_guard<std::mutex> lk(b->mu);
  // ---- growth for the insert phase (may synchronise)
  for (int i = 0; i < n_ops; ++i) {
    if (phase_of(ops[i].op) == kPhaseInsert && ops[i].n > 0) {
      ash_status s = ensure_room(ops[i].map, ops[i].n, st);
      if (s != ASH_OK) return s;
    }
  }
  ash_batch::Slot& sl = b->slot[b->next];
  b->next = (b->next + 1) % kBatchRing;
  if (sl.used && cudaEventSynchronize(sl.done) != cudaSuccess) return cuda_fail(cudaGetLastError(), "batch slot wait");
  if (sl.scratch_n < erase_total) {
    batch_free(b, sl.scratch, st);
    sl.scratch_n = std::max<int64_t>(erase_total, 2 * sl.scratch_n);
    sl.scratch = static_cast<int32_t*>(batch_alloc(b, sl.scratch_n * 4, st));
    if (!sl.scratch) {
      sl.scratch_n = 0;
      return fail(ASH_ERR_OOM, "batch scratch allocation failed");
    }
  }
  // ---- descriptor table, grouped by phase
  BatchTable* tb = sl.h;
  int k = 0;
  int64_t scratch_off = 0;
  for (int ph = 0; ph < kPhases; ++ph) {
    tb->ph[ph].first = k;
    int64_t tiles = 0;
    for (int i = 0; i < n_ops; ++i) {
      const ash_batch_op& o = ops[i];
      if (phase_of(o.op) != ph || o.n == 0) continue;
      BatchOp& d = tb->ops[k++];
      d.t = view_of(o.map);
      d.keys = o.keys;
      d.mask = o.masks;
      d.n = o.n;
      d.key_dim = o.map->key_dim;
      d.S = o.map->S;
      d.tile0 = tiles;
      d.v = ValueRow{};
      if (ph == kPhaseErase) {
        d.idx = sl.scratch + scratch_off;
        scratch_off += o.n;
      } else {
        d.idx = o.buf_indices;
      }
      if (o.op == ASH_OP_INSERT && o.map->n_values == 1) {
        d.v.dst = o.map->vb[0];
        d.v.src = o.values;
        d.v.row_bytes = o.map->row_bytes[0];
        d.v.vec = static_cast<int>(o.map->row_bytes[0]);
      }
      tiles += (o.n + kBatchThreads - 1) / kBatchThreads;
      o.map->last_stream = st;
      if (ph == kPhaseInsert) {
        o.map->size_ub += o.n;
        o.map->used_ub += o.n;
        o.map->added_since_snap += o.n;
        note_insert_stream(o.map, st);
      }
    }
    tb->ph[ph].count = k - tb->ph[ph].first;
    tb->ph[ph].tiles = tiles;
  }
  tb->n_ops = k;
  bool wide = false;
  for (int i = 0; i < k; ++i) wide |= tb->ops[i].S != 4;
  // ---- the snapshots that the maps ask for, published by the batch's last kernel
  std::vector<ash_map*> snapped;
  tb->n_snaps = 0;
  for (int i = 0; i < n_ops; ++i)
    if (ops[i].op == ASH_OP_ERASE) ops[i].map->erased_since_snap += ops[i].n;
  for (int i = 0; i < n_ops; ++i) {
    ash_map* m = ops[i].map;
    if (ops[i].op == ASH_OP_FIND || std::find(snapped.begin(), snapped.end(), m) != snapped.end()) continue;
    if (!snapshot_wanted(m, st, 0)) continue;
    snapped.push_back(m);
    tb->snaps[tb->n_snaps++] = {m->ctrl, m->snap_dev, m->snap_seq};
  }
  // What the batch does to the maps' invariants holds from its first launch on,
  // also when a later one is refused.
  for (int i = 0; i < n_ops; ++i)
    if (ops[i].op == ASH_OP_INSERT || ops[i].op == ASH_OP_ACTIVATE) ops[i].map->pref_placed = false;  // keys placed in slot order
    else if (ops[i].op == ASH_OP_ERASE) ops[i].map->heap_identity = false;
  ash_status s = ASH_OK;
  if (k > 0 || tb->n_snaps > 0) {  // snapshots that were numbered have to be published, work or not
    TraceScope ts(kKBatch, st, batch_launches(*tb));
    if (wide) launch_batch<true>(b, sl, st);
    else launch_batch<false>(b, sl, st);
    s = check_launch("batch_run");
  }
  // the upload reads the slot's table until then, whatever followed it
  if (cudaEventRecord(sl.done, st) != cudaSuccess) return cuda_fail(cudaGetLastError(), "cudaEventRecord");
  sl.used = true;
  if (s != ASH_OK) return s;
  for (ash_map* m : snapped) snapshot_issued(m);
  return ASH_OK;
}

}  // extern "C"
