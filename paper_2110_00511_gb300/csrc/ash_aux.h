// Host-side launchers of the dimension-independent kernels (ash_aux.cu).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "ash_device.cuh"

namespace ash {

struct Launch;

// Lists live buffer indices in ascending order (the complement of the free
// part of the heap).  scratch: list_scratch_bytes(capacity) bytes of device
// memory.  Writes at most out_cap indices; the live count goes to ctrl->count.
int64_t list_scratch_bytes(int64_t capacity);
// count_out (optional): device int64 receiving the live count.  The scratch
// bitmap must be zero on entry; the listing leaves it zero.  heap_identity:
// the heap's free part is h[j] = j (no erase since create, clear or a
// compacting rehash), so the live indices are 0..t-1 and are written directly.
void launch_list_active(bool heap_identity, const int32_t* heap, int64_t capacity, Ctrl* ctrl, void* scratch,
                        int32_t* out, int64_t out_cap, long long* count_out, const Launch& L);
// Byte ranges of a map's storage that one kernel fills or copies together:
// what create, clear and a rebuild have to lay down (table EMPTY, value rows
// zero, the heap's identity, buffers moved to larger ones, counters).
struct InitSeg {
  char* dst;
  const char* src;   // kCopy: source (any alignment; 16-byte alike is fast)
  uint64_t word;     // kWord: the 8-byte value; kIota: the first int32
  int64_t bytes;
  int64_t chunks;
  int32_t kind;
};

struct InitPlan {
  enum { kZero = 0, kOnes, kCopy, kIota, kWord };
  static constexpr int kMax = 24;  // table, kB, heap (2), 8 value buffers (2 each), counters, flags
  static constexpr int64_t kChunk = 16384;
  int n = 0;
  InitSeg seg[kMax];
  void add(int kind, void* dst, const void* src, uint64_t word, int64_t bytes) {
    if (bytes <= 0) return;
    seg[n++] = {static_cast<char*>(dst), static_cast<const char*>(src), word, bytes, (bytes + kChunk - 1) / kChunk, kind};
  }
  void zero(void* dst, int64_t bytes) { add(kZero, dst, nullptr, 0, bytes); }
  void ones(void* dst, int64_t bytes) { add(kOnes, dst, nullptr, 0, bytes); }
  void copy(void* dst, const void* src, int64_t bytes) { add(kCopy, dst, src, 0, bytes); }
  // h[i] = i for i in [from, to)
  void iota(int32_t* h, int64_t from, int64_t to) {
    add(kIota, h + from, nullptr, static_cast<uint64_t>(from), (to - from) * 4);
  }
  void word(void* dst, uint64_t v) { add(kWord, dst, nullptr, v, 8); }
};
void launch_init(const InitPlan& plan, const Launch& L);
// Copies the control block to its pinned mirror.
void launch_read_ctrl(const Ctrl* ctrl, Ctrl* host, const Launch& L);
// Publishes the control block to a host-visible snapshot (publish_snapshot).
void launch_snapshot(Ctrl* ctrl, Snap* snap, uint32_t seq, const Launch& L);
// Value rows of an insert's winners (idx[p] >= 0): dst_j row idx[p] <- src_j row p.
void launch_scatter_rows(const ValueCopy& vc, const int32_t* idx, int64_t n, const Launch& L);
// dst_j row r <- src_j row list[r] for every value buffer (compacting rehash;
// the list's indices lie below the source buffers' capacity).
void launch_gather_rows(const ValueCopy& vc, int64_t capacity, const int32_t* list, int64_t n, const Launch& L);
void launch_gather_keys(const int32_t* kb, int ks, int d, int64_t capacity, const int32_t* indices, int64_t n,
                        const long long* n_dev, int32_t* out, const Launch& L);
void launch_gather_values(const void* src, int64_t row_bytes, int vec, int64_t capacity, const int32_t* indices,
                          int64_t n, const long long* n_dev, void* out, const Launch& L);
void launch_quantize(const float* pts, int64_t n, float cell, int32_t* keys, const Launch& L);
void launch_probe_atomic(void* buf, int64_t buf_bytes, int64_t n_ops, int mode, uint32_t seed, uint32_t* sink,
                         int64_t sink_len, const Launch& L);
void launch_probe(const void* buf, int64_t buf_bytes, int64_t n_reads, int sector, int loads_per_thread,
                  uint32_t seed, uint32_t* sink, int64_t sink_len, const Launch& L);

}  // namespace ash
