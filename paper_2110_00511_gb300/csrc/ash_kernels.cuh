// Hash map kernels, templated on the key dimension D and the bucket size S.
//
// find            KPT query keys per thread: hash, load the home buckets of all
//                 KPT keys back to back, verify the fingerprint match of each
//                 against kB (Eq. (4)); keys that their home bucket does not
//                 settle go on from the next one (find_keys).
// insert/activate two kernels (Sec. 4.3.1 lazy insertion, redesigned):
//   claim         a key already committed is rejected.  Otherwise the thread
//                 claims an EMPTY slot with a CAS writing {fingerprint,
//                 kClaimBit | input position}: either the key's preferred
//                 slot of its home bucket, CASed with no load before it
//                 (claim_pref_kernel, while the table fits in L2; keys that
//                 find it taken are queued per warp and claimed from their
//                 buckets in dense rounds), or the first EMPTY slot of the
//                 loaded home bucket (claim_bucket_kernel).  A key whose home
//                 bucket is full walks its chain (claim_key) and may take a
//                 tombstone on it.  A thread that
//                 meets a claimed slot compares its key with the READ-ONLY
//                 input row of the claimant (never with a half-written kB
//                 row, which removes the torn-copy race of Sec. 4.4.2) and,
//                 if equal, lowers the recorded position with atomicMin,
//                 marking the position it displaced in the winner flags.
//                 After the kernel each claimed slot names the lowest input
//                 position of its key.  The slot index goes to
//                 buf_indices[p] as scratch.
//   commit        one thread per input key: a position holding a slot index
//                 whose winner flag is clear wins, takes a buffer index from
//                 the heap (one atomicAdd per block on t, Sec. 4.3), writes
//                 kB(i) and small value rows, then replaces the claim with
//                 {fingerprint, i}.  Only winners allocate ("allocate only on
//                 success", Sec. 4.3.1).
// erase           two kernels: mark (atomicMin of the input position into the
//                 slot's high word, keeping the buffer index) and resolve (the
//                 lowest position wins, frees the index with one atomic per
//                 block, and empties the slot, or leaves a tombstone when a
//                 probe chain may pass its bucket or, under the preferred-
//                 slot invariant, another live key prefers it).  Allocation and
//                 free never run in the same kernel (the atomicAdd/atomicSub
//                 conflict that Sec. 4.3.1 warns about).
// rebuild         inserts already-unique keys (rehash, Sec. 4.5) into an empty
//                 table: the preferred slot first, else the first EMPTY slot
//                 of the probe sequence, no key comparisons.
#pragma once

#include <atomic>
#include <type_traits>

#include "ash_device.cuh"
#include "ash_trace.h"

namespace ash {

// ---------------------------------------------------------------------- find
// Scalar lookup of key k from its home bucket.
template <int D, int S>
__device__ __forceinline__ int32_t find_key(const TableView& t, const int32_t (&k)[D]) {
  const uint64_t h = hash_key<D>(k);
  const uint32_t fp = fingerprint(h);
  uint32_t b = home_bucket(h, t.n_buckets);
  for (uint32_t probe = 0; probe < t.max_probes; ++probe) {
    uint64_t w[S];
    load_bucket<S, true>(t.slots + static_cast<size_t>(b) * S, w);
    bool stop = false;
    int32_t out = -1;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      stop |= (w[s] == kEmpty);
      if (out < 0 && hi32(w[s]) == fp && lo32(w[s]) < kClaimBit && kb_equal<D>(t.kb, lo32(w[s]), k))
        out = static_cast<int32_t>(lo32(w[s]));
    }
    if (out >= 0) return out;
    if (stop) return -1;
    b = next_bucket(b, t.n_buckets);
  }
  return -1;
}

// The same out of line, for find_keys when a fingerprint match is not the key.
template <int D>
struct KeyOf {
  int32_t v[D];
};

template <int D, int S>
__device__ __noinline__ int32_t find_slow(const TableView t, const KeyOf<D> k) {
  return find_key<D, S>(t, k.v);
}

// One probe round of KPT keys: the buckets b[q] of the keys still searched
// (go[q]) are loaded together, then the verify loads of their first
// fingerprint matches, then everything is compared.  Settled keys leave go;
// a match that is another key, or one of several, raises rare.
template <int D, int S, int KPT, bool ALL>
__device__ __forceinline__ void probe_round(const TableView& t, const int32_t (&k)[KPT][D], const uint32_t (&fp)[KPT],
                                            const uint32_t (&b)[KPT], bool (&go)[KPT], int32_t (&out)[KPT],
                                            bool& rare) {
  constexpr int KS = KeyStride<D>::value;
  uint64_t w[KPT][S];
#pragma unroll
  for (int q = 0; q < KPT; ++q)
    if (ALL || go[q]) load_bucket<S, true>(t.slots + static_cast<size_t>(b[q]) * S, w[q]);
  uint32_t cand[KPT];
  int ncand[KPT];
  bool stop[KPT];
#pragma unroll
  for (int q = 0; q < KPT; ++q) {
    cand[q] = kNoIndex;
    ncand[q] = 0;
    stop[q] = false;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      stop[q] |= (w[q][s] == kEmpty);
      const bool m = hi32(w[q][s]) == fp[q] && lo32(w[q][s]) < kClaimBit;
      if (m && ncand[q] == 0) cand[q] = lo32(w[q][s]);
      ncand[q] += m ? 1 : 0;
    }
    if (!ALL && !go[q]) ncand[q] = 0;
  }
  int32_t row[KPT][KS];
#pragma unroll
  for (int q = 0; q < KPT; ++q) {
    if (ncand[q] > 0) {
      load_kb<D>(t.kb, cand[q], row[q]);
    } else {
#pragma unroll
      for (int j = 0; j < KS; ++j) row[q][j] = 0;
    }
  }
#pragma unroll
  for (int q = 0; q < KPT; ++q) {
    bool eq = ncand[q] > 0;
#pragma unroll
    for (int j = 0; j < D; ++j) eq &= (row[q][j] == k[q][j]);
    if (eq) out[q] = static_cast<int32_t>(cand[q]);
    rare |= go[q] && ncand[q] > 0 && !eq;
    go[q] &= !eq && !stop[q];
  }
}

// Looks KPT keys up together (ok[q] false: a key that nobody asked for; its
// bucket is loaded, in bounds, and its result unused).  At the usual load of
// one half, about one home bucket in six is full without the key, so nearly
// every warp has lanes that probe on: they go on from the next bucket, with
// hash and key in registers.  Searching such a key again from its home
// bucket in an out-of-line loop instead made the 27-neighbourhood kernel
// issue 495 instructions per warp and query at 12 active lanes of 32 (now
// 270 at 19).  GB300: 6M finds, half absent, on 5M entries 161 -> 127 us; 4M
// finds, all present, 72 -> 61 us.
//
// With several keys per lane only the home buckets are probed together.  A
// second probe_round over all of them cost their registers twice over (3-D, 16
// slots, two keys: 128 instead of 64): 8M finds, half absent, of two keys per
// lane in 16-slot buckets 221 us, now 174 (178 before the lookups went on in
// place); of four keys 244, now 183; 8-D, 16 slots, two keys 334, now 221.
template <int D, int S, int KPT>
__device__ __forceinline__ void find_keys(const TableView& t, const int32_t (&k)[KPT][D], const bool (&ok)[KPT],
                                          int32_t (&out)[KPT]) {
  uint32_t fp[KPT], b[KPT];
  bool go[KPT];
  bool rare = false;
#pragma unroll
  for (int q = 0; q < KPT; ++q) {
    const uint64_t h = hash_key<D>(k[q]);
    fp[q] = fingerprint(h);
    b[q] = home_bucket(h, t.n_buckets);
    go[q] = ok[q];
    out[q] = -1;
  }
  probe_round<D, S, KPT, true>(t, k, fp, b, go, out, rare);
  if constexpr (KPT == 1) {
    for (uint32_t probe = 1; probe < t.max_probes && go[0]; ++probe) {
      b[0] = next_bucket(b[0], t.n_buckets);
      probe_round<D, S, 1, false>(t, k, fp, b, go, out, rare);
    }
  } else {
    // a lane's unsettled keys one after the other, in one piece of code
    while (true) {
      int at = -1;
#pragma unroll
      for (int q = KPT - 1; q >= 0; --q) at = go[q] ? q : at;
      if (at < 0) break;
      int32_t k1[1][D], out1[1] = {-1};
      uint32_t fp1[1] = {0u}, b1[1] = {0u};
      bool go1[1] = {true};
#pragma unroll
      for (int q = 0; q < KPT; ++q) {
        if (q == at) {
#pragma unroll
          for (int j = 0; j < D; ++j) k1[0][j] = k[q][j];
          fp1[0] = fp[q];
          b1[0] = b[q];
          go[q] = false;
        }
      }
#pragma unroll 1
      for (uint32_t probe = 1; probe < t.max_probes && go1[0]; ++probe) {
        b1[0] = next_bucket(b1[0], t.n_buckets);
        probe_round<D, S, 1, false>(t, k1, fp1, b1, go1, out1, rare);
      }
#pragma unroll
      for (int q = 0; q < KPT; ++q)
        if (q == at) out[q] = out1[0];
    }
  }
  if (rare) {
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      if (ok[q] && out[q] < 0) {
        KeyOf<D> key;
#pragma unroll
        for (int j = 0; j < D; ++j) key.v[j] = k[q][j];
        out[q] = find_slow<D, S>(t, key);
      }
    }
  }
}

// A warp's keys that their home bucket did not settle, in shared memory: they
// probe on 32 at a time, so that the rounds past the home bucket run on full
// warps.  Entry: key, fingerprint, the bucket looked at last, how many buckets
// that makes, and the output row.  Every lane of the warp calls push and
// round.
template <int D>
struct ProbeList {
  static constexpr int kCap = 64;  // fewer than 32 before a push of up to 32
  struct Store {
    int64_t row[kCap];
    int32_t key[D][kCap];
    uint32_t fp[kCap], bucket[kCap], probes[kCap];
  };
  Store& s;
  int n = 0;  // warp-uniform
  __device__ explicit ProbeList(Store& store) : s(store) {}

  __device__ __forceinline__ void push(bool mine, const int32_t (&k)[D], uint32_t fp, uint32_t b, uint32_t probes,
                                       int64_t row) {
    const unsigned bal = __ballot_sync(0xFFFFFFFFu, mine);
    if (mine) {
      const int at = n + __popc(bal & ((1u << (threadIdx.x & 31)) - 1u));
      s.row[at] = row;
#pragma unroll
      for (int j = 0; j < D; ++j) s.key[j][at] = k[j];
      s.fp[at] = fp;
      s.bucket[at] = b;
      s.probes[at] = probes;
    }
    n += __popc(bal);
    __syncwarp();
  }

  // The next bucket of up to 32 entries; those that it does not settle are
  // pushed again.
  template <int S>
  __device__ __forceinline__ void round(const TableView& t, int32_t* __restrict__ idx, uint8_t* __restrict__ mask) {
    const int lane = threadIdx.x & 31;
    const int from = n > 32 ? n - 32 : 0;
    const bool v = from + lane < n;
    const int at = v ? from + lane : 0;
    int32_t k[1][D];
#pragma unroll
    for (int j = 0; j < D; ++j) k[0][j] = s.key[j][at];
    const uint32_t fp[1] = {s.fp[at]};
    const uint32_t b[1] = {next_bucket(s.bucket[at], t.n_buckets)};
    const uint32_t probes = s.probes[at] + 1;
    const int64_t row = s.row[at];
    __syncwarp();
    n = from;
    bool go[1] = {v && probes <= t.max_probes};
    int32_t out[1] = {-1};
    bool rare = false;
    probe_round<D, S, 1, false>(t, k, fp, b, go, out, rare);
    if (rare && out[0] < 0) {
      KeyOf<D> key;
#pragma unroll
      for (int j = 0; j < D; ++j) key.v[j] = k[0][j];
      out[0] = find_slow<D, S>(t, key);
      go[0] = false;
    }
    if (v && !go[0]) {
      idx[row] = out[0];
      mask[row] = out[0] >= 0 ? 1 : 0;
    }
    push(go[0], k[0], fp[0], b[0], probes, row);
  }
};

// Looks up KPT keys of each lane (ok[q]: wanted; row[q]: their output rows),
// writing what their home buckets settle and listing the rest.  For kernels
// bound by issue; the plain find, bound by random sectors, is the faster the
// more warps it has and keeps find_keys (with the list, at 48 registers, 4M
// finds took 78 us against 61, 6M on 80 MB of table 150 against 127).
template <int D, int S, int KPT>
__device__ __forceinline__ void find_or_list(const TableView& t, const int32_t (&k)[KPT][D], const bool (&ok)[KPT],
                                             const int64_t (&row)[KPT], ProbeList<D>& list, int32_t* __restrict__ idx,
                                             uint8_t* __restrict__ mask) {
  uint32_t fp[KPT], b[KPT];
  int32_t out[KPT];
  bool go[KPT];
  bool rare = false;
#pragma unroll
  for (int q = 0; q < KPT; ++q) {
    const uint64_t h = hash_key<D>(k[q]);
    fp[q] = fingerprint(h);
    b[q] = home_bucket(h, t.n_buckets);
    go[q] = ok[q];
    out[q] = -1;
  }
  probe_round<D, S, KPT, true>(t, k, fp, b, go, out, rare);
  if (rare) {
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      if (ok[q] && out[q] < 0) {
        KeyOf<D> key;
#pragma unroll
        for (int j = 0; j < D; ++j) key.v[j] = k[q][j];
        out[q] = find_slow<D, S>(t, key);
        go[q] = false;
      }
    }
  }
#pragma unroll
  for (int q = 0; q < KPT; ++q) {
    if (ok[q] && !go[q]) {
      idx[row[q]] = out[q];
      mask[row[q]] = out[q] >= 0 ? 1 : 0;
    }
    list.push(go[q], k[q], fp[q], b[q], 1u, row[q]);
    while (list.n >= 32) list.template round<S>(t, idx, mask);
  }
}

// Offsets of a neighbour query.  RadiusOffsets: [-radius, radius]^D row-major
// (the last coordinate fastest), digit by digit of the offset's number in
// base width = 2 radius + 1; the division by width is a multiplication by
// magic = ceil(2^32 / width), exact for the offset numbers allowed (below
// 2^20, with width <= 17), and 0 for width 1, whose only number is 0.
struct RadiusOffsets {
  uint32_t radius, width, magic;
  template <int D>
  __device__ __forceinline__ void add(uint32_t o, int32_t (&k)[D]) const {
#pragma unroll
    for (int j = D - 1; j >= 0; --j) {
      const uint32_t q = __umulhi(o, magic);
      k[j] = static_cast<int32_t>(static_cast<uint32_t>(k[j]) + (o - q * width) - radius);
      o = q;
    }
  }
};

// TableOffsets: an explicit [n_off, D] int32 table in device memory.
struct TableOffsets {
  const int32_t* __restrict__ table;
  template <int D>
  __device__ __forceinline__ void add(uint32_t o, int32_t (&k)[D]) const {
#pragma unroll
    for (int j = 0; j < D; ++j)
      k[j] = static_cast<int32_t>(static_cast<uint32_t>(k[j]) + static_cast<uint32_t>(__ldg(table + o * D + j)));
  }
};

// GB300, 200k keys x 27 offsets over a table in L2 (5.4M queries), bound by
// instruction issue: 110 -> 70 us with the keys that their home bucket does
// not settle probing on in place, -> 51 us with those in a list per warp
// (ProbeList) on a grid of the blocks that fit at once (54 on 8 per SM).  One
// pair per thread: two 4 us slower, four 32 us (before the list); held to 48
// or fewer registers for more warps, 64-80 us.  L1 allocation of the buckets
// that neighbouring queries share gained 1 %, so they bypass it.
constexpr int kNeighborUnroll = 1;

// Neighbour query (the radius search and the neighbour tables of Sec.
// 6.2-6.4): the n x n_off (query, offset) pairs flattened, outputs [n, n_off].
// Offsets are added with int32 wrap-around; the query keys are never
// materialised.  Blocks take tiles of U * blockDim consecutive pairs, U per
// thread, so the key rows of a tile come from L1 and the outputs are
// coalesced; a thread's (query, offset) moves by two constant strides, so
// the only divisions are at its start.
template <int D, int S, int U, class Off>
__global__ void __launch_bounds__(256) neighbors_kernel(TableView t, const int32_t* __restrict__ keys, int64_t n,
                                                        const Off off, uint32_t n_off, int32_t* __restrict__ idx,
                                                        uint8_t* __restrict__ mask) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t total = n * n_off;
  const int64_t tile = static_cast<int64_t>(blockDim.x) * U;
  const int64_t jump = (gridDim.x - 1) * tile;
  const int64_t first = static_cast<int64_t>(blockIdx.x) * tile + threadIdx.x;
  const uint32_t step_r = blockDim.x / n_off, step_o = blockDim.x - step_r * n_off;
  const int64_t jump_r = jump / n_off;
  const uint32_t jump_o = static_cast<uint32_t>(jump - jump_r * n_off);
  int64_t r = first / n_off;
  uint32_t o = static_cast<uint32_t>(first - r * n_off);
  __shared__ typename ProbeList<D>::Store s_list[8];
  ProbeList<D> list(s_list[threadIdx.x >> 5]);
  const int lane = threadIdx.x & 31;
  for (int64_t e = first; e - lane < total; e += gridDim.x * tile) {
    int32_t k[U][D];
    bool ok[U];
    int64_t row[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      row[u] = e + u * blockDim.x;
      ok[u] = row[u] < total;
      if (ok[u]) {
        load_input_key<D>(keys, r, k[u]);
        off.add(o, k[u]);
      } else {
#pragma unroll
        for (int j = 0; j < D; ++j) k[u][j] = 0;
      }
      r += step_r;
      o += step_o;
      if (o >= n_off) {
        o -= n_off;
        ++r;
      }
    }
    find_or_list<D, S, U>(t, k, ok, row, list, idx, mask);
    r += jump_r;
    o += jump_o;
    if (o >= n_off) {
      o -= n_off;
      ++r;
    }
  }
  while (list.n > 0) list.template round<S>(t, idx, mask);
}

// Resident blocks that the find is compiled for, 0 where the compiler's own
// choice is the best.  One key of a 16-slot bucket: left alone it keeps 36
// registers and loads the bucket piece by piece (8M finds, half absent, 3-D
// 223 us, 1-D 191), at four blocks the bucket's loads are in flight together
// (184 and 155); at five 199 and 174.  The rest gives the register counts at
// which the options with more keys per thread ran before the lookups went on
// in place (8-D, 8 slots, four keys stay slower, 229 against 206 us).
template <int D, int S, int KPT>
constexpr int find_min_blocks() {
  if (KPT == 1) return S == 16 ? 4 : 0;
  if (KPT == 2) return D == 1 ? 4 : (S == 16 && D > 6 ? 3 : 0);
  return D == 8 ? 2 : 0;
}

// KPT keys per thread: positions base, base + blockDim.x, ... so every load
// instruction stays coalesced across the warp.
template <int D, int S, int KPT, class In = const int32_t*>
__global__ void __launch_bounds__(256, find_min_blocks<D, S, KPT>()) find_kernel(TableView t, const In keys, int64_t n,
                                                   int32_t* __restrict__ idx, uint8_t* __restrict__ mask) {
  // a programmatic dependent of the previous kernel: wait for its grid (a no-op otherwise)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t step = static_cast<int64_t>(gridDim.x) * blockDim.x * KPT;
  for (int64_t base = static_cast<int64_t>(blockIdx.x) * blockDim.x * KPT + threadIdx.x; base < n; base += step) {
    int32_t k[KPT][D], out[KPT];
    bool ok[KPT];
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      const int64_t pos = base + static_cast<int64_t>(q) * blockDim.x;
      ok[q] = pos < n;
      if (ok[q]) {
        load_input_key<D>(keys, pos, k[q]);
      } else {
#pragma unroll
        for (int j = 0; j < D; ++j) k[q][j] = 0;
      }
    }
    find_keys<D, S, KPT>(t, k, ok, out);
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      const int64_t pos = base + static_cast<int64_t>(q) * blockDim.x;
      if (ok[q]) {
        idx[pos] = out[q];
        mask[pos] = out[q] >= 0 ? 1 : 0;
      }
    }
  }
}

// find, and the index found for row r goes to link[link_at[r]] as well.
template <int D, int S>
__global__ void __launch_bounds__(256) find_link_kernel(TableView t, const int32_t* __restrict__ keys, int64_t n,
                                                        int32_t* __restrict__ idx, int32_t* __restrict__ link,
                                                        const int32_t* __restrict__ link_at) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t step = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t r = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; r < n; r += step) {
    int32_t k[1][D], out[1];
    const bool ok[1] = {true};
    load_input_key<D>(keys, r, k[0]);
    const int32_t at = __ldg(link_at + r);
    find_keys<D, S, 1>(t, k, ok, out);
    idx[r] = out[0];
    link[at] = out[0];
  }
}

// Warp-cooperative find: a group of G = S / 2 lanes takes one key, each lane
// loading two slots (one 16-byte load; the group reads the whole bucket in one
// coalesced request), so a warp has 32 / G keys in flight.  Fingerprint
// matches are verified by the lane that holds them with one 128-bit kB load;
// the group agrees through __ballot_sync and the result comes from the
// lowest verified lane (__shfl_sync).  Probing continues while no lane saw an
// EMPTY slot.  Groups of one warp proceed together (warp-wide ballots), a
// finished group voting false.  The alternative to find_kernel's thread per
// key; the tuning's warp_probe picks one.
template <int D, int S>
__global__ void __launch_bounds__(256) find_group_kernel(TableView t, const int32_t* __restrict__ keys, int64_t n,
                                                         int32_t* __restrict__ idx, uint8_t* __restrict__ mask) {
  constexpr int G = S / 2;
  constexpr int KEYS_PER_WARP = 32 / G;
  constexpr uint32_t kGroupBits = (G == 32) ? 0xFFFFFFFFu : ((1u << G) - 1u);
  const int lane = threadIdx.x & 31;
  const int sub = lane % G;               // lane within the group
  const int grp = lane / G;               // group within the warp
  const uint32_t gshift = static_cast<uint32_t>(grp * G);
  const int64_t warp_global = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int64_t n_warps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
  for (int64_t base = warp_global * KEYS_PER_WARP; base < n; base += n_warps * KEYS_PER_WARP) {
    const int64_t pos = base + grp;
    bool active = pos < n;
    int32_t k[D];
    if (active) {
      load_input_key<D>(keys, pos, k);
    } else {
#pragma unroll
      for (int j = 0; j < D; ++j) k[j] = 0;
    }
    const uint64_t h = hash_key<D>(k);
    const uint32_t fp = fingerprint(h);
    uint32_t b = home_bucket(h, t.n_buckets);
    int32_t out = -1;
    for (uint32_t probe = 0; probe < t.max_probes; ++probe) {
      const bool live = active;
      bool found = false, empty = false;
      uint32_t my = kNoIndex;
      if (live) {
        const ulonglong2 w = __ldg(reinterpret_cast<const ulonglong2*>(t.slots + static_cast<size_t>(b) * S) + sub);
        empty = (w.x == kEmpty) || (w.y == kEmpty);
        const bool m0 = hi32(w.x) == fp && lo32(w.x) < kClaimBit;
        const bool m1 = hi32(w.y) == fp && lo32(w.y) < kClaimBit;
        if (m0 && kb_equal<D>(t.kb, lo32(w.x), k)) my = lo32(w.x);
        else if (m1 && kb_equal<D>(t.kb, lo32(w.y), k)) my = lo32(w.y);
        found = my != kNoIndex;
      }
      const uint32_t fb = (__ballot_sync(0xFFFFFFFFu, found) >> gshift) & kGroupBits;
      const uint32_t eb = (__ballot_sync(0xFFFFFFFFu, empty) >> gshift) & kGroupBits;
      const int src = fb ? static_cast<int>(gshift) + __ffs(fb) - 1 : lane;
      const uint32_t hit = __shfl_sync(0xFFFFFFFFu, my, src);
      if (live) {
        if (fb) {
          out = static_cast<int32_t>(hit);
          active = false;
        } else if (eb) {
          active = false;
        } else {
          b = next_bucket(b, t.n_buckets);
        }
      }
      if (!__any_sync(0xFFFFFFFFu, active)) break;
    }
    if (pos < n && sub == 0) {
      idx[pos] = out;
      mask[pos] = out >= 0 ? 1 : 0;
    }
  }
}

// ------------------------------------------------------------- insert: claim
// Result codes written to buf_indices[p] by the claim kernel.
constexpr int32_t kClaimExists = -2;  // key already committed
constexpr int32_t kClaimJoined = -3;  // an equal key of this batch with a lower position holds the claim
constexpr int32_t kClaimFailed = -1;  // no slot within max_probes

// 0: no match.  1: slot claimed by an equal key in this batch.  2: committed equal key.
template <int D, class In>
__device__ __forceinline__ int claim_match(uint64_t w, uint32_t fp, const int32_t (&k)[D], const In& keys,
                                           const int32_t* kb) {
  const uint32_t lo = lo32(w);
  if (lo == kNoIndex || hi32(w) != fp) return 0;
  if (lo & kClaimBit) return input_key_equal<D>(keys, lo & ~kClaimBit, k) ? 1 : 0;
  return kb_equal<D>(kb, lo, k) ? 2 : 0;
}

// This position meets an equal key's claim, with position seen_lo, at slot p:
// the lower position keeps the claim (atomicMin on the word, whose high half
// is the shared fingerprint).  Returns false when this position lost for
// sure (a lower one holds the claim); true when it holds the claim for now.
// With winner flags (FLAGS and t.lost) the position it displaced is marked
// lost.
template <bool FLAGS = true>
__device__ __forceinline__ bool join_claim(const TableView& t, uint64_t* p, uint32_t seen_lo, uint64_t mine,
                                           uint32_t pos) {
  if (!FLAGS) {
    // no winner flags: the commit reads the slot word to see who won
    if ((seen_lo & ~kClaimBit) > pos)
      atomicMin(reinterpret_cast<unsigned long long*>(p), static_cast<unsigned long long>(mine));
    return true;
  }
  if ((seen_lo & ~kClaimBit) < pos) return false;
  if (!t.lost) {
    atomicMin(reinterpret_cast<unsigned long long*>(p), static_cast<unsigned long long>(mine));
    return true;
  }
  const uint64_t old = atomicMin(reinterpret_cast<unsigned long long*>(p), static_cast<unsigned long long>(mine));
  const uint32_t op = lo32(old) & ~kClaimBit;
  if (op < pos) return false;
  atomicOr(t.lost + (op >> 5), 1u << (op & 31));
  return true;
}

// Order in which a claim takes the EMPTY slots of a bucket (claim_key):
//   kClaimSlotOrder  slot order, used out of line as a slow path
//   kClaimSlotMask   slot order, one compare site for all slots (a loop over
//                    the matches): fewer registers, for the batched kernel
//                    that inlines the protocol for every key dimension and
//                    runs it on full warps (claims of 24 maps 32 -> 28 us;
//                    out of line in claim_bucket_kernel the same compares
//                    made 10^8 ranged keys 5 % slower)
//   kClaimPrefFirst  the key's preferred slot first in its home bucket, then
//                    slot order (keeps the preferred-slot invariant)
constexpr int kClaimSlotOrder = 0;
constexpr int kClaimSlotMask = 1;
constexpr int kClaimPrefFirst = 2;

// The full claim protocol for one key, a walk from its home bucket: 1) any
// slot holding an equal key ends the search; 2) the walk ends at the first
// bucket with an EMPTY slot, where the key is known to be absent; 3) the key
// takes the first TOMBSTONE of the buckets without an EMPTY slot that it
// walked past, else an EMPTY slot of the last bucket.  A lost CAS compares
// with the winner's word and starts the walk again.  A walk that meets no
// EMPTY slot within max_probes buckets fails even past a tombstone: when
// max_probes was lowered on a filled map, the key may sit further along.
//
// Equal keys of one batch cannot take two slots.  A slot only goes from free
// (EMPTY or TOMBSTONE, and of one kind while it is free) to taken during an
// insert, and every path prefers free slots in one order: by bucket along the
// chain, within a bucket EMPTY before TOMBSTONE, then by position.  Had two
// equal keys taken slots x and then y, both slots were free in both walks
// (the second walk passed x before it was taken, else it would have met the
// equal key there; y was free until taken last), and the walks preferred
// them differently.
//
// Reusing tombstones keeps the runs of full buckets from growing: a run of
// length L collects the keys that hash into it, and when these could only be
// placed past its end, every insert / erase cycle of a sliding window left
// the run longer by a share of L, until the tombstone count called for a
// rebuild.  GB300: a window of 262k keys over 1M entries 101 -> 69 us a pass
// (no rebuild in 1200 passes, 19 before), 24 maps in one batch 514 -> 118 us.
//
// FLAGS: winner flags may be set (t.lost); the batched kernel, which has
// none, compiles without them.
template <int D, int S, class In, int ORDER, bool FLAGS = true>
__device__ __forceinline__ int32_t claim_key(const TableView& t, const In& keys, int64_t pos) {
  int32_t k[D];
  load_input_key<D>(keys, pos, k);
  const uint64_t h = hash_key<D>(k);
  const uint32_t fp = fingerprint(h);
  const uint64_t mine = (static_cast<uint64_t>(fp) << 32) | (kClaimBit | static_cast<uint32_t>(pos));
  const uint32_t home = home_bucket(h, t.n_buckets);
  uint32_t b = home;
  uint32_t tomb = kNoIndex;  // first tombstone passed, as a slot index
  for (uint32_t probe = 0; probe < t.max_probes;) {
    uint64_t* bp = t.slots + static_cast<size_t>(b) * S;
    uint64_t w[S];
    load_bucket<S, false>(bp, w);
    if constexpr (ORDER == kClaimSlotMask) {
      // the first fingerprint match is picked before anything is compared, so
      // the lanes of a warp wait for one compare, not for one per slot
      int at = -1, matches = 0;
      uint64_t seen = 0;
#pragma unroll
      for (int s = S - 1; s >= 0; --s) {
        if (lo32(w[s]) != kNoIndex && hi32(w[s]) == fp) {
          at = s;
          seen = w[s];
          ++matches;
        }
      }
      while (matches > 0) {
        const int m = claim_match<D, In>(seen, fp, k, keys, t.kb);
        if (m == 2) return kClaimExists;
        if (m == 1)
          return join_claim<FLAGS>(t, bp + at, lo32(seen), mine, static_cast<uint32_t>(pos)) ? static_cast<int32_t>(b * S + at)
                                                                                      : kClaimJoined;
        if (--matches == 0) break;
        const int after = at;  // another key with this fingerprint: the next match
#pragma unroll
        for (int s = S - 1; s >= 0; --s) {
          if (s > after && lo32(w[s]) != kNoIndex && hi32(w[s]) == fp) {
            at = s;
            seen = w[s];
          }
        }
      }
    } else {
#pragma unroll
      for (int s = 0; s < S; ++s) {
        const int m = claim_match<D, In>(w[s], fp, k, keys, t.kb);
        if (m == 2) return kClaimExists;
        if (m == 1)
          return join_claim<FLAGS>(t, bp + s, lo32(w[s]), mine, static_cast<uint32_t>(pos)) ? static_cast<int32_t>(b * S + s)
                                                                                      : kClaimJoined;
      }
    }
    uint32_t empty = 0, tombs = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      empty |= (w[s] == kEmpty ? 1u : 0u) << s;
      tombs |= (w[s] == kTombstone ? 1u : 0u) << s;
    }
    if (!empty) {
      if (tomb == kNoIndex && tombs) tomb = b * S + __ffs(tombs) - 1;
      b = next_bucket(b, t.n_buckets);
      ++probe;
      continue;
    }
    uint32_t slot = tomb;
    uint64_t free_word = kTombstone;
    if (tomb == kNoIndex) {
      const uint32_t pref = pref_slot<S>(fp);
      slot = b * S + (ORDER == kClaimPrefFirst && probe == 0 && ((empty >> pref) & 1u) ? pref : __ffs(empty) - 1);
      free_word = kEmpty;
    }
    const uint64_t old = atomicCAS(reinterpret_cast<unsigned long long*>(t.slots + slot),
                                   static_cast<unsigned long long>(free_word), static_cast<unsigned long long>(mine));
    if (old == free_word) {
      // the commit counts every winner's slot as newly used
      if (free_word == kTombstone) atomicAdd(&t.ctrl->top_used, 0ull - (1ull << 32));
      return static_cast<int32_t>(slot);
    }
    const int m = claim_match<D, In>(old, fp, k, keys, t.kb);
    if (m == 2) return kClaimExists;
    if (m == 1)
      return join_claim<FLAGS>(t, t.slots + slot, lo32(old), mine, static_cast<uint32_t>(pos)) ? static_cast<int32_t>(slot)
                                                                                        : kClaimJoined;
    b = home;  // another key was faster
    tomb = kNoIndex;
    probe = 0;
  }
  atomicOr(&t.ctrl->status, kStatusTableFull);
  return kClaimFailed;
}

// Out-of-line copy of the full protocol: the rare slow path of the claim
// kernels (kept out of line so it does not raise their register count).
template <int D, int S, class In, bool PrefFirst>
__device__ __noinline__ int32_t claim_one(const TableView t, const In keys, int64_t pos) {
  return claim_key<D, S, In, PrefFirst ? kClaimPrefFirst : kClaimSlotOrder>(t, keys, pos);
}

// Claim from the loaded home bucket, DK keys per lane (pos[q] valid where
// v[q]; an invalid lane hashes key 0 and loads that bucket, in bounds).  Per
// key: if the bucket holds exactly one slot with the key's fingerprint,
// compare once (claimant's input row or kB row); on no match, CAS the first
// EMPTY slot (PrefFirst: the preferred slot when it is EMPTY).  The loads,
// compares and CASes of the DK keys are issued back to back.  Anything else
// (several fingerprint matches, a lost CAS, a full bucket) is left to
// claim_one (slow[q]), which is safe because this path changed nothing then.
template <int D, int S, int DK, class In, bool PrefFirst>
__device__ __forceinline__ void claim_from_bucket(const TableView& t, const In& keys, const int64_t (&pos)[DK],
                                                  const bool (&v)[DK], int32_t* __restrict__ slot_out,
                                                  bool (&slow)[DK]) {
  constexpr int KS = KeyStride<D>::value;
  int32_t k[DK][D];
  uint32_t fp[DK], b[DK];
#pragma unroll
  for (int q = 0; q < DK; ++q) {
    if (v[q]) {
      load_input_key<D>(keys, pos[q], k[q]);
    } else {
#pragma unroll
      for (int j = 0; j < D; ++j) k[q][j] = 0;
    }
    const uint64_t h = hash_key<D>(k[q]);
    fp[q] = fingerprint(h);
    b[q] = home_bucket(h, t.n_buckets);
  }
  uint64_t w[DK][S];
#pragma unroll
  for (int q = 0; q < DK; ++q) load_bucket<S, false>(t.slots + static_cast<size_t>(b[q]) * S, w[q]);
  int cs[DK], nc[DK], es[DK];
  uint32_t clo[DK];
#pragma unroll
  for (int q = 0; q < DK; ++q) {
    cs[q] = -1;
    nc[q] = 0;
    es[q] = -1;
    clo[q] = kNoIndex;
    const uint32_t pref = pref_slot<S>(fp[q]);
    int pe = -1;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const bool m = lo32(w[q][s]) != kNoIndex && hi32(w[q][s]) == fp[q];
      if (m && nc[q] == 0) {
        cs[q] = s;
        clo[q] = lo32(w[q][s]);
      }
      nc[q] += m ? 1 : 0;
      if (es[q] < 0 && w[q][s] == kEmpty) es[q] = s;
      if (PrefFirst && static_cast<uint32_t>(s) == pref && w[q][s] == kEmpty) pe = s;
    }
    if (PrefFirst && pe >= 0) es[q] = pe;  // preferred slot first (preferred-slot invariant)
  }
  int32_t row[DK][KS];
#pragma unroll
  for (int q = 0; q < DK; ++q) {
    if (nc[q] > 0) {
      if (clo[q] & kClaimBit) {
        int32_t o[D];
        load_input_key<D>(keys, clo[q] & ~kClaimBit, o);
#pragma unroll
        for (int j = 0; j < KS; ++j) row[q][j] = j < D ? o[j] : 0;
      } else {
        load_kb<D>(t.kb, clo[q], row[q]);
      }
    } else {
#pragma unroll
      for (int j = 0; j < KS; ++j) row[q][j] = 0;
    }
  }
  int32_t res[DK];
  bool cas[DK];
#pragma unroll
  for (int q = 0; q < DK; ++q) {
    res[q] = kClaimFailed;
    cas[q] = false;
    slow[q] = false;
    if (v[q]) {
      bool eq = nc[q] > 0;
#pragma unroll
      for (int j = 0; j < D; ++j) eq &= (row[q][j] == k[q][j]);
      if (eq) {
        if (clo[q] & kClaimBit) {
          const uint64_t mine = (static_cast<uint64_t>(fp[q]) << 32) | (kClaimBit | static_cast<uint32_t>(pos[q]));
          res[q] = join_claim(t, t.slots + static_cast<size_t>(b[q]) * S + cs[q], clo[q], mine,
                              static_cast<uint32_t>(pos[q]))
                       ? static_cast<int32_t>(b[q] * S + cs[q])
                       : kClaimJoined;
        } else {
          res[q] = kClaimExists;
        }
      } else if (nc[q] > 1 || es[q] < 0) {
        slow[q] = true;
      } else {
        cas[q] = true;
      }
    }
  }
  uint64_t old[DK];
#pragma unroll
  for (int q = 0; q < DK; ++q) {
    old[q] = 0;
    if (cas[q]) {
      const uint64_t mine = (static_cast<uint64_t>(fp[q]) << 32) | (kClaimBit | static_cast<uint32_t>(pos[q]));
      old[q] = atomicCAS(reinterpret_cast<unsigned long long*>(t.slots + static_cast<size_t>(b[q]) * S + es[q]),
                         static_cast<unsigned long long>(kEmpty), static_cast<unsigned long long>(mine));
    }
  }
#pragma unroll
  for (int q = 0; q < DK; ++q) {
    if (cas[q]) {
      if (old[q] == kEmpty) res[q] = static_cast<int32_t>(b[q] * S + es[q]);
      else slow[q] = true;
    }
    if (v[q] && !slow[q]) slot_out[pos[q]] = res[q];
  }
}

// A warp's list in shared memory of positions put off to a round of their
// own, so that slower paths run on full warps instead of stalling every warp
// for a few lanes.  Every lane of the warp calls push and take.
struct WarpList {
  int32_t* at;
  int n = 0;  // warp-uniform
  __device__ explicit WarpList(int32_t* storage) : at(storage) {}
  __device__ __forceinline__ void push(bool mine, int64_t pos) {
    const int lane = threadIdx.x & 31;
    const unsigned bal = __ballot_sync(0xFFFFFFFFu, mine);
    if (mine) at[n + __popc(bal & ((1u << lane) - 1u))] = static_cast<int32_t>(pos);
    n += __popc(bal);
    __syncwarp();
  }
  // Removes the last 32 entries (or what there is): this lane's, -1 for none.
  __device__ __forceinline__ int64_t take() {
    const int lane = threadIdx.x & 31;
    const int from = n > 32 ? n - 32 : 0;
    const int64_t pos = from + lane < n ? at[from + lane] : -1;
    __syncwarp();
    n = from;
    return pos;
  }
};

// Claims a round of put-off positions by the full protocol.
template <int D, int S, class In, bool PrefFirst>
__device__ __forceinline__ void claim_slow_round(const TableView& t, const In& keys, WarpList& list,
                                                 int32_t* __restrict__ slot_out) {
  const int64_t pos = list.take();
  if (pos >= 0) slot_out[pos] = claim_one<D, S, In, PrefFirst>(t, keys, pos);
  __syncwarp();
}

// Claim kernel, bucket load first: KPT keys per thread, each claimed from its
// loaded home bucket (two dependent accesses per key: bucket load, CAS) in
// slot order; keys that need the full protocol (mostly full home buckets) are
// queued per warp and claimed 32 at a time: though 2 % of the keys, most
// warps have one, and running the protocol for it at once cost more than all
// its other keys' CASes (GB300, 10^8 keys by ranges: activate and find 9.18 ->
// 8.56 ms).  The better choice when the table does not stay in L2: the loads
// bring the buckets in with deep miss queues and the CASes then hit L2.  It
// takes as many blocks as are resident at once: 10^7 keys in input order 307
// us, 328 with eight blocks per SM (a thin second wave); the ranged calls on
// 10^8 keys 2579 us, 2785 with eight.  Beyond L2, in input order, the host
// picks the grid (claim_launch).  8-slot buckets: compiled for four
// blocks, the loads of both keys' buckets in flight, 8M keys 248 -> 230 us;
// 4-slot ones with four or five blocks asked for 239 and 225 against 230, but
// 20M inserts with values 728 and 776 against 761.  Slot order does
// not keep the preferred-slot invariant (preferred-first placement measured
// 5-10 % slower here), so the host clears the map's flag.
template <int D, int S, int KPT, class In = const int32_t*>
__global__ void __launch_bounds__(256, S == 8 && KPT == 2 ? 4 : 0) claim_bucket_kernel(TableView t, const In keys, int64_t n,
                                                           int32_t* __restrict__ slot_out) {
  // a programmatic dependent of the previous kernel: wait for its grid (a no-op otherwise)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ int32_t s_slow[8][32 + 32 * KPT];
  WarpList slow(s_slow[threadIdx.x >> 5]);
  const int lane = threadIdx.x & 31;
  const int64_t step = static_cast<int64_t>(gridDim.x) * blockDim.x * KPT;
  for (int64_t base = static_cast<int64_t>(blockIdx.x) * blockDim.x * KPT + threadIdx.x; base - lane < n; base += step) {
    int64_t p[KPT];
    bool v[KPT], put_off[KPT];
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      p[q] = base + static_cast<int64_t>(q) * blockDim.x;
      v[q] = p[q] < n;
    }
    claim_from_bucket<D, S, KPT, In, false>(t, keys, p, v, slot_out, put_off);
#pragma unroll
    for (int q = 0; q < KPT; ++q) slow.push(put_off[q], p[q]);
    while (slow.n >= 32) claim_slow_round<D, S, In, false>(t, keys, slow, slot_out);
  }
  if (slow.n > 0) claim_slow_round<D, S, In, false>(t, keys, slow, slot_out);
}

// Claim kernel, preferred slot first.  Each warp takes 32 * KPT consecutive
// keys per iteration (KPT per lane; the launcher uses 1).  Fast path per key:
// CAS the preferred slot of the home bucket, with no bucket load before it.
// EMPTY there: claimed.  An occupant with the key's fingerprint: compare once
// (claimant's input row or kB row); an equal key joins the claim (lowest
// position wins) or reports the committed key.  Any other key (the preferred
// slot holds another key, a tombstone, or a fingerprint collision) is queued
// in the warp's shared-memory list; whenever the list holds 32 * kDL keys the
// warp claims them from their buckets together, kDL per lane
// (claim_from_bucket), so the slower path runs on dense warps instead of
// stalling every warp for a few lanes (a second queue for those that then
// need the full protocol cost registers and 3 % at 4M keys).  A CAS that
// misses L2 waits on DRAM inside the atomic unit, so this path pays off while
// the table stays in L2.  Six blocks per SM for 4-slot buckets and up to four
// dimensions (40 registers): 4M claims 90 us, against 107 with four blocks and
// 105 with eight; points 117 (80 bytes spilled), against 121 with five and 126
// with the compiler's choice.  Elsewhere the compiler's choice (0) is the best
// one, and asking for any block at all (1) is not the same as leaving it: it
// raises the registers by half.  2M claims with 1 | 0 | a bound: 3-D, 8 slots
// 67 | 54 | 56 us (five blocks), 16 slots 88 | 63 | 65 (four), 5-D 61 | 53 |
// 57 (five), 8-D 79 | 71 | 72 (four).
template <int D, int S, int KPT, class In = const int32_t*>
__global__ void __launch_bounds__(256, S == 4 && D <= 4 ? 6 : 0) claim_pref_kernel(TableView t, const In keys, int64_t n,
                                                         int32_t* __restrict__ slot_out) {
  // a programmatic dependent of the previous kernel: wait for its grid (a no-op otherwise)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  constexpr int KS = KeyStride<D>::value;
  constexpr int kDL = KPT == 1 ? 1 : 2;      // queued keys per lane in a dense round
  constexpr int kDrain = 32 * kDL;
  constexpr int kCap = kDrain + 32 * KPT;    // a round starts before a tile could overflow
  __shared__ int32_t s_queue[8][kCap];
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int32_t* queue = s_queue[threadIdx.x >> 5];
  int qn = 0;  // warp-uniform
  const int64_t n_warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
  const int64_t warp_id = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  for (int64_t wbase = warp_id * 32 * KPT; wbase < n; wbase += n_warps * 32 * KPT) {
    int32_t k[KPT][D];
    uint32_t fp[KPT], ps[KPT];
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      const int64_t pos = wbase + q * 32 + lane;
      if (pos < n) {
        load_input_key<D>(keys, pos, k[q]);
      } else {
#pragma unroll
        for (int j = 0; j < D; ++j) k[q][j] = 0;
      }
      const uint64_t h = hash_key<D>(k[q]);
      fp[q] = fingerprint(h);
      ps[q] = home_bucket(h, t.n_buckets) * S + pref_slot<S>(fp[q]);
    }
    // A key equal to the one before it has lost to it, whatever becomes of
    // that one: points in scan order come in such runs, and without this all
    // of a run meet in one slot (block keys of a depth frame, 307k in 2k
    // blocks: 12.6 -> 7.0 us; random keys level).
    bool follows[KPT];
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      bool same = lane > 0;
#pragma unroll
      for (int j = 0; j < D; ++j) same &= __shfl_up_sync(0xFFFFFFFFu, k[q][j], 1) == k[q][j];
      follows[q] = same;
    }
    uint64_t old[KPT];
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      const int64_t pos = wbase + q * 32 + lane;
      old[q] = kTombstone;
      if (pos < n && !follows[q]) {
        const uint64_t mine = (static_cast<uint64_t>(fp[q]) << 32) | (kClaimBit | static_cast<uint32_t>(pos));
        old[q] = atomicCAS(reinterpret_cast<unsigned long long*>(t.slots + ps[q]),
                           static_cast<unsigned long long>(kEmpty), static_cast<unsigned long long>(mine));
      }
    }
    bool fm[KPT];
    int32_t row[KPT][KS];
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      const uint32_t lo = lo32(old[q]);
      fm[q] = lo != kNoIndex && hi32(old[q]) == fp[q];
      if (fm[q]) {
        if (lo & kClaimBit) {
          int32_t o[D];
          load_input_key<D>(keys, lo & ~kClaimBit, o);
#pragma unroll
          for (int j = 0; j < KS; ++j) row[q][j] = j < D ? o[j] : 0;
        } else {
          load_kb<D>(t.kb, lo, row[q]);
        }
      } else {
#pragma unroll
        for (int j = 0; j < KS; ++j) row[q][j] = 0;
      }
    }
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      const int64_t pos = wbase + q * 32 + lane;
      bool pending = false;
      if (pos < n) {
        const uint32_t lo = lo32(old[q]);
        bool eq = fm[q];
#pragma unroll
        for (int j = 0; j < D; ++j) eq &= (row[q][j] == k[q][j]);
        if (follows[q]) {
          slot_out[pos] = kClaimJoined;
        } else if (old[q] == kEmpty) {
          slot_out[pos] = static_cast<int32_t>(ps[q]);
        } else if (!eq) {
          pending = true;
        } else if (lo & kClaimBit) {
          const uint64_t mine = (static_cast<uint64_t>(fp[q]) << 32) | (kClaimBit | static_cast<uint32_t>(pos));
          slot_out[pos] = join_claim(t, t.slots + ps[q], lo, mine, static_cast<uint32_t>(pos))
                              ? static_cast<int32_t>(ps[q])
                              : kClaimJoined;
        } else {
          slot_out[pos] = kClaimExists;
        }
      }
      const unsigned bal = __ballot_sync(0xFFFFFFFFu, pending);
      if (pending) queue[qn + __popc(bal & lt)] = static_cast<int32_t>(pos);
      qn += __popc(bal);
    }
    __syncwarp();
    while (qn >= kDrain) {
      int64_t p[kDL];
      bool v[kDL], slow[kDL];
#pragma unroll
      for (int r = 0; r < kDL; ++r) {
        v[r] = true;
        p[r] = queue[qn - kDrain + r * 32 + lane];
      }
      __syncwarp();
      qn -= kDrain;
      claim_from_bucket<D, S, kDL, In, true>(t, keys, p, v, slot_out, slow);
#pragma unroll
      for (int r = 0; r < kDL; ++r)
        if (slow[r]) slot_out[p[r]] = claim_one<D, S, In, true>(t, keys, p[r]);
    }
  }
  __syncwarp();
  if (qn > 0) {
    int64_t p[kDL];
    bool v[kDL], slow[kDL];
#pragma unroll
    for (int r = 0; r < kDL; ++r) {
      v[r] = r * 32 + lane < qn;
      p[r] = v[r] ? queue[r * 32 + lane] : 0;
    }
    claim_from_bucket<D, S, kDL, In, true>(t, keys, p, v, slot_out, slow);
#pragma unroll
    for (int r = 0; r < kDL; ++r)
      if (slow[r]) slot_out[p[r]] = claim_one<D, S, In, true>(t, keys, p[r]);
  }
}

// ------------------------------------------------------------ insert: commit
// One value buffer whose rows are exactly 4, 8 or 16 bytes with both bases
// aligned to the row size: the committing thread copies its row as one
// vector.  Other layouts use the scatter kernel after the commit.
struct ValueRow {
  void* dst;
  const void* src;
  int64_t row_bytes;  // 4, 8 or 16
  int vec;
  int pad;
};

__device__ __forceinline__ void copy_small_row(const ValueRow& v, int32_t i, int64_t pos) {
  char* d = static_cast<char*>(v.dst) + static_cast<int64_t>(i) * v.row_bytes;
  const char* s = static_cast<const char*>(v.src) + pos * v.row_bytes;
  if (v.row_bytes == 16) *reinterpret_cast<uint4*>(d) = __ldg(reinterpret_cast<const uint4*>(s));
  else if (v.row_bytes == 8) *reinterpret_cast<uint2*>(d) = __ldg(reinterpret_cast<const uint2*>(s));
  else *reinterpret_cast<uint32_t*>(d) = __ldg(reinterpret_cast<const uint32_t*>(s));
}

// KPT keys per thread per block iteration (blockDim.x * KPT keys).  Who won
// each key: FLAGS, a position holding a slot index whose winner-flag bit
// (t.lost) is clear, from two streamed reads; otherwise the slot word, read
// at random, names the winning position.  The first warp scans the warps'
// counts of winners and ONE heap atomic serves the iteration (Sec. 4.3: t is
// raised by the number of indices taken).  Winners then write kB(i), the value
// row, the committed slot word and their outputs.  `turn` alternates between 0
// and 1 from tile to tile (TileShared).
//
// Bound by random sectors (the slot words); past L2 by DRAM, and then by how
// many warps are resident and how early their loads go out.  So the prefix is
// left in shared memory rather than in every warp's registers, the winners'
// key rows are asked for right after the barrier, and two keys per thread are
// held to eight blocks.  With every warp scanning for itself and the rows
// loaded last, 8M keys of 5 dimensions took 156 us (now 149), of 8 163 (153),
// of 3 131 (130), two per thread 137 (129) and, 2M in L2, 24 (20).
template <int D, int KPT, bool VAL, class In, bool FLAGS = false>
__device__ __forceinline__ void commit_tile(const TableView& t, const In& keys, int64_t n,
                                            int64_t base0, int32_t* __restrict__ idx, uint8_t* __restrict__ mask,
                                            const ValueRow& v, TileShared& sh, int turn) {
  // points are quantised as they are loaded, and the batched kernel holds every
  // dimension's code: both were slower with the rows' registers held longer
  // (4M points 54 for 52 us)
  constexpr bool kRowsEarly = FLAGS && std::is_pointer<In>::value;
  const int64_t base = base0 + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int n_warps = blockDim.x >> 5;
  int32_t s[KPT];
#pragma unroll
  for (int q = 0; q < KPT; ++q) {
    const int64_t pos = base + static_cast<int64_t>(q) * blockDim.x;
    s[q] = pos < n ? idx[pos] : -1;
  }
  uint64_t w[KPT];
  unsigned won[KPT];  // of this warp
  if constexpr (FLAGS) {
    uint32_t lw[KPT];
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      const int64_t pos = base + static_cast<int64_t>(q) * blockDim.x;
      w[q] = 0;
      lw[q] = pos < n ? t.lost[pos >> 5] : 0u;
    }
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      const int64_t pos = base + static_cast<int64_t>(q) * blockDim.x;
      won[q] = __ballot_sync(0xFFFFFFFFu, s[q] >= 0 && !((lw[q] >> (pos & 31)) & 1u));
      // leave the flags clear for the next insert (blockDim and the tile base
      // are multiples of 32, so a warp's 32 positions of one slice are one
      // word, which no other warp reads)
      if (lane == 0 && lw[q] != 0u) t.lost[pos >> 5] = 0u;
    }
  } else {
#pragma unroll
    for (int q = 0; q < KPT; ++q) w[q] = s[q] >= 0 ? load_slot_relaxed(t.slots + s[q]) : 0ull;
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      const int64_t pos = base + static_cast<int64_t>(q) * blockDim.x;
      won[q] = __ballot_sync(0xFFFFFFFFu, s[q] >= 0 && lo32(w[q]) == (kClaimBit | static_cast<uint32_t>(pos)));
    }
  }
  if (lane == 0) {
#pragma unroll
    for (int q = 0; q < KPT; ++q) sh.cnt[turn][q * n_warps + warp] = __popc(won[q]);
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const int c = lane < KPT * n_warps ? sh.cnt[turn][lane] : 0;
    const int upto = warp_scan(c);
    sh.cnt[turn][lane] = upto - c;
    const int total = __shfl_sync(0xFFFFFFFFu, upto, 31);
    if (threadIdx.x == 0) {
      int got = 0, top = 0;
      if (total > 0) {
        const unsigned long long add = (static_cast<unsigned long long>(total) << 32) | static_cast<unsigned long long>(total);
        const unsigned long long old = atomicAdd(&t.ctrl->top_used, add);
        top = static_cast<int>(static_cast<uint32_t>(old));
        got = t.capacity - top;
        got = got < 0 ? 0 : (got > total ? total : got);
        if (got < total) {
          // give back the part of t that the heap could not serve
          atomicAdd(&t.ctrl->top_used, 0ull - static_cast<unsigned long long>(total - got));
          atomicOr(&t.ctrl->status, kStatusCapacity);
        }
      }
      sh.base[turn] = top;
      sh.got[turn] = got;
    }
  }
  __syncthreads();
  const int got = sh.got[turn];
  const int hbase = sh.base[turn];
#pragma unroll
  for (int q = 0; q < KPT; ++q) {
    const int64_t pos = base + static_cast<int64_t>(q) * blockDim.x;
    const bool win = (won[q] >> lane) & 1u;
    int32_t k[D];
    if (kRowsEarly && win) load_input_key<D>(keys, pos, k);
    const int r = sh.cnt[turn][q * n_warps + warp] + __popc(won[q] & ((1u << lane) - 1u));
    if (pos < n) {
      if (win) {
        if (r < got) {
          const int32_t i = (t.flags & kViewHeapIdentity) ? hbase + r : t.heap[hbase + r];
          if (!kRowsEarly) load_input_key<D>(keys, pos, k);
          store_kb<D>(t.kb, static_cast<uint32_t>(i), k);
          if constexpr (VAL) copy_small_row(v, i, pos);
          const uint32_t fp = FLAGS ? fingerprint(hash_key<D>(k)) : hi32(w[q]);
          t.slots[s[q]] = (static_cast<uint64_t>(fp) << 32) | static_cast<uint32_t>(i);
          idx[pos] = i;
          mask[pos] = 1;
        } else {
          t.slots[s[q]] = kTombstone;
          idx[pos] = -1;
          mask[pos] = 0;
        }
      } else {
        idx[pos] = -1;
        mask[pos] = 0;
      }
    }
  }
}

template <int D, int KPT, bool VAL, class In = const int32_t*, bool FLAGS = false>
__global__ void __launch_bounds__(256, KPT == 2 ? 8 : 0) commit_kernel(TableView t, const In keys, int64_t n,
                                                     int32_t* __restrict__ idx, uint8_t* __restrict__ mask,
                                                     ValueRow v) {
  __shared__ TileShared sh;
  // a programmatic dependent of the previous kernel: wait for its grid (a no-op otherwise)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t step = static_cast<int64_t>(gridDim.x) * blockDim.x * KPT;
  int turn = 0;
  for (int64_t base0 = static_cast<int64_t>(blockIdx.x) * blockDim.x * KPT; base0 < n; base0 += step, turn ^= 1)
    commit_tile<D, KPT, VAL, In, FLAGS>(t, keys, n, base0, idx, mask, v, sh, turn);
  if (t.snap != nullptr && threadIdx.x == 0) publish_when_last(t);
}

// ------------------------------------------------------- key partitioning
// For tables larger than L2, a call's keys are first put in the order of
// their home buckets' ranges: P = 2^log_p ranges of consecutive buckets (the
// top log_p bits of the hash word the home bucket comes from), a stable
// partition, so that equal keys keep their input order and the lowest
// position still wins.  The claim, commit and find kernels walk their keys
// in order, so each then works on one range of the table at a time, and of
// kB too once the commit has handed out indices in the same order, and
// finds it in L2.
//
// Each of G blocks owns a contiguous span of whole tiles of kPartTile input
// keys.  A count pass histograms each block's span per range (counts[P][G]);
// a scan turns each range's row into the blocks' offsets within the range
// (and the range totals); the scatter pass sorts each tile by range in
// shared memory (stable: each warp holds consecutive tile positions in
// steps of 32, ranked by __match_any_sync) and writes each range's part of
// the tile as one run after the block's previous tiles' runs.  dest[pos]
// records where input row pos went, for the outputs' way back.
//
// The scatter is bound by instruction issue and by its tiles' barriers, not by
// HBM (10^8 rows of 12 bytes: 894 -> 683 us, 4.1 TB/s).  What brought it
// there: the count pass hands over each key's range in a byte (752 -> 683,
// count 215 -> 229), up to 32 ranges are scanned by one warp (806 -> 765),
// dest is written by the thread that holds the row, in input order, and the
// counts take shared memory for P ranges only (894 -> 806 together).  Sorted
// rows leave row by row (word by word, so that stores coalesce, 765 against
// 752).  512 or 1024 threads per tile: 974 and 1420 us; tiles of 1024 or 4096
// keys: 798 and 777; 3, 5 or 6 blocks per SM: 714, 785, 920.
constexpr int kPartTile = 2048;     // keys per tile
constexpr int kCountThreads = 256;
constexpr int kScatterThreads = 256;
constexpr int kPartBlocksPerSm = 4;
constexpr int kPartMaxLog = 8;      // at most 256 ranges
constexpr uint32_t kNoRange = 0xFFFFFFFFu;

__device__ __forceinline__ uint32_t key_range(uint64_t h, int log_p) { return hi32(h) >> (32 - log_p); }

// The STEPS key rows of one lane in warp w's part of a tile (local positions
// 32 (STEPS w + j) + lane); zeros past the tile.
template <int D, int STEPS>
__device__ __forceinline__ void load_tile_rows(const int32_t* __restrict__ keys, int64_t base, int tn,
                                               int32_t (&k)[STEPS][D]) {
  const int first = (threadIdx.x >> 5) * 32 * STEPS + (threadIdx.x & 31);
#pragma unroll
  for (int j = 0; j < STEPS; ++j) {
    if (first + j * 32 < tn) {
      load_input_key<D>(keys, base + first + j * 32, k[j]);
    } else {
#pragma unroll
      for (int c = 0; c < D; ++c) k[j][c] = 0;
    }
  }
}

// Their ranges (kNoRange past the tile).
template <int D, int STEPS>
__device__ __forceinline__ void tile_ranges(const int32_t (&k)[STEPS][D], int tn, int log_p, uint32_t (&r)[STEPS]) {
  const int first = (threadIdx.x >> 5) * 32 * STEPS + (threadIdx.x & 31);
#pragma unroll
  for (int j = 0; j < STEPS; ++j)
    r[j] = first + j * 32 < tn ? key_range(hash_key<D>(k[j]), log_p) : kNoRange;
}

// Keys in tile at `base` of a span ending at t1.
__device__ __forceinline__ int tile_keys(int64_t base, int64_t t1) {
  return t1 - base < kPartTile ? static_cast<int>(t1 - base) : kPartTile;
}

// counts[p * G + b]: keys of range p in block b's span; ranges[pos]: the range
// of each key, so that the scatter need not hash again.
template <int D>
__global__ void __launch_bounds__(kCountThreads) partition_count_kernel(const int32_t* __restrict__ keys, int64_t n, int log_p,
                                                              int tiles_per_block, uint32_t* __restrict__ counts,
                                                              uint8_t* __restrict__ ranges) {
  __shared__ uint32_t s_hist[1 << kPartMaxLog];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int P = 1 << log_p;
  for (int p = threadIdx.x; p < P; p += blockDim.x) s_hist[p] = 0u;
  __syncthreads();
  const int64_t t0 = static_cast<int64_t>(blockIdx.x) * tiles_per_block * kPartTile;
  const int64_t t1 = t0 + static_cast<int64_t>(tiles_per_block) * kPartTile < n
                         ? t0 + static_cast<int64_t>(tiles_per_block) * kPartTile
                         : n;
  // each tile's rows are loaded while the tile before is being counted
  constexpr int kSteps = kPartTile / kCountThreads;
  int32_t k[kSteps][D];
  if (t0 < t1) load_tile_rows<D, kSteps>(keys, t0, tile_keys(t0, t1), k);
  for (int64_t base = t0; base < t1; base += kPartTile) {
    const int tn = tile_keys(base, t1);
    uint32_t r[kSteps];
    tile_ranges<D, kSteps>(k, tn, log_p, r);
    if (base + kPartTile < t1) load_tile_rows<D, kSteps>(keys, base + kPartTile, tile_keys(base + kPartTile, t1), k);
#pragma unroll
    for (int j = 0; j < kSteps; ++j) {
      if (r[j] != kNoRange) {
        atomicAdd(&s_hist[r[j]], 1u);
        ranges[base + ((threadIdx.x >> 5) * kSteps + j) * 32 + (threadIdx.x & 31)] = static_cast<uint8_t>(r[j]);
      }
    }
  }
  __syncthreads();
  for (int p = threadIdx.x; p < P; p += blockDim.x) counts[static_cast<int64_t>(p) * gridDim.x + blockIdx.x] = s_hist[p];
}

// Dynamic shared memory of the scatter kernel: the tile's key rows, their
// places, and each warp's counts per range.
template <int D>
constexpr size_t partition_scatter_smem(int P) {
  return sizeof(int32_t) * (kPartTile * (D + 1) + kScatterThreads / 32 * P);
}

// row_offsets: counts after the scan (block b's first place within range p);
// range_totals: keys per range.
template <int D>
__global__ void __launch_bounds__(kScatterThreads) partition_scatter_kernel(
    const int32_t* __restrict__ keys, const uint8_t* __restrict__ ranges, int64_t n, int log_p, int tiles_per_block,
    const uint32_t* __restrict__ row_offsets, const uint32_t* __restrict__ range_totals,
    int32_t* __restrict__ keys_out, int32_t* __restrict__ dest) {
  constexpr int kWarps = kScatterThreads / 32;
  constexpr int kSteps = kPartTile / kScatterThreads;
  extern __shared__ int32_t s_keys[];             // [kPartTile][D], the tile in range order
  uint32_t* s_to = reinterpret_cast<uint32_t*>(s_keys) + kPartTile * D;  // place in keys_out of each of its rows
  uint32_t* s_cnt = s_to + kPartTile;             // [kWarps][P]: keys of each range, then the warp's offset in it
  __shared__ uint32_t s_run[1 << kPartMaxLog];    // next place of each range for this block
  __shared__ uint32_t s_start[1 << kPartMaxLog];  // first tile slot of each range
  __shared__ int s_warp[33];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int P = 1 << log_p;
  const int tid = threadIdx.x;
  const int w = tid >> 5;
  const int lane = tid & 31;
  const unsigned lt = (1u << lane) - 1u;
  uint32_t* mine = s_cnt + w * P;
  {
    int unused;
    const uint32_t tot = tid < P ? range_totals[tid] : 0u;
    const uint32_t start = static_cast<uint32_t>(block_exclusive_scan(static_cast<int>(tot), unused, s_warp));
    if (tid < P) s_run[tid] = start + row_offsets[static_cast<int64_t>(tid) * gridDim.x + blockIdx.x];
    __syncthreads();
  }
  const int64_t t0 = static_cast<int64_t>(blockIdx.x) * tiles_per_block * kPartTile;
  const int64_t t1 = t0 + static_cast<int64_t>(tiles_per_block) * kPartTile < n
                         ? t0 + static_cast<int64_t>(tiles_per_block) * kPartTile
                         : n;
  for (int64_t base = t0; base < t1; base += kPartTile) {
    const int tn = tile_keys(base, t1);
    for (int p = lane; p < P; p += 32) mine[p] = 0u;
    __syncwarp();
    int32_t k[kSteps][D];
    uint32_t r[kSteps];
#pragma unroll
    for (int j = 0; j < kSteps; ++j) {
      const int local = (w * kSteps + j) * 32 + lane;
      r[j] = local < tn ? __ldg(ranges + base + local) : kNoRange;
    }
    load_tile_rows<D, kSteps>(keys, base, tn, k);
    uint32_t rank[kSteps];
#pragma unroll
    for (int j = 0; j < kSteps; ++j) {
      const bool valid = r[j] != kNoRange;
      const unsigned peers = __match_any_sync(0xFFFFFFFFu, r[j]);
      const uint32_t c = valid ? mine[r[j]] : 0u;
      rank[j] = c + __popc(peers & lt);
      __syncwarp();
      if (valid && lane == __ffs(peers) - 1) mine[r[j]] = c + __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    // per range: the warps' counts to their offsets within it, then the
    // ranges' first slots; up to 32 ranges are one warp's work, with no
    // barrier in it
    uint32_t tc = 0;  // the tile's keys of range tid
    if (tid < P) {
#pragma unroll
      for (int ww = 0; ww < kWarps; ++ww) {
        const uint32_t c = s_cnt[ww * P + tid];
        s_cnt[ww * P + tid] = tc;
        tc += c;
      }
    }
    if (P <= 32) {
      if (w == 0) {
        uint32_t x = tc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
          if (lane >= o) x += y;
        }
        s_start[lane] = x - tc;
      }
    } else {
      int tile_total;
      const uint32_t st = static_cast<uint32_t>(block_exclusive_scan(static_cast<int>(tc), tile_total, s_warp));
      if (tid < P) s_start[tid] = st;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSteps; ++j) {
      if (r[j] != kNoRange) {
        const uint32_t off = mine[r[j]] + rank[j];
        const uint32_t slot = s_start[r[j]] + off;
        const uint32_t to = s_run[r[j]] + off;
#pragma unroll
        for (int c = 0; c < D; ++c) s_keys[slot * D + c] = k[j][c];
        s_to[slot] = to;
        dest[base + (w * kSteps + j) * 32 + lane] = static_cast<int32_t>(to);
      }
    }
    __syncthreads();
    for (int slot = tid; slot < tn; slot += kScatterThreads) {
      int32_t* row = keys_out + static_cast<int64_t>(s_to[slot]) * D;
#pragma unroll
      for (int c = 0; c < D; ++c) row[c] = s_keys[slot * D + c];
    }
    if (tid < P) s_run[tid] += tc;
    __syncthreads();
  }
}

// --------------------------------------------------------------- erase: mark
// Finds input row pos and marks its slot with the lowest position seen
// (atomicMin into the high word, the buffer index kept in the low word).
// Returns the slot index, or -1 if the key is absent.
template <int D, int S>
__device__ __forceinline__ int32_t erase_mark_one(const TableView& t, const int32_t* __restrict__ keys, int64_t pos) {
  int32_t k[D];
  load_input_key<D>(keys, pos, k);
  const uint64_t h = hash_key<D>(k);
  const uint32_t fp = fingerprint(h);
  uint32_t b = home_bucket(h, t.n_buckets);
  int32_t res = -1;
  for (uint32_t probe = 0; probe < t.max_probes && res < 0; ++probe) {
    uint64_t* bp = t.slots + static_cast<size_t>(b) * S;
    uint64_t w[S];
    load_bucket<S, false>(bp, w);
    // candidates: committed with an equal fingerprint, or already marked
    // (fingerprint gone); the former first, each compared by itself, so the
    // lanes of a warp usually wait for one compare
    bool stop = false;
    uint32_t same = 0, marked = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const uint32_t lo = lo32(w[s]), hi = hi32(w[s]);
      stop |= (w[s] == kEmpty);
      same |= (lo < kClaimBit && hi == fp ? 1u : 0u) << s;
      marked |= (lo < kClaimBit && hi < kFpBit ? 1u : 0u) << s;
    }
    while (same | marked) {
      const int at = __ffs(same ? same : marked) - 1;
      if (same) same &= same - 1;
      else marked &= marked - 1;
      uint64_t word = 0;
#pragma unroll
      for (int s = 0; s < S; ++s)
        if (s == at) word = w[s];
      if (kb_equal<D>(t.kb, lo32(word), k)) {
        if (hi32(word) > static_cast<uint32_t>(pos))
          atomicMin(reinterpret_cast<unsigned long long*>(bp + at),
                    (static_cast<unsigned long long>(pos) << 32) | lo32(word));
        res = static_cast<int32_t>(b * S + at);
        break;
      }
    }
    if (stop) break;
    b = next_bucket(b, t.n_buckets);
  }
  return res;
}

template <int D, int S>
__global__ void __launch_bounds__(256) erase_mark_kernel(TableView t, const int32_t* __restrict__ keys, int64_t n,
                                                         int32_t* __restrict__ slot_out) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int64_t pos = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; pos < n; pos += stride)
    slot_out[pos] = erase_mark_one<D, S>(t, keys, pos);
}

// ------------------------------------------------------------ erase: resolve
// For every lane with `asks`: whether no key that stays in the table probes
// on past its bucket b.  Such a key would have to sit in the next bucket (which
// holds an EMPTY slot, so none of its chains goes further) with another home
// bucket.  Marked words leave the table in this kernel, so they do not count;
// a slot of the next bucket that another thread empties meanwhile only makes
// the answer truer.  Few lanes ask, so the warp answers 32 / S of them at a
// time, a lane per slot of the next bucket: one slot load and one kB row deep
// (a lane that walked its bucket alone held its warp for four of each, and the
// resolve of 262k erases took 18.8 us instead of 14.2).
template <int S>
__device__ __forceinline__ bool nobody_probes_past(const TableView& t, bool asks, uint32_t b, uint32_t* ask) {
  constexpr int G = 32 / S;
  const int lane = threadIdx.x & 31;
  const unsigned asking = __ballot_sync(0xFFFFFFFFu, asks);
  const int n = __popc(asking);
  const int rank = __popc(asking & ((1u << lane) - 1u));
  bool none = false;
  for (int r = 0; r < n; r += G) {
    const bool mine = asks && rank >= r && rank < r + G;
    if (mine) ask[rank - r] = b;
    __syncwarp();
    const int g = lane / S;
    bool empty = false, displaced = false;
    if (r + g < n) {
      const uint32_t nb = next_bucket(ask[g], t.n_buckets);
      const uint64_t w = load_slot_relaxed(t.slots + static_cast<size_t>(nb) * S + lane % S);
      empty = w == kEmpty;
      displaced = nb == ask[g] || (is_committed(w) && home_of_row(t.kb, t.key_dim, t.n_buckets, lo32(w)) != nb);
    }
    const unsigned eb = __ballot_sync(0xFFFFFFFFu, empty), db = __ballot_sync(0xFFFFFFFFu, displaced);
    if (mine) {
      const unsigned group = ((1u << S) - 1u) << ((rank - r) * S);
      none = (eb & group) != 0u && (db & group) == 0u;
    }
    __syncwarp();
  }
  return none;
}

// One tile of blockDim.x positions starting at base0.  Every thread of the
// block must call it (block-wide scan and barriers).
template <int S>
__device__ __forceinline__ void erase_resolve_tile(const TableView& t, int64_t n, int64_t base0,
                                                   const int32_t* __restrict__ slot_in, uint8_t* __restrict__ mask,
                                                   TileShared& sh, int turn) {
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int64_t pos = base0 + threadIdx.x;
  const bool active = pos < n;
  const int32_t s = active ? slot_in[pos] : -1;
  uint64_t w = 0;
  bool win = false, to_empty = false;
  bool past_home = false;  // its bucket has no EMPTY slot: chains may pass
  bool held = false;       // another live key prefers the slot
  if (s >= 0) {
    // EMPTY only when no probe chain passes through the bucket (it already has
    // an EMPTY slot, or nobody_probes_past it) and, while the map keeps the
    // preferred-slot invariant, no other live key of the bucket prefers the
    // freed slot; a TOMBSTONE otherwise (the freed slot itself holds a marked
    // word, which never counts).  The bucket is read 32 bytes at a time, the
    // slot's own 32 bytes first: they tell the winner.
    const uint64_t* bp = t.slots + static_cast<size_t>(s / S) * S;
    const uint32_t own = static_cast<uint32_t>(s) & (S - 1);
    bool preferred = false;
#pragma unroll 1
    for (int c = 0; c < S / 4; ++c) {
      const uint32_t part = (own / 4 + c) % (S / 4);
      uint64_t cw[4];
      load32<false>(bp + 4 * part, cw[0], cw[1], cw[2], cw[3]);
      if (c == 0) {
        w = (own & 2) ? ((own & 1) ? cw[3] : cw[2]) : ((own & 1) ? cw[1] : cw[0]);
        win = hi32(w) == static_cast<uint32_t>(pos);
        if (!win) break;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        to_empty |= (cw[j] == kEmpty);
        preferred |= is_committed(cw[j]) && pref_slot<S>(hi32(cw[j])) == own;
      }
    }
    past_home = win && !to_empty;
    held = preferred && (t.flags & kViewPrefPlaced);
  }
  if (nobody_probes_past<S>(t, past_home && !held, static_cast<uint32_t>(s) / S, sh.ask[warp])) to_empty = true;
  to_empty &= !held;
  // winners in the low half, slots that become EMPTY in the high half
  const unsigned won = __ballot_sync(0xFFFFFFFFu, win);
  const unsigned emptied = __ballot_sync(0xFFFFFFFFu, to_empty);
  if (lane == 0) sh.cnt[turn][warp] = __popc(won) | __popc(emptied) << 16;
  __syncthreads();
  const int c = lane < static_cast<int>(blockDim.x >> 5) ? sh.cnt[turn][lane] : 0;
  const int upto = warp_scan(c);
  if (threadIdx.x < 32) {
    const int both = __shfl_sync(0xFFFFFFFFu, upto, 31);
    if (threadIdx.x == 0) {
      const int total = both & 0xFFFF;
      int top = 0;
      if (total > 0) {
        const unsigned long long sub = (static_cast<unsigned long long>(both >> 16) << 32) + static_cast<unsigned long long>(total);
        const unsigned long long old = atomicAdd(&t.ctrl->top_used, 0ull - sub);
        top = static_cast<int>(static_cast<uint32_t>(old));
      }
      sh.base[turn] = top - total;
    }
  }
  __syncthreads();
  const int before = __shfl_sync(0xFFFFFFFFu, upto - c, warp) & 0xFFFF;
  if (win) {
    t.heap[sh.base[turn] + before + __popc(won & ((1u << lane) - 1u))] = static_cast<int32_t>(lo32(w));
    t.slots[s] = to_empty ? kEmpty : kTombstone;
    mask[pos] = 1;
  } else if (active) {
    mask[pos] = 0;
  }
}

template <int S>
__global__ void __launch_bounds__(256) erase_resolve_kernel(TableView t, int64_t n, const int32_t* __restrict__ slot_in,
                                                            uint8_t* __restrict__ mask) {
  __shared__ TileShared sh;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  int turn = 0;
  for (int64_t base = static_cast<int64_t>(blockIdx.x) * blockDim.x; base < n; base += stride, turn ^= 1)
    erase_resolve_tile<S>(t, n, base, slot_in, mask, sh, turn);
  if (t.snap != nullptr && threadIdx.x == 0) publish_when_last(t);
}

// ------------------------------------------------------------------ rebuild
// Inserts n unique keys taken from kb_src rows list[j] into an empty table
// (list == nullptr: rows 0..n-1, the live entries while the heap is the
// identity).  preserve: the entry keeps buffer index list[j]; otherwise it
// becomes j.  The key row is copied to kb_dst when kb_dst != kb_src or
// !preserve.  How many entries there are: kCountExact, n; otherwise at most
// n, the listing's count or the heap top as the device knows them (so that a
// rebuild can be enqueued without the host knowing), and the used-slot count
// becomes that number.
constexpr int kCountExact = 0;
constexpr int kCountListed = 1;
constexpr int kCountTop = 2;

template <int D, int S>
__global__ void __launch_bounds__(256) rebuild_kernel(TableView t, const int32_t* __restrict__ kb_src,
                                                      const int32_t* __restrict__ list, int64_t n, int count,
                                                      int preserve, int copy_keys) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (count != kCountExact) {
    // the low word (the heap top) does not change, so blocks may read it
    // before or after the first one's store
    const unsigned long long top = t.ctrl->top_used & 0xFFFFFFFFull;
    const unsigned long long live = count == kCountListed ? t.ctrl->count : top;
    n = min(n, static_cast<int64_t>(live));
    if (blockIdx.x == 0 && threadIdx.x == 0) t.ctrl->top_used = (live << 32) | top;
  }
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; j < n; j += stride) {
    const uint32_t a = static_cast<uint32_t>(list ? list[j] : j);
    int32_t row[KeyStride<D>::value];
    load_kb<D>(kb_src, a, row);
    int32_t k[D];
#pragma unroll
    for (int c = 0; c < D; ++c) k[c] = row[c];
    const uint32_t i = preserve ? a : static_cast<uint32_t>(j);
    const uint64_t h = hash_key<D>(k);
    const uint64_t word = (static_cast<uint64_t>(fingerprint(h)) << 32) | i;
    uint32_t b = home_bucket(h, t.n_buckets);
    // the preferred slot first (preferred-slot invariant), then the full probe
    const uint32_t ps = b * S + pref_slot<S>(fingerprint(h));
    bool placed = atomicCAS(reinterpret_cast<unsigned long long*>(t.slots + ps), static_cast<unsigned long long>(kEmpty),
                            static_cast<unsigned long long>(word)) == kEmpty;
    for (uint32_t probe = 0; probe < t.max_probes && !placed; ++probe) {
      uint64_t* bp = t.slots + static_cast<size_t>(b) * S;
      uint64_t w[S];
      load_bucket<S, false>(bp, w);
#pragma unroll
      for (int s = 0; s < S; ++s) {
        if (!placed && w[s] == kEmpty) {
          const uint64_t old = atomicCAS(reinterpret_cast<unsigned long long*>(bp + s),
                                         static_cast<unsigned long long>(kEmpty), static_cast<unsigned long long>(word));
          placed = (old == kEmpty);
        }
      }
      b = next_bucket(b, t.n_buckets);
    }
    if (!placed) atomicOr(&t.ctrl->status, kStatusTableFull);
    if (copy_keys) store_kb<D>(t.kb, i, k);
  }
}

// ----------------------------------------------------------------- launchers
struct Launch {
  cudaStream_t stream;
  int grid_cap;  // SMs x blocks_per_sm
  int block;
  int sms = 0;   // SM count (0: unknown)
  bool one_wave = true;  // resident_grid holds a grid to the blocks that fit at once
};

// Launch with programmatic stream serialisation: the kernel's blocks may be
// scheduled while the previous kernel on the stream drains, hiding the
// launch latency between the two.  The kernel must execute
// griddepcontrol.wait before it touches memory the previous kernel writes.
// The result also stays behind as the last error, which the calls check at
// their end (check_launch).
template <class... P, class... A>
inline cudaError_t launch_dependent_smem(void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t st,
                                         A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(grid));
  cfg.blockDim = dim3(static_cast<unsigned>(block));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

template <class... P, class... A>
inline cudaError_t launch_dependent(void (*kernel)(P...), int grid, int block, cudaStream_t st, A... args) {
  return launch_dependent_smem(kernel, grid, block, 0, st, args...);
}

// Blocks of Kernel (block threads `block`, no dynamic shared memory) that fit
// on one SM, from the occupancy API.  The kernel is a template argument, so
// each has a cache of its own: kernels of one signature differ in registers,
// and who was called first must not set the others' grids.  (One architecture
// is built, so the answer is the same on every device.)
template <auto Kernel>
inline int resident_blocks(int block) {
  static std::atomic<int> cache[9] = {};  // block / 32 in 1..8
  const int slot = block / 32;
  if (slot < 1 || slot > 8) return 1;
  int nb = cache[slot].load(std::memory_order_relaxed);
  if (nb == 0) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, Kernel, block, 0) != cudaSuccess || nb < 1) nb = 1;
    cache[slot].store(nb, std::memory_order_relaxed);
  }
  return nb;
}

// Grid of a grid-stride kernel whose registers allow fewer resident blocks
// than the Launch's cap: no more blocks than fit at once, so no thin second
// wave runs at low occupancy.
template <auto Kernel>
inline int resident_grid(int want, const Launch& L) {
  if (!L.one_wave || L.sms <= 0) return want;
  const int cap = L.sms * resident_blocks<Kernel>(L.block);
  return want < cap ? want : cap;
}

inline int grid_for(int64_t n, const Launch& L) {
  int64_t g = (n + L.block - 1) / L.block;
  if (g > L.grid_cap) g = L.grid_cap;
  return g < 1 ? 1 : static_cast<int>(g);
}

// Defined in ash_aux.cu.  Per range (one block each): the row of per-block
// counts counts[p][0..G) becomes its exclusive scan, the row's total goes to
// range_totals[p].
cudaError_t launch_partition_scan(uint32_t* counts, int G, int P, uint32_t* range_totals, const Launch& L);
// idx[pos] = idx_p[dest[pos]], mask[pos] = idx[pos] >= 0: a partitioned call's
// outputs back in input order.
void launch_unpermute(const int32_t* dest, int64_t n, const int32_t* idx_p, int32_t* idx, uint8_t* mask,
                      const Launch& L);

// Blocks of a partition pass over n keys (G) and whole tiles per block.
inline int partition_grid(int64_t n, const Launch& L, int* tiles_per_block) {
  const int64_t tiles = (n + kPartTile - 1) / kPartTile;
  const int64_t cap = L.sms > 0 ? static_cast<int64_t>(L.sms) * kPartBlocksPerSm : 512;
  const int64_t g0 = tiles < cap ? tiles : cap;
  const int64_t tpb = (tiles + g0 - 1) / g0;
  *tiles_per_block = static_cast<int>(tpb);
  const int64_t g = (tiles + tpb - 1) / tpb;
  return static_cast<int>(g < 1 ? 1 : g);
}

// Count words of a partitioned call on n keys (counts[P][G] and the P range
// totals).
inline int64_t partition_count_words(int64_t n, int log_p, const Launch& L) {
  int tpb = 0;
  const int64_t G = partition_grid(n, L, &tpb);
  return (G + 1) * (int64_t{1} << log_p);
}

// Function table for one key dimension (filled in by ash_dim.cu).  S: slots
// per bucket (4, 8, 16); kpt: keys per thread (1, 2, 4).
struct DimKernels {
  void (*find)(int S, int kpt, const TableView&, const int32_t*, int64_t, int32_t*, uint8_t*, const Launch&);
  void (*claim)(int S, int kpt, int pref, const TableView&, const int32_t*, int64_t, int32_t*, const Launch&);
  void (*commit)(int kpt, const TableView&, const int32_t*, int64_t, int32_t*, uint8_t*, const ValueRow*,
                 const Launch&);
  void (*erase_mark)(int S, const TableView&, const int32_t*, int64_t, int32_t*, const Launch&);
  void (*rebuild)(int S, const TableView&, const int32_t*, const int32_t*, int64_t, int, int, int, const Launch&);
  void (*neighbors)(int S, const TableView&, const int32_t*, int64_t, int, int64_t, int32_t*, uint8_t*, const Launch&);
  void (*offsets)(int S, const TableView&, const int32_t*, int64_t, const int32_t*, int64_t, int32_t*, uint8_t*,
                  const Launch&);
  void (*find_link)(int S, const TableView&, const int32_t*, int64_t, int32_t*, int32_t*, const int32_t*,
                    const Launch&);
  void (*find_group)(int S, const TableView&, const int32_t*, int64_t, int32_t*, uint8_t*, const Launch&);
  // stable partition of n key rows by home-bucket range; false: it was not enqueued whole
  bool (*partition)(const int32_t*, int64_t, int, uint32_t*, uint8_t*, int32_t*, int32_t*, const Launch&);
  // the same operations on float32 points quantised in the kernels
  void (*find_pts)(int S, int kpt, const TableView&, const PointRows&, int64_t, int32_t*, uint8_t*, const Launch&);
  void (*claim_pts)(int S, int kpt, int pref, const TableView&, const PointRows&, int64_t, int32_t*, const Launch&);
  void (*commit_pts)(int kpt, const TableView&, const PointRows&, int64_t, int32_t*, uint8_t*, const ValueRow*,
                     const Launch&);
};

template <int D>
struct DimLaunchers {
  template <int S, int KPT, class In>
  static void find_sk(const TableView& t, const In& keys, int64_t n, int32_t* idx, uint8_t* mask, const Launch& L) {
    TraceScope ts(kKFind, L.stream);
    // one key per thread: no more blocks than fit at once (8M finds of 8-D keys
    // 219 -> 211 us, 20M 428 -> 354; up to 6-D all of the cap's fit); with
    // several the second wave evens the rounds out (two keys, 3-D 158, 164 held)
    constexpr auto k = find_kernel<D, S, KPT, In>;
    const int g = grid_for((n + KPT - 1) / KPT, L);
    launch_dependent(k, KPT == 1 ? resident_grid<k>(g, L) : g, L.block, L.stream, t, keys, n, idx, mask);
  }
  template <int S, class In>
  static void find_s(int kpt, const TableView& t, const In& keys, int64_t n, int32_t* idx, uint8_t* mask,
                     const Launch& L) {
    if (kpt >= 4) find_sk<S, 4>(t, keys, n, idx, mask, L);
    else if (kpt == 2) find_sk<S, 2>(t, keys, n, idx, mask, L);
    else find_sk<S, 1>(t, keys, n, idx, mask, L);
  }
  template <class In>
  static void find_in(int S, int kpt, const TableView& t, const In& keys, int64_t n, int32_t* idx, uint8_t* mask,
                      const Launch& L) {
    if (S == 4) find_s<4>(kpt, t, keys, n, idx, mask, L);
    else if (S == 8) find_s<8>(kpt, t, keys, n, idx, mask, L);
    else find_s<16>(kpt, t, keys, n, idx, mask, L);
  }
  static void find(int S, int kpt, const TableView& t, const int32_t* keys, int64_t n, int32_t* idx, uint8_t* mask,
                   const Launch& L) {
    find_in(S, kpt, t, keys, n, idx, mask, L);
  }
  static void find_pts(int S, int kpt, const TableView& t, const PointRows& p, int64_t n, int32_t* idx,
                       uint8_t* mask, const Launch& L) {
    find_in(S, kpt, t, p, n, idx, mask, L);
  }
  // pref: 1 = preferred slot first (claim_pref_kernel), 0 = bucket load first.
  // The preferred-slot claim always takes one key per thread, which with one
  // queued key per lane in its dense rounds leaves more warps resident than
  // two keys per thread (4-8 % faster on GB300).
  template <int S, int KPT, class In>
  static void claim_sk(int pref, const TableView& t, const In& keys, int64_t n, int32_t* slot_out,
                       const Launch& L) {
    TraceScope ts(kKClaim, L.stream);
    const int g = grid_for((n + KPT - 1) / KPT, L);
    if (pref) {
      constexpr auto k = claim_pref_kernel<D, S, 1, In>;
      launch_dependent(k, resident_grid<k>(grid_for(n, L), L), L.block, L.stream, t, keys, n, slot_out);
    } else {
      constexpr auto k = claim_bucket_kernel<D, S, KPT, In>;
      launch_dependent(k, resident_grid<k>(g, L), L.block, L.stream, t, keys, n, slot_out);
    }
  }
  template <int S, class In>
  static void claim_s(int kpt, int pref, const TableView& t, const In& keys, int64_t n, int32_t* slot_out,
                      const Launch& L) {
    if (kpt >= 4) claim_sk<S, 4>(pref, t, keys, n, slot_out, L);
    else if (kpt == 2) claim_sk<S, 2>(pref, t, keys, n, slot_out, L);
    else claim_sk<S, 1>(pref, t, keys, n, slot_out, L);
  }
  template <class In>
  static void claim_in(int S, int kpt, int pref, const TableView& t, const In& keys, int64_t n, int32_t* slot_out,
                       const Launch& L) {
    if (S == 4) claim_s<4>(kpt, pref, t, keys, n, slot_out, L);
    else if (S == 8) claim_s<8>(kpt, pref, t, keys, n, slot_out, L);
    else claim_s<16>(kpt, pref, t, keys, n, slot_out, L);
  }
  static void claim(int S, int kpt, int pref, const TableView& t, const int32_t* keys, int64_t n, int32_t* slot_out,
                    const Launch& L) {
    claim_in(S, kpt, pref, t, keys, n, slot_out, L);
  }
  static void claim_pts(int S, int kpt, int pref, const TableView& t, const PointRows& p, int64_t n,
                        int32_t* slot_out, const Launch& L) {
    claim_in(S, kpt, pref, t, p, n, slot_out, L);
  }
  template <int KPT, bool VAL, class In>
  static void commit_kv(const TableView& t, const In& keys, int64_t n, int32_t* idx, uint8_t* mask,
                        const ValueRow& v, const Launch& L) {
    TraceScope ts(kKCommit, L.stream);
    const int g = grid_for((n + KPT - 1) / KPT, L);
    if (t.lost) launch_dependent(commit_kernel<D, KPT, VAL, In, true>, g, L.block, L.stream, t, keys, n, idx, mask, v);
    else launch_dependent(commit_kernel<D, KPT, VAL, In, false>, g, L.block, L.stream, t, keys, n, idx, mask, v);
  }
  template <bool VAL, class In>
  static void commit_v(int kpt, const TableView& t, const In& keys, int64_t n, int32_t* idx, uint8_t* mask,
                       const ValueRow& v, const Launch& L) {
    if (kpt >= 4) commit_kv<4, VAL>(t, keys, n, idx, mask, v, L);
    else if (kpt == 2) commit_kv<2, VAL>(t, keys, n, idx, mask, v, L);
    else commit_kv<1, VAL>(t, keys, n, idx, mask, v, L);
  }
  // v == nullptr: no inline value copy.
  template <class In>
  static void commit_in(int kpt, const TableView& t, const In& keys, int64_t n, int32_t* idx, uint8_t* mask,
                        const ValueRow* v, const Launch& L) {
    if (v) commit_v<true>(kpt, t, keys, n, idx, mask, *v, L);
    else commit_v<false>(kpt, t, keys, n, idx, mask, ValueRow{}, L);
  }
  static void commit(int kpt, const TableView& t, const int32_t* keys, int64_t n, int32_t* idx, uint8_t* mask,
                     const ValueRow* v, const Launch& L) {
    commit_in(kpt, t, keys, n, idx, mask, v, L);
  }
  static void commit_pts(int kpt, const TableView& t, const PointRows& p, int64_t n, int32_t* idx, uint8_t* mask,
                         const ValueRow* v, const Launch& L) {
    commit_in(kpt, t, p, n, idx, mask, v, L);
  }
  template <int S>
  static void erase_mark_s(const TableView& t, const int32_t* keys, int64_t n, int32_t* slot_out, const Launch& L) {
    TraceScope ts(kKEraseMark, L.stream);
    launch_dependent(erase_mark_kernel<D, S>, grid_for(n, L), L.block, L.stream, t, keys, n, slot_out);
  }
  static void erase_mark(int S, const TableView& t, const int32_t* keys, int64_t n, int32_t* slot_out, const Launch& L) {
    if (S == 4) erase_mark_s<4>(t, keys, n, slot_out, L);
    else if (S == 8) erase_mark_s<8>(t, keys, n, slot_out, L);
    else erase_mark_s<16>(t, keys, n, slot_out, L);
  }
  template <int S>
  static void rebuild_s(const TableView& t, const int32_t* kb_src, const int32_t* list, int64_t n,
                        int count, int preserve, int copy_keys, const Launch& L) {
    TraceScope ts(kKRebuild, L.stream);
    launch_dependent(rebuild_kernel<D, S>, grid_for(n, L), L.block, L.stream, t, kb_src, list, n, count, preserve,
                     copy_keys);
  }
  static void rebuild(int S, const TableView& t, const int32_t* kb_src, const int32_t* list, int64_t n,
                      int count, int preserve, int copy_keys, const Launch& L) {
    if (S == 4) rebuild_s<4>(t, kb_src, list, n, count, preserve, copy_keys, L);
    else if (S == 8) rebuild_s<8>(t, kb_src, list, n, count, preserve, copy_keys, L);
    else rebuild_s<16>(t, kb_src, list, n, count, preserve, copy_keys, L);
  }
  template <int S, class Off>
  static void neighbors_s(const TableView& t, const int32_t* keys, int64_t n, const Off& off, int64_t n_off,
                          int32_t* idx, uint8_t* mask, const Launch& L) {
    TraceScope ts(kKNeighbors, L.stream);
    constexpr int U = kNeighborUnroll;
    constexpr auto k = neighbors_kernel<D, S, U, Off>;
    launch_dependent(k, resident_grid<k>(grid_for((n * n_off + U - 1) / U, L), L), L.block, L.stream, t, keys, n, off,
                     static_cast<uint32_t>(n_off), idx, mask);
  }
  template <class Off>
  static void neighbors_off(int S, const TableView& t, const int32_t* keys, int64_t n, const Off& off, int64_t n_off,
                            int32_t* idx, uint8_t* mask, const Launch& L) {
    if (S == 4) neighbors_s<4>(t, keys, n, off, n_off, idx, mask, L);
    else if (S == 8) neighbors_s<8>(t, keys, n, off, n_off, idx, mask, L);
    else neighbors_s<16>(t, keys, n, off, n_off, idx, mask, L);
  }
  static void neighbors(int S, const TableView& t, const int32_t* keys, int64_t n, int radius, int64_t n_off,
                        int32_t* idx, uint8_t* mask, const Launch& L) {
    const uint32_t width = 2 * static_cast<uint32_t>(radius) + 1;
    const uint32_t magic = width > 1 ? static_cast<uint32_t>(((uint64_t{1} << 32) + width - 1) / width) : 0u;
    neighbors_off(S, t, keys, n, RadiusOffsets{static_cast<uint32_t>(radius), width, magic}, n_off, idx, mask, L);
  }
  static void offsets(int S, const TableView& t, const int32_t* keys, int64_t n, const int32_t* off, int64_t n_off,
                      int32_t* idx, uint8_t* mask, const Launch& L) {
    neighbors_off(S, t, keys, n, TableOffsets{off}, n_off, idx, mask, L);
  }
  template <int S>
  static void find_link_s(const TableView& t, const int32_t* keys, int64_t n, int32_t* idx, int32_t* link,
                          const int32_t* link_at, const Launch& L) {
    TraceScope ts(kKFind, L.stream);
    launch_dependent(find_link_kernel<D, S>, grid_for(n, L), L.block, L.stream, t, keys, n, idx, link, link_at);
  }
  static void find_link(int S, const TableView& t, const int32_t* keys, int64_t n, int32_t* idx, int32_t* link,
                        const int32_t* link_at, const Launch& L) {
    if (S == 4) find_link_s<4>(t, keys, n, idx, link, link_at, L);
    else if (S == 8) find_link_s<8>(t, keys, n, idx, link, link_at, L);
    else find_link_s<16>(t, keys, n, idx, link, link_at, L);
  }
  template <int S>
  static void find_group_s(const TableView& t, const int32_t* keys, int64_t n, int32_t* idx, uint8_t* mask,
                           const Launch& L) {
    TraceScope ts(kKFind, L.stream);
    constexpr int kKeysPerBlock = 256 / (S / 2);
    int64_t g = (n + kKeysPerBlock - 1) / kKeysPerBlock;
    if (g > L.grid_cap) g = L.grid_cap;
    find_group_kernel<D, S><<<static_cast<int>(g < 1 ? 1 : g), 256, 0, L.stream>>>(t, keys, n, idx, mask);
  }
  static void find_group(int S, const TableView& t, const int32_t* keys, int64_t n, int32_t* idx, uint8_t* mask,
                         const Launch& L) {
    if (S == 4) find_group_s<4>(t, keys, n, idx, mask, L);
    else if (S == 8) find_group_s<8>(t, keys, n, idx, mask, L);
    else find_group_s<16>(t, keys, n, idx, mask, L);
  }
  // counts: partition_count_words(n, log_p, L) words; ranges: n bytes;
  // keys_out: n rows; dest: n.  False when the device refuses a step (its
  // opt-in to the scatter's shared memory, or a launch): the outputs are then
  // not to be used.
  static bool partition(const int32_t* keys, int64_t n, int log_p, uint32_t* counts, uint8_t* ranges,
                        int32_t* keys_out, int32_t* dest, const Launch& L) {
    int tpb = 0;
    const int G = partition_grid(n, L, &tpb);
    const int P = 1 << log_p;
    uint32_t* range_totals = counts + static_cast<int64_t>(P) * G;
    // Above 48 KB with the static arrays (4 dimensions with 256 ranges, or 5
    // and more) the kernel must opt in, on each device.  The call is cheap
    // beside the 10^6 keys that a ranged call has, so nothing is remembered;
    // always the dimension's most, so that concurrent calls ask for the same.
    const size_t smem = partition_scatter_smem<D>(P);
    if (smem > 44 * 1024 && cudaFuncSetAttribute(partition_scatter_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 static_cast<int>(partition_scatter_smem<D>(1 << kPartMaxLog))) !=
                                cudaSuccess)
      return false;
    TraceScope ts(kKPartition, L.stream, 3);
    return launch_dependent(partition_count_kernel<D>, G, kCountThreads, L.stream, keys, n, log_p, tpb, counts,
                            ranges) == cudaSuccess &&
           launch_partition_scan(counts, G, P, range_totals, L) == cudaSuccess &&
           launch_dependent_smem(partition_scatter_kernel<D>, G, kScatterThreads, smem, L.stream, keys,
                                 static_cast<const uint8_t*>(ranges), n, log_p, tpb,
                                 static_cast<const uint32_t*>(counts), static_cast<const uint32_t*>(range_totals),
                                 keys_out, dest) == cudaSuccess;
  }
  static DimKernels table() {
    DimKernels k;
    k.partition = &partition;
    k.neighbors = &neighbors;
    k.offsets = &offsets;
    k.find_group = &find_group;
    k.find_link = &find_link;
    k.find_pts = &find_pts;
    k.claim_pts = &claim_pts;
    k.commit_pts = &commit_pts;
    k.find = &find;
    k.claim = &claim;
    k.commit = &commit;
    k.erase_mark = &erase_mark;
    k.rebuild = &rebuild;
    return k;
  }
};

// Defined in ash_dim.cu (one translation unit per key dimension).
DimKernels dim_kernels_1();
DimKernels dim_kernels_2();
DimKernels dim_kernels_3();
DimKernels dim_kernels_4();
DimKernels dim_kernels_5();
DimKernels dim_kernels_6();
DimKernels dim_kernels_7();
DimKernels dim_kernels_8();

// Defined in ash_aux.cu.
void launch_erase_resolve(int S, const TableView& t, int64_t n, const int32_t* slot_in, uint8_t* mask, const Launch& L);

}  // namespace ash
