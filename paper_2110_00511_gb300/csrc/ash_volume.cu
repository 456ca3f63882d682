// Geometry consumers of the hash map (Sec. 6.2 of the ASH paper):
//   * block keys of a depth frame: pinhole unprojection, then Eq. (11);
//   * the double hash map block allocation (local activate -> the frame's
//     distinct new keys -> global activate + find -> local values := global
//     indices), with an ordered compaction between the two maps;
//   * TSDF integration over hashed voxel blocks: projection and signed
//     distance (Eq. (7)), truncation, the running mean of Eq. (9);
//   * ray casting through the hashed blocks, optionally through the frame's
//     local map (the speed-up described with the double hash map).
//
// Every step that decides something discrete (a pixel, a skip, a voxel, a
// zero crossing) is written with explicitly rounded float32 intrinsics
// (__fmul_rn / __fadd_rn / __fdiv_rn: no contraction into fused
// multiply-adds) in a fixed operation order, so the decisions are
// reproducible bit for bit by any IEEE float32 implementation of the same
// steps.
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

#include "ash.h"
#include "ash_internal.h"
#include "ash_trace.h"

namespace ash {
namespace vol {

constexpr int kThreads = 256;
constexpr int kItems = 2;
constexpr int kTile = kThreads * kItems;  // items per compaction tile
constexpr int kScanThreads = 1024;

// Pinhole intrinsics and a world-to-camera pose [R | t] (row-major 3x4).
struct Cam {
  float fx, fy, cx, cy;
  float e[12];
};

__device__ __forceinline__ float rot_t_row(const Cam& k, int a, float x, float y, float z) {
  // (R^T v)_a = ((R_0a x + R_1a y) + R_2a z)
  return __fadd_rn(__fadd_rn(__fmul_rn(k.e[a], x), __fmul_rn(k.e[4 + a], y)), __fmul_rn(k.e[8 + a], z));
}

// Camera centre c = -R^T t.
__device__ __forceinline__ void camera_centre(const Cam& k, float (&c)[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) c[a] = -rot_t_row(k, a, k.e[3], k.e[7], k.e[11]);
}

// x_c = R x + t, row by row: ((r0 x + r1 y) + r2 z) + t.
__device__ __forceinline__ float transform_row(const Cam& k, int a, float x, float y, float z) {
  return __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(k.e[4 * a], x), __fmul_rn(k.e[4 * a + 1], y)),
                             __fmul_rn(k.e[4 * a + 2], z)),
                   k.e[4 * a + 3]);
}

__device__ __forceinline__ bool depth_valid(float d, float depth_max) { return d > 0.0f && d <= depth_max; }

// ------------------------------------------------------ ordered compaction
// Per-tile counts, then a write pass in which every tile places its flagged
// items at its offset in input order.  Tiles are kTile consecutive items; item
// q * kThreads + tid of a tile belongs to thread tid, so loads stay coalesced
// and the rank order (q, then tid) is input order.  Up to kSummedTiles tiles,
// each block of the write pass adds up the counts before its own (16 KB from
// L2 at most) and the last one writes the total, to the host too when it
// waits for it; above, a one-block scan of the counts comes between.  Launches
// and the copy of the count to the host are most of a call on an image: 640 x
// 480 pixels 33 us with the wait for the count, 50 with three launches and a
// copy.
constexpr int64_t kSummedTiles = 4096;

template <class Pred>
__global__ void __launch_bounds__(kThreads) tile_count_kernel(Pred pred, int64_t n, int32_t* __restrict__ tile_count) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ int s_warp[kThreads / 32 + 1];
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kTile;
  int c = 0;
#pragma unroll
  for (int q = 0; q < kItems; ++q) {
    const int64_t i = base + q * kThreads + threadIdx.x;
    c += (i < n && pred(i)) ? 1 : 0;
  }
  int total = 0;
  block_exclusive_scan(c, total, s_warp);
  if (threadIdx.x == 0) tile_count[blockIdx.x] = total;
}

// Exclusive scan of n_tiles counts in place; the grand total goes to *total
// (and *host).
__global__ void __launch_bounds__(kScanThreads) tile_scan_kernel(int32_t* __restrict__ tile, int64_t n_tiles,
                                                                 int64_t* __restrict__ total, int64_t* host) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ int s_warp[kScanThreads / 32 + 1];
  int64_t carry = 0;
  for (int64_t base = 0; base < n_tiles; base += kScanThreads) {
    const int64_t i = base + threadIdx.x;
    const int v = i < n_tiles ? tile[i] : 0;
    int chunk = 0;
    const int off = block_exclusive_scan(v, chunk, s_warp);
    if (i < n_tiles) tile[i] = static_cast<int32_t>(carry + off);
    carry += chunk;
    __syncthreads();  // s_warp is reused by the next chunk
  }
  if (threadIdx.x == 0) {
    *total = carry;
    if (host) *host = carry;
  }
}

// SUMMED: tile holds the counts, else their exclusive scan (total and host
// unused then).
template <class Pred, class Write, bool SUMMED>
__global__ void __launch_bounds__(kThreads) tile_write_kernel(Pred pred, Write write, int64_t n,
                                                              const int32_t* __restrict__ tile,
                                                              int64_t* __restrict__ total, int64_t* host) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ int s_warp[kThreads / 32 + 1];
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kTile;
  int64_t out = 0;
  if constexpr (SUMMED) {
    int sum = 0;
    for (int i = threadIdx.x; i < static_cast<int>(blockIdx.x); i += kThreads) sum += __ldg(tile + i);
    int before = 0;
    block_exclusive_scan(sum, before, s_warp);
    out = before;
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
      *total = out + tile[blockIdx.x];
      if (host) *host = out + tile[blockIdx.x];
    }
    __syncthreads();  // s_warp is reused below
  } else {
    out = tile[blockIdx.x];
  }
#pragma unroll 1
  for (int q = 0; q < kItems; ++q) {
    const int64_t i = base + q * kThreads + threadIdx.x;
    const bool f = i < n && pred(i);
    int rank = 0, total_q = 0;
    block_rank(f, rank, total_q, s_warp);
    if (f) write(i, out + rank);
    out += total_q;
    __syncthreads();  // s_warp is reused by the next round
  }
}

// ------------------------------------------------------ depth -> block keys
struct DepthValid {
  const float* depth;
  float depth_max;
  __device__ bool operator()(int64_t i) const { return depth_valid(__ldg(depth + i), depth_max); }
};

// Pixel i = py * width + px with depth D: camera point
// [(px - cx) / fx * D, (py - cy) / fy * D, D], world point R^T x_c + c, block
// key floor(x_w / edge) (Eq. (11)).
struct DepthKeyWrite {
  const float* depth;
  Cam cam;
  int32_t width;
  float edge;
  int32_t* keys;
  __device__ void operator()(int64_t i, int64_t o) const {
    const float d = __ldg(depth + i);
    const int32_t py = static_cast<int32_t>(i / width);
    const int32_t px = static_cast<int32_t>(i - static_cast<int64_t>(py) * width);
    const float xc = __fmul_rn(__fdiv_rn(__fsub_rn(static_cast<float>(px), cam.cx), cam.fx), d);
    const float yc = __fmul_rn(__fdiv_rn(__fsub_rn(static_cast<float>(py), cam.cy), cam.fy), d);
    float c[3];
    camera_centre(cam, c);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float xw = __fadd_rn(rot_t_row(cam, a, xc, yc, d), c[a]);
      keys[o * 3 + a] = static_cast<int32_t>(floorf(__fdiv_rn(xw, edge)));
    }
  }
};

// ------------------------------------------------------ double hash map
struct MaskSet {
  const uint8_t* mask;
  __device__ bool operator()(int64_t i) const { return __ldg(mask + i) != 0; }
};

struct UniqueWrite {
  const int32_t* keys;
  const int32_t* idx;
  int key_dim;
  int32_t* unique_keys;
  int32_t* local_idx;
  __device__ void operator()(int64_t i, int64_t o) const {
    for (int j = 0; j < key_dim; ++j) unique_keys[o * key_dim + j] = __ldg(keys + i * key_dim + j);
    local_idx[o] = __ldg(idx + i);
  }
};

// local value row li[r] := global index gi[r] (int32 rows).
__global__ void __launch_bounds__(kThreads) scatter_index_kernel(int32_t* __restrict__ local_values,
                                                                 const int32_t* __restrict__ li,
                                                                 const int32_t* __restrict__ gi, int64_t u) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int64_t r = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; r < u;
       r += static_cast<int64_t>(gridDim.x) * blockDim.x)
    local_values[__ldg(li + r)] = __ldg(gi + r);
}

// ------------------------------------------------------ TSDF integration
// One CTA per listed block.  Voxel slot v = (vz * ELL + vy) * ELL + vx (x
// fastest) is handled by thread v mod kThreads, so the value rows are read
// and written in coalesced runs (every row is read; only updated voxels are
// written).  For voxel g = K * ELL + v at x = g * s:
// x_c = R x + t; skipped when z_c <= 0, when the pixel
// (floor(fx * (x_c / z_c) + cx + 1/2), likewise v) is outside the image, when
// the depth there is missing or beyond depth_max, or when
// d^j = D - z_c < -mu.  Otherwise d := (w d + Psi) / (w + 1), w := w + 1 with
// Psi = min(d^j, mu) (Eq. (9) with w^j = 1).
template <int ELL>
__global__ void __launch_bounds__(kThreads) integrate_kernel(const int32_t* __restrict__ kb, int ks, int32_t capacity,
                                                             const int32_t* __restrict__ block_idx,
                                                             float* __restrict__ tsdf, float* __restrict__ weight,
                                                             const float* __restrict__ depth, int32_t width,
                                                             int32_t height, Cam cam, float voxel, float trunc,
                                                             float depth_max) {
  constexpr int kVox = ELL * ELL * ELL;
  constexpr int kPer = kVox / kThreads;  // voxels per thread (2 for 8^3, 16 for 16^3)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int32_t bi = __ldg(block_idx + blockIdx.x);
  if (bi < 0 || bi >= capacity) return;
  float* trow = tsdf + static_cast<int64_t>(bi) * kVox;
  float* wrow = weight + static_cast<int64_t>(bi) * kVox;
  // the rows' loads go out together with the key's; they do not depend on it
  float dv[kPer], wv[kPer];
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    dv[q] = trow[threadIdx.x + q * kThreads];
    wv[q] = wrow[threadIdx.x + q * kThreads];
  }
  const int32_t* key = kb + static_cast<int64_t>(bi) * ks;
  const uint32_t k0 = static_cast<uint32_t>(__ldg(key)) * ELL;
  const uint32_t k1 = static_cast<uint32_t>(__ldg(key + 1)) * ELL;
  const uint32_t k2 = static_cast<uint32_t>(__ldg(key + 2)) * ELL;
  const float fw = static_cast<float>(width), fh = static_cast<float>(height);
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int v = threadIdx.x + q * kThreads;
    const int vx = v % ELL, vy = (v / ELL) % ELL, vz = v / (ELL * ELL);
    const float x = __fmul_rn(static_cast<float>(static_cast<int32_t>(k0 + vx)), voxel);
    const float y = __fmul_rn(static_cast<float>(static_cast<int32_t>(k1 + vy)), voxel);
    const float z = __fmul_rn(static_cast<float>(static_cast<int32_t>(k2 + vz)), voxel);
    const float zc = transform_row(cam, 2, x, y, z);
    if (!(zc > 0.0f)) continue;
    const float xc = transform_row(cam, 0, x, y, z);
    const float yc = transform_row(cam, 1, x, y, z);
    const float uf = floorf(__fadd_rn(__fadd_rn(__fmul_rn(cam.fx, __fdiv_rn(xc, zc)), cam.cx), 0.5f));
    const float vf = floorf(__fadd_rn(__fadd_rn(__fmul_rn(cam.fy, __fdiv_rn(yc, zc)), cam.cy), 0.5f));
    if (!(uf >= 0.0f && uf < fw && vf >= 0.0f && vf < fh)) continue;
    // uf, vf are in [0, 2^31): 32-bit conversions (64-bit ones run on the FP64 pipe)
    const float dm = __ldg(depth + static_cast<int64_t>(static_cast<int32_t>(vf)) * width + static_cast<int32_t>(uf));
    if (!depth_valid(dm, depth_max)) continue;
    const float sdf = __fsub_rn(dm, zc);
    if (sdf < -trunc) continue;
    const float psi = fminf(sdf, trunc);
    const float den = __fadd_rn(wv[q], 1.0f);
    trow[v] = __fdiv_rn(__fadd_rn(__fmul_rn(wv[q], dv[q]), psi), den);
    wrow[v] = den;
  }
}

// ------------------------------------------------------ per-tile depth range
// The min-max range estimate of Sec. 6.2: the live blocks of the map a ray
// casting looks up are projected into tiles of kRangeTile x kRangeTile
// pixels, each tile keeping the least and greatest camera depth any of those
// blocks reaches over it.  A ray then samples only inside its tile's range.
// The estimate is conservative, so the result is unchanged: a block's cell of
// samples (the lattice points within half a voxel of it) is widened by half
// a voxel more, its corners' pixel rectangle by one pixel, and a cell that
// reaches the camera plane covers every tile from depth 0.  Samples outside
// every listed cell read missing blocks, which are invalid.
constexpr int kRangeTile = 8;

// Occupancy of the block lattice, wrapped to 128 blocks per axis (one bit per
// block), and of its cells of 4 x 4 x 4 blocks.  A clear bit proves a block (or
// a whole cell) missing; a set one may stand for another block 128 away.
constexpr int kOccBits = 7;
constexpr int kOccCell = 2;  // log2 blocks per cell edge
constexpr int kOccFineWords = 1 << (3 * kOccBits - 5);
constexpr int kOccWords = kOccFineWords + (1 << (3 * (kOccBits - kOccCell) - 5));

template <int BITS>
__device__ __forceinline__ uint32_t occ_bit(int32_t x, int32_t y, int32_t z) {
  constexpr uint32_t M = (1u << BITS) - 1u;
  return (((static_cast<uint32_t>(z) & M) << BITS | (static_cast<uint32_t>(y) & M)) << BITS) | (static_cast<uint32_t>(x) & M);
}

__device__ __forceinline__ uint32_t fine_bit(const int32_t (&K)[3]) { return occ_bit<kOccBits>(K[0], K[1], K[2]); }

__device__ __forceinline__ uint32_t cell_bit(const int32_t (&K)[3]) {
  return 32u * kOccFineWords + occ_bit<kOccBits - kOccCell>(K[0] >> kOccCell, K[1] >> kOccCell, K[2] >> kOccCell);
}

__global__ void range_reset_kernel(unsigned int* __restrict__ zmin, unsigned int* __restrict__ zmax, int n_tiles,
                                   uint32_t* __restrict__ occupied, unsigned long long* __restrict__ next_chunk) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  const int stride = gridDim.x * blockDim.x;
  if (tid == 0) *next_chunk = 0ull;
  for (int i = tid; i < kOccWords / 4; i += stride) reinterpret_cast<uint4*>(occupied)[i] = make_uint4(0u, 0u, 0u, 0u);
  for (int i = tid; i < n_tiles; i += stride) {
    zmin[i] = 0x7F800000u;  // +inf: no block over this tile yet
    zmax[i] = 0u;
  }
}

__device__ __forceinline__ float min_of_8(float v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o, 8));
  return v;
}

__device__ __forceinline__ float max_of_8(float v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o, 8));
  return v;
}

// Warp per live block: lane c (mod 8) projects corner c, then the lanes share
// out the tiles under the block.  live == nullptr: the live blocks are kB rows
// 0..t-1 (identity heap), else the first *count_dev entries of `live`, n_max
// at most.  Depths are positive, so their float bit patterns order like the
// values and integer atomics keep the extremes.  Each block also sets its
// occupancy bits; zmin == nullptr: nothing else.  (A thread per block, going
// through corners and tiles one after the other, took 11.5 us for 2000 blocks
// and few of the chip's warps.)
__global__ void __launch_bounds__(kThreads) block_range_kernel(const int32_t* __restrict__ kb, int ks, int ell,
                                                               const Ctrl* __restrict__ ctrl,
                                                               const int32_t* __restrict__ live, int64_t n_max,
                                                               const int64_t* __restrict__ count_dev, Cam cam,
                                                               float voxel, int32_t width, int32_t height,
                                                               int tiles_x, int tiles_y, unsigned int* __restrict__ zmin,
                                                               unsigned int* __restrict__ zmax,
                                                               uint32_t* __restrict__ occupied) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  int64_t n = live ? *count_dev : static_cast<int64_t>(static_cast<uint32_t>(ctrl->top_used));
  if (n > n_max) n = n_max;
  const int lane = threadIdx.x & 31;
  const int64_t n_warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
  for (int64_t r = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); r < n; r += n_warps) {
    const int32_t* key = kb + (live ? static_cast<int64_t>(__ldg(live + r)) : r) * ks;
    bool far_out = false;  // beyond |g| < 2^18 the margins are not proven: cover everything
    const int32_t K[3] = {__ldg(key), __ldg(key + 1), __ldg(key + 2)};
    if (lane < 2) {
      const uint32_t bit = lane == 0 ? fine_bit(K) : cell_bit(K);
      atomicOr(occupied + (bit >> 5), 1u << (bit & 31));
    }
    if (zmin == nullptr) continue;
    float at[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int32_t kk = K[a];
      far_out |= (kk >= (1 << 18) / ell || kk <= -(1 << 18) / ell);
      const float k = static_cast<float>(kk) * static_cast<float>(ell);
      at[a] = (lane >> a) & 1 ? (k + static_cast<float>(ell)) * voxel : (k - 1.0f) * voxel;
    }
    const float xc = cam.e[0] * at[0] + cam.e[1] * at[1] + cam.e[2] * at[2] + cam.e[3];
    const float yc = cam.e[4] * at[0] + cam.e[5] * at[1] + cam.e[6] * at[2] + cam.e[7];
    const float zc = cam.e[8] * at[0] + cam.e[9] * at[1] + cam.e[10] * at[2] + cam.e[11];
    const bool corner_behind = zc <= 1.0e-6f;
    const float u = cam.fx * (xc / zc) + cam.cx, v = cam.fy * (yc / zc) + cam.cy;
    const float z_lo = min_of_8(fminf(3.0e38f, zc));
    float z_hi = max_of_8(fmaxf(-3.0e38f, zc));
    const float u_lo = min_of_8(corner_behind ? 3.0e38f : fminf(3.0e38f, u));
    const float u_hi = max_of_8(corner_behind ? -3.0e38f : fmaxf(-3.0e38f, u));
    const float v_lo = min_of_8(corner_behind ? 3.0e38f : fminf(3.0e38f, v));
    const float v_hi = max_of_8(corner_behind ? -3.0e38f : fmaxf(-3.0e38f, v));
    const bool behind = __any_sync(0xFFFFFFFFu, corner_behind);
    if (!far_out && !(z_hi > 0.0f)) continue;  // wholly behind the camera: no sample (t > 0) reaches it
    int tx0, tx1, ty0, ty1;
    unsigned int zl;
    if (far_out) z_hi = __uint_as_float(0x7F800000u);
    if (behind || far_out) {
      tx0 = 0;
      ty0 = 0;
      tx1 = tiles_x - 1;
      ty1 = tiles_y - 1;
      zl = 0u;
    } else {
      const float px0 = fmaxf(floorf(u_lo) - 1.0f, 0.0f), px1 = fminf(ceilf(u_hi) + 1.0f, width - 1.0f);
      const float py0 = fmaxf(floorf(v_lo) - 1.0f, 0.0f), py1 = fminf(ceilf(v_hi) + 1.0f, height - 1.0f);
      if (!(px0 <= px1 && py0 <= py1)) continue;  // outside the image (or not finite)
      tx0 = static_cast<int>(px0) / kRangeTile;
      tx1 = static_cast<int>(px1) / kRangeTile;
      ty0 = static_cast<int>(py0) / kRangeTile;
      ty1 = static_cast<int>(py1) / kRangeTile;
      zl = __float_as_uint(fmaxf(z_lo, 0.0f));
    }
    const unsigned int zh = __float_as_uint(z_hi);
    const int nx = tx1 - tx0 + 1;
    const int n_over = nx * (ty1 - ty0 + 1);
    for (int j = lane; j < n_over; j += 32) {
      const int tile = (ty0 + j / nx) * tiles_x + tx0 + j % nx;
      atomicMin(zmin + tile, zl);
      atomicMax(zmax + tile, zh);
    }
  }
}

// ------------------------------------------------------ ray casting
// Thread per pixel.  The ray of pixel (px, py) leaves the camera centre along
// R^T [(px - cx) / fx, (py - cy) / fy, 1]; sample i sits at depth
// t_i = depth_min + i * step, at p = c + t_i * dir, and reads the nearest
// lattice point g = floor(p / s + 1/2) (IEEE float32 division) in block K = floor(g / ELL),
// voxel v = g - K * ELL.  A sample is valid when K is in the map and its
// weight is positive.  The first valid pair d_{i-1} > 0 >= d_i gives the depth
// t_{i-1} + step * d_{i-1} / (d_{i-1} - d_i); 0 when there is none.  With a
// local index map, K is looked up there and its int32 value row names the
// block's index in the volume's buffers.
//
// Two shortcuts leave the result unchanged.  A block is looked up once for all
// consecutive samples in it.  And every rounding step of the sample arithmetic
// is monotone, so each coordinate of g, of K and of K's 4 x 4 x 4 cell is
// monotone in i: if samples i and m > i fall in the same block (or cell), so
// do all samples between them.  When the occupancy bits or the lookup show
// that the block or its cell is missing, the kernel estimates the last sample
// m inside it from the ray's exit, recomputes sample m exactly as above, and
// when it still falls there jumps over the samples up to m (all invalid by
// definition).
//
// What bounds it: the serial chain of each ray (sample -> block -> voxel
// loads), few rays being much longer than the rest, and the issue slots of
// the sample arithmetic.  So a ray takes kRaySamples consecutive samples at
// once, loads the voxels of those that share the first one's block together
// and looks at them in order; the division by the voxel size, three per
// sample, is three instructions (divide_by_voxel); and a warp takes 8 x 4
// pixels, whose rays pass much the same blocks under one depth range.  Empty
// space is passed by occupancy bits (two loads that mostly hit L1, no hash),
// a cell of blocks at a time where it is empty: rays past a sphere's edge made
// 40-70 lookups each and set the kernel's time.  GB300, 640 x 480 rays, 2000
// live blocks, up to 850 samples per ray: 164 us -> 117 (tiles, division,
// samples together) -> 73 (occupancy); 2, 3, 6 samples at once 75, 75, 83.
//
// x / b correctly rounded from y = 1 / b correctly rounded (Markstein, IBM J.
// Res. Dev. 34, 1990): q = x y is within 1.5 ulp of the quotient, the remainder
// x - b q takes 25 bits at most, so one fused multiply-add gives it to a unit
// in its last place, and q + remainder * y before its rounding is off by less
// than 2.5 ulp(q) / b (mantissas as integers).  Only quotients that close to a
// midpoint of two floats could round the other way; of all pairs of mantissas
// none does (the test enumerates them).  Over- and underflow change nothing
// here: only floor(q + 1/2) is used, which is 0 for every tiny quotient, and a
// quotient past the range is refused whether it is huge, infinite or NaN.  y
// itself has to be a normal number: for voxel sizes outside [2^-60, 2^60] the
// division is made by __fdiv_rn (MUL false).
template <bool MUL>
__device__ __forceinline__ float divide_by_voxel(float x, float voxel, float inv_voxel) {
  if constexpr (!MUL) return __fdiv_rn(x, voxel);
  const float q = __fmul_rn(x, inv_voxel);
  return __fmaf_rn(__fmaf_rn(-q, voxel, x), inv_voxel, q);
}

struct RaySample {
  int32_t g[3];
  bool in_range;
};

// i < 2^24, so the conversion to float32 is exact (and int32 keeps it off the
// 64-bit conversion path).
template <bool MUL>
__device__ __forceinline__ RaySample ray_sample(const float (&c)[3], const float (&dw)[3], float depth_min,
                                                float step, float voxel, float inv_voxel, int32_t i) {
  RaySample r;
  r.in_range = true;
  const float t = __fadd_rn(depth_min, __fmul_rn(__int2float_rn(i), step));
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float gf = floorf(__fadd_rn(divide_by_voxel<MUL>(__fadd_rn(c[a], __fmul_rn(t, dw[a])), voxel, inv_voxel), 0.5f));
    r.in_range &= fabsf(gf) < 1.0e9f;
    r.g[a] = r.in_range ? static_cast<int32_t>(gf) : 0;
  }
  return r;
}

constexpr int kRaySamples = 4;

template <int ELL, int S, bool MUL>
__device__ __forceinline__ float cast_ray(const TableView& tv, const TableView& local_tv,
                                          const int32_t* __restrict__ local_values, int use_local,
                                          const float* __restrict__ tsdf, const float* __restrict__ weight,
                                          const uint32_t* __restrict__ occupied,
                                          int32_t volume_capacity, const Cam& cam, int32_t px, int32_t py,
                                          float voxel, float inv_voxel, float depth_min, float step, float inv_step,
                                          int32_t i_begin, int32_t n_steps) {
  constexpr int kVox = ELL * ELL * ELL;
  constexpr int kShift = ELL == 8 ? 3 : 4;
  float c[3];
  camera_centre(cam, c);
  const float dcx = __fdiv_rn(__fsub_rn(static_cast<float>(px), cam.cx), cam.fx);
  const float dcy = __fdiv_rn(__fsub_rn(static_cast<float>(py), cam.cy), cam.fy);
  float dw[3], inv_dw[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    dw[a] = rot_t_row(cam, a, dcx, dcy, 1.0f);
    inv_dw[a] = __fdividef(1.0f, dw[a]);  // only for the skip estimate
  }

  int32_t K[3] = {0, 0, 0};
  int32_t bi = -1;  // block K's index in the volume, -1 until a block was found
  bool prev_valid = false;
  float prev_d = 0.0f;
  int32_t i = i_begin;
  while (true) {
    // 1. on to the next sample in a block that exists
    while (i < n_steps) {
      const RaySample r = ray_sample<MUL>(c, dw, depth_min, step, voxel, inv_voxel, i);
      if (r.in_range) {
#pragma unroll
        for (int a = 0; a < 3; ++a) K[a] = r.g[a] >> kShift;
        // missing: K's cell of blocks, or only K itself
        int shift = kShift + kOccCell;
        uint32_t bit = cell_bit(K);
        if ((__ldg(occupied + (bit >> 5)) >> (bit & 31)) & 1u) {
          shift = kShift;
          bit = fine_bit(K);
          if ((__ldg(occupied + (bit >> 5)) >> (bit & 31)) & 1u) {
            if (use_local) {
              const int32_t li = find_key<3, S>(local_tv, K);
              bi = li >= 0 ? __ldg(local_values + li) : -1;
            } else {
              bi = find_key<3, S>(tv, K);
            }
            if (bi >= 0 && bi < volume_capacity) break;
          }
        }
        // the ray's exit from what is missing: the lattice points [lo, lo + 2^shift) per axis
        const float t = __fadd_rn(depth_min, __fmul_rn(__int2float_rn(i), step));
        const float edge = static_cast<float>(1 << shift);
        float t_exit = 3.0e38f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const float lo = static_cast<float>((r.g[a] >> shift) << shift) - 0.5f;
          const float face = dw[a] > 0.0f ? lo + edge : lo;
          if (dw[a] != 0.0f) t_exit = fminf(t_exit, (face * voxel - c[a]) * inv_dw[a]);
        }
        const float est = floorf((t_exit - t) * inv_step);
        if (est >= 1.0f) {
          int32_t m = i + static_cast<int32_t>(fminf(est, static_cast<float>(n_steps)));
          if (m > n_steps - 1) m = n_steps - 1;
          // confirm with the exact sample arithmetic; one step back if the
          // estimate crossed the face
          for (int tries = 0; tries < 2 && m > i; ++tries, --m) {
            const RaySample rm = ray_sample<MUL>(c, dw, depth_min, step, voxel, inv_voxel, m);
            if (rm.in_range && (rm.g[0] >> shift) == (r.g[0] >> shift) && (rm.g[1] >> shift) == (r.g[1] >> shift) &&
                (rm.g[2] >> shift) == (r.g[2] >> shift)) {
              i = m;  // samples i+1..m are in the missing part
              break;
            }
          }
        }
      }
      prev_valid = false;
      ++i;
    }
    if (i >= n_steps) return 0.0f;
    // 2. its samples in that block, kRaySamples at a time
    const float* w_row = weight + static_cast<int64_t>(bi) * kVox;
    const float* d_row = tsdf + static_cast<int64_t>(bi) * kVox;
    int m = kRaySamples;
    while (m == kRaySamples) {
      int at[kRaySamples];
      m = 0;
#pragma unroll
      for (int q = 0; q < kRaySamples; ++q) {
        const RaySample r = ray_sample<MUL>(c, dw, depth_min, step, voxel, inv_voxel, i + q);
        at[q] = ((r.g[2] & (ELL - 1)) * ELL + (r.g[1] & (ELL - 1))) * ELL + (r.g[0] & (ELL - 1));
        const bool same = i + q < n_steps && r.in_range && (r.g[0] >> kShift) == K[0] && (r.g[1] >> kShift) == K[1] &&
                          (r.g[2] >> kShift) == K[2];
        if (same && m == q) m = q + 1;
      }
      float w[kRaySamples], d[kRaySamples];
#pragma unroll
      for (int q = 0; q < kRaySamples; ++q) {
        w[q] = q < m ? __ldg(w_row + at[q]) : 0.0f;
        d[q] = q < m ? __ldg(d_row + at[q]) : 0.0f;
      }
#pragma unroll
      for (int q = 0; q < kRaySamples; ++q) {
        if (q < m) {
          const bool valid = w[q] > 0.0f;
          if (valid && prev_valid && prev_d > 0.0f && d[q] <= 0.0f) {
            const float prev_t = __fadd_rn(depth_min, __fmul_rn(__int2float_rn(i + q - 1), step));
            return __fadd_rn(prev_t, __fmul_rn(step, __fdiv_rn(prev_d, __fsub_rn(prev_d, d[q]))));
          }
          prev_valid = valid;
          prev_d = d[q];
        }
      }
      i += m;
    }
  }
}

// Persistent grid; each warp takes the next 8 x 4 pixels (half a range tile)
// from a counter, so rays of uneven length do not leave the tail of the
// launch idle.  Each ray samples only i in [i_begin, i_end) from its tile's
// depth range, widened by two steps on either side; the sample before i_begin
// lies outside every listed cell, so starting there with no valid predecessor
// is the same as marching from 0.
template <int ELL, int S, bool MUL>
__global__ void __launch_bounds__(kThreads) raycast_kernel(TableView tv, TableView local_tv,
                                                           const int32_t* __restrict__ local_values, int use_local,
                                                           const float* __restrict__ tsdf,
                                                           const float* __restrict__ weight,
                                                           const uint32_t* __restrict__ occupied,
                                                           int32_t volume_capacity,
                                                           Cam cam, int32_t width, int32_t height, float voxel,
                                                           float inv_voxel, float depth_min, float step,
                                                           float inv_step, int32_t n_steps,
                                                           const unsigned int* __restrict__ zmin,
                                                           const unsigned int* __restrict__ zmax, int tiles_x,
                                                           int tiles_y, int use_range,
                                                           unsigned long long* __restrict__ next_chunk,
                                                           float* __restrict__ depth_out) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int lane = threadIdx.x & 31;
  const uint64_t n_chunks = static_cast<uint64_t>(tiles_x) * static_cast<uint64_t>(tiles_y) * 2u;
  while (true) {
    unsigned long long chunk = 0;
    if (lane == 0) chunk = atomicAdd(next_chunk, 1ull);
    chunk = __shfl_sync(0xFFFFFFFFu, chunk, 0);
    if (chunk >= n_chunks) break;
    const uint32_t tile = static_cast<uint32_t>(chunk >> 1);
    const int32_t ty = static_cast<int32_t>(tile / static_cast<uint32_t>(tiles_x));
    const int32_t tx = static_cast<int32_t>(tile) - ty * tiles_x;
    const int32_t px = tx * kRangeTile + (lane & 7);
    const int32_t py = ty * kRangeTile + static_cast<int32_t>(chunk & 1u) * 4 + (lane >> 3);
    int32_t i0 = 0, i1 = n_steps;
    if (use_range) {
      const float z0 = __uint_as_float(__ldg(zmin + tile));
      const float z1 = __uint_as_float(__ldg(zmax + tile));
      if (z0 <= z1) {
        const float f0 = floorf((z0 - depth_min) * inv_step) - 2.0f;
        const float f1 = ceilf((z1 - depth_min) * inv_step) + 2.0f;
        i0 = f0 <= 0.0f ? 0 : (f0 >= static_cast<float>(n_steps) ? n_steps : static_cast<int32_t>(f0));
        i1 = f1 >= static_cast<float>(n_steps) ? n_steps : (f1 <= 0.0f ? 0 : static_cast<int32_t>(f1));
      } else {
        i1 = 0;  // no listed block over this tile
      }
    }
    if (px < width && py < height)
      depth_out[static_cast<int64_t>(py) * width + px] =
          cast_ray<ELL, S, MUL>(tv, local_tv, local_values, use_local, tsdf, weight, occupied, volume_capacity, cam, px, py, voxel,
                           inv_voxel, depth_min, step, inv_step, i0, i1);
    __syncwarp();
  }
}

// ------------------------------------------------------ host side
using host::fail;

Cam cam_of(const float* intr, const float* extr) {
  Cam k;
  k.fx = intr[0];
  k.fy = intr[1];
  k.cx = intr[2];
  k.cy = intr[3];
  std::memcpy(k.e, extr, sizeof(k.e));
  return k;
}

void* scratch_alloc(size_t bytes, cudaStream_t st) {
  void* p = nullptr;
  if (cudaMallocAsync(&p, bytes, st) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return p;
}

// Ordered compaction with a caller-provided predicate and writer; the count
// lands in *count_dev, and in *count_host (mapped) unless null.  tile
// scratch: n_tiles int32.
template <class Pred, class Write>
void compact(Pred pred, Write write, int64_t n, int32_t* tile, int64_t* count_dev, int64_t* count_host,
             cudaStream_t st, int kind) {
  const int64_t n_tiles = (n + kTile - 1) / kTile;
  if (n_tiles == 0) {
    cudaMemsetAsync(count_dev, 0, sizeof(int64_t), st);
    if (count_host) *count_host = 0;
    return;
  }
  const int grid = static_cast<int>(n_tiles);
  TraceScope ts(kind, st, n_tiles <= kSummedTiles ? 2 : 3);
  launch_dependent(tile_count_kernel<Pred>, grid, kThreads, st, pred, n, tile);
  if (n_tiles <= kSummedTiles) {
    launch_dependent(tile_write_kernel<Pred, Write, true>, grid, kThreads, st, pred, write, n, tile, count_dev,
                     count_host);
  } else {
    launch_dependent(tile_scan_kernel, 1, kScanThreads, st, tile, n_tiles, count_dev, count_host);
    launch_dependent(tile_write_kernel<Pred, Write, false>, grid, kThreads, st, pred, write, n, tile, count_dev,
                     count_host);
  }
}

int ell_of(const ash_map* m, int j) {
  if (j < 0 || j >= m->n_values) return 0;
  if (m->row_bytes[j] == 4 * 8 * 8 * 8) return 8;
  if (m->row_bytes[j] == 4 * 16 * 16 * 16) return 16;
  return 0;
}

thread_local int64_t* t_pinned_count = nullptr;

int64_t* pinned_count() {
  if (!t_pinned_count) {
    if (cudaMallocHost(&t_pinned_count, sizeof(int64_t)) != cudaSuccess) {
      cudaGetLastError();
      t_pinned_count = nullptr;
    }
  }
  return t_pinned_count;
}

}  // namespace vol
}  // namespace ash

using namespace ash::host;
using ash::vol::Cam;

extern "C" {

ash_status ash_depth_to_block_keys(const float* depth, int32_t width, int32_t height, const float* intrinsics_host,
                                   const float* extrinsic_host, float block_edge, float depth_max, int32_t* keys,
                                   int64_t* count_dev, int64_t* count_host, ash_stream stream) {
  if (width < 0 || height < 0) return fail(ASH_ERR_INVALID, "width and height must be >= 0");
  const int64_t n = static_cast<int64_t>(width) * height;
  if (n >= (int64_t{1} << 31)) return fail(ASH_ERR_INVALID, "image too large");
  if (!intrinsics_host || !extrinsic_host) return fail(ASH_ERR_INVALID, "camera arguments are required");
  if (n > 0 && (!depth || !keys)) return fail(ASH_ERR_INVALID, "depth and keys are required");
  if (!count_dev && !count_host) return fail(ASH_ERR_INVALID, "count_dev or count_host is required");
  if (!(block_edge > 0.0f)) return fail(ASH_ERR_INVALID, "block_edge must be > 0");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int64_t n_tiles = (n + ash::vol::kTile - 1) / ash::vol::kTile;
  char* scratch = static_cast<char*>(ash::vol::scratch_alloc(16 + 4 * (n_tiles + 1), st));
  if (!scratch) return fail(ASH_ERR_OOM, "scratch allocation failed");
  int64_t* cnt = count_dev ? count_dev : reinterpret_cast<int64_t*>(scratch);
  int32_t* tile = reinterpret_cast<int32_t*>(scratch + 16);
  const Cam cam = ash::vol::cam_of(intrinsics_host, extrinsic_host);
  int64_t* pin = count_host ? ash::vol::pinned_count() : nullptr;
  ash_status s = count_host && !pin ? fail(ASH_ERR_OOM, "pinned allocation failed") : ASH_OK;
  if (s == ASH_OK) {
    ash::vol::compact(ash::vol::DepthValid{depth, depth_max},
                      ash::vol::DepthKeyWrite{depth, cam, width, block_edge, keys}, n, tile, cnt, pin, st,
                      ash::kKDepthKeys);
    s = check_launch("depth_to_block_keys");
  }
  if (s == ASH_OK && count_host) {
    const cudaError_t e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) s = cuda_fail(e, "depth_to_block_keys");
    else *count_host = *pin;
  }
  cudaFreeAsync(scratch, st);
  return s;
}

ash_status ash_double_map_activate(ash_map* local, ash_map* global, const int32_t* keys, int64_t n,
                                   int32_t* unique_keys, int32_t* local_indices, int32_t* global_indices,
                                   int64_t* n_unique_host, ash_stream stream) {
  if (!local || !global || local == global) return fail(ASH_ERR_INVALID, "two distinct maps are required");
  if (local->device != global->device) return fail(ASH_ERR_INVALID, "maps on different devices");
  if (local->key_dim != global->key_dim) return fail(ASH_ERR_INVALID, "maps with different key dimensions");
  if (local->n_values != 1 || local->row_bytes[0] != 4 || local->dtype[0] != ASH_I32)
    return fail(ASH_ERR_INVALID, "the local map needs exactly one int32 value buffer of one element");
  if (!n_unique_host) return fail(ASH_ERR_INVALID, "n_unique_host is required");
  ash_status s = check_keys(local, keys, n);
  if (s != ASH_OK) return s;
  *n_unique_host = 0;
  if (n == 0) return ASH_OK;
  if (!unique_keys || !local_indices || !global_indices) return fail(ASH_ERR_INVALID, "outputs are required");
  DeviceGuard g(local->device);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int64_t n_tiles = (n + ash::vol::kTile - 1) / ash::vol::kTile;
  // scratch: count (16 B) | tile counts | local indices (n) | masks (n)
  const size_t off_tile = 16, off_idx = off_tile + ((4 * n_tiles + 15) / 16) * 16, off_mask = off_idx + 4 * n;
  char* scratch = static_cast<char*>(ash::vol::scratch_alloc(off_mask + n, st));
  if (!scratch) return fail(ASH_ERR_OOM, "scratch allocation failed");
  int64_t* cnt = reinterpret_cast<int64_t*>(scratch);
  int32_t* tile = reinterpret_cast<int32_t*>(scratch + off_tile);
  int32_t* idx_all = reinterpret_cast<int32_t*>(scratch + off_idx);
  uint8_t* mask_all = reinterpret_cast<uint8_t*>(scratch + off_mask);
  int64_t u = 0;
  // 1. local activate
  s = ash_activate(local, keys, n, idx_all, mask_all, stream);
  // 2. the frame's distinct new keys, in input order
  int64_t* pin = ash::vol::pinned_count();
  if (s == ASH_OK && !pin) s = fail(ASH_ERR_OOM, "pinned allocation failed");
  if (s == ASH_OK) {
    ash::vol::compact(ash::vol::MaskSet{mask_all},
                      ash::vol::UniqueWrite{keys, idx_all, local->key_dim, unique_keys, local_indices}, n, tile, cnt,
                      pin, st, ash::kKCompact);
    s = check_launch("double_map_activate");
  }
  if (s == ASH_OK) {
    const cudaError_t e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) s = cuda_fail(e, "double_map_activate");
    else u = *pin;
  }
  // 3. global activate + find; 4. local values := global indices
  if (s == ASH_OK && u > 0) {
    s = ash_activate(global, unique_keys, u, global_indices, mask_all, stream);
    if (s == ASH_OK && global->tuning.warp_probe == 0 && partition_log(global, u) == 0) {
      // in one kernel: the lookup's thread links the local entry
      global->last_stream = st;
      global->K.find_link(global->S, view_of(global), unique_keys, u, global_indices,
                          static_cast<int32_t*>(local->vb[0]), local_indices, launch_of(global, st));
      s = check_launch("double_map_activate");
    } else if (s == ASH_OK) {
      s = ash_find(global, unique_keys, u, global_indices, mask_all, stream);
      if (s == ASH_OK) {
        ash::TraceScope ts(ash::kKScatterRows, st);
        ash::launch_dependent(ash::vol::scatter_index_kernel, grid_for(u, launch_of(local, st)), ash::vol::kThreads, st,
                              static_cast<int32_t*>(local->vb[0]), local_indices, global_indices, u);
        s = check_launch("double_map_activate");
      }
    }
  }
  cudaFreeAsync(scratch, st);
  if (s == ASH_OK) *n_unique_host = u;
  return s;
}

ash_status ash_tsdf_integrate(ash_map* blocks, int tsdf_buffer, int weight_buffer, const int32_t* block_indices,
                              int64_t n_blocks, const float* depth, int32_t width, int32_t height,
                              const float* intrinsics_host, const float* extrinsic_host, float voxel_size,
                              float trunc, float depth_max, ash_stream stream) {
  if (!blocks) return fail(ASH_ERR_INVALID, "map is NULL");
  if (blocks->key_dim != 3) return fail(ASH_ERR_INVALID, "the block map needs key_dim 3");
  const int ell = ash::vol::ell_of(blocks, tsdf_buffer);
  if (ell == 0 || ash::vol::ell_of(blocks, weight_buffer) != ell || tsdf_buffer == weight_buffer ||
      blocks->dtype[tsdf_buffer] != ASH_F32 || blocks->dtype[weight_buffer] != ASH_F32)
    return fail(ASH_ERR_INVALID, "tsdf and weight buffers must be distinct float32 rows of 8^3 or 16^3");
  if (n_blocks < 0 || n_blocks >= (int64_t{1} << 31)) return fail(ASH_ERR_INVALID, "n_blocks out of range");
  if (width <= 0 || height <= 0 || !depth) return fail(ASH_ERR_INVALID, "a depth image is required");
  if (!intrinsics_host || !extrinsic_host) return fail(ASH_ERR_INVALID, "camera arguments are required");
  if (!(voxel_size > 0.0f) || !(trunc > 0.0f)) return fail(ASH_ERR_INVALID, "voxel_size and trunc must be > 0");
  if (n_blocks == 0) return ASH_OK;
  if (!block_indices) return fail(ASH_ERR_INVALID, "block_indices is NULL");
  DeviceGuard g(blocks->device);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  blocks->last_stream = st;
  const Cam cam = ash::vol::cam_of(intrinsics_host, extrinsic_host);
  float* tsdf = static_cast<float*>(blocks->vb[tsdf_buffer]);
  float* weight = static_cast<float*>(blocks->vb[weight_buffer]);
  const int32_t cap = static_cast<int32_t>(blocks->capacity);
  ash::TraceScope ts(ash::kKIntegrate, st);
  if (ell == 8)
    ash::launch_dependent(ash::vol::integrate_kernel<8>, static_cast<int>(n_blocks), ash::vol::kThreads, st,
                          blocks->kb, blocks->ks, cap, block_indices, tsdf, weight, depth, width, height, cam,
                          voxel_size, trunc, depth_max);
  else
    ash::launch_dependent(ash::vol::integrate_kernel<16>, static_cast<int>(n_blocks), ash::vol::kThreads, st,
                          blocks->kb, blocks->ks, cap, block_indices, tsdf, weight, depth, width, height, cam,
                          voxel_size, trunc, depth_max);
  return check_launch("tsdf_integrate");
}

ash_status ash_tsdf_raycast(ash_map* blocks, int tsdf_buffer, int weight_buffer, ash_map* local_index_map,
                            const float* intrinsics_host, const float* extrinsic_host, int32_t width, int32_t height,
                            float voxel_size, float depth_min, float step, int64_t n_steps, float* depth_out,
                            ash_stream stream) {
  if (!blocks) return fail(ASH_ERR_INVALID, "map is NULL");
  if (blocks->key_dim != 3) return fail(ASH_ERR_INVALID, "the block map needs key_dim 3");
  const int ell = ash::vol::ell_of(blocks, tsdf_buffer);
  if (ell == 0 || ash::vol::ell_of(blocks, weight_buffer) != ell || blocks->dtype[tsdf_buffer] != ASH_F32 ||
      blocks->dtype[weight_buffer] != ASH_F32)
    return fail(ASH_ERR_INVALID, "tsdf and weight buffers must be float32 rows of 8^3 or 16^3");
  if (local_index_map) {
    if (local_index_map->key_dim != 3 || local_index_map->n_values != 1 || local_index_map->row_bytes[0] != 4 ||
        local_index_map->dtype[0] != ASH_I32 || local_index_map->device != blocks->device ||
        local_index_map->S != blocks->S)
      return fail(ASH_ERR_INVALID, "the local index map needs key_dim 3, one int32 value and the same bucket size");
  }
  if (width <= 0 || height <= 0) return fail(ASH_ERR_INVALID, "width and height must be > 0");
  const int64_t n_pix = static_cast<int64_t>(width) * height;
  if (n_pix >= (int64_t{1} << 31)) return fail(ASH_ERR_INVALID, "image too large");
  if (!depth_out || !intrinsics_host || !extrinsic_host) return fail(ASH_ERR_INVALID, "outputs and camera required");
  if (!(voxel_size > 0.0f) || !(step > 0.0f) || n_steps < 0 || n_steps > (int64_t{1} << 24))
    return fail(ASH_ERR_INVALID, "voxel_size and step must be > 0, n_steps in [0, 2^24]");
  DeviceGuard g(blocks->device);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  blocks->last_stream = st;
  const Cam cam = ash::vol::cam_of(intrinsics_host, extrinsic_host);
  const ash::TableView tv = view_of(blocks);
  const ash::TableView ltv = local_index_map ? view_of(local_index_map) : tv;
  const int32_t* lvals = local_index_map ? static_cast<const int32_t*>(local_index_map->vb[0]) : nullptr;
  const float* tsdf = static_cast<const float*>(blocks->vb[tsdf_buffer]);
  const float* weight = static_cast<const float*>(blocks->vb[weight_buffer]);
  const int32_t cap = static_cast<int32_t>(blocks->capacity);
  const int use_local = local_index_map ? 1 : 0;
  const float inv_step = 1.0f / step;
  // Markstein's division needs a normal reciprocal (divide_by_voxel)
  const bool mul = voxel_size >= 0x1p-60f && voxel_size <= 0x1p60f;
  const float inv_voxel = mul ? 1.0f / voxel_size : 0.0f;
  // scratch: chunk counter | live count | occupancy bits | tile zmin | tile
  // zmax | live indices (only listed when the live blocks are not simply rows
  // 0..t-1)
  ash_map* lookup = local_index_map ? local_index_map : blocks;
  const int tiles_x = (width + ash::vol::kRangeTile - 1) / ash::vol::kRangeTile;
  const int tiles_y = (height + ash::vol::kRangeTile - 1) / ash::vol::kRangeTile;
  const int n_tiles = tiles_x * tiles_y;
  const bool listed = !lookup->heap_identity;
  lookup->last_stream = st;
  const size_t off_tiles = 16 + 4 * static_cast<size_t>(ash::vol::kOccWords), off_live = off_tiles + ((8 * static_cast<size_t>(n_tiles) + 15) / 16) * 16;
  char* scratch = static_cast<char*>(
      ash::vol::scratch_alloc(off_live + (listed ? 4 * static_cast<size_t>(lookup->capacity) : 0), st));
  if (!scratch) return fail(ASH_ERR_OOM, "scratch allocation failed");
  unsigned long long* counter = reinterpret_cast<unsigned long long*>(scratch);
  int64_t* live_count = reinterpret_cast<int64_t*>(scratch + 8);
  uint32_t* occupied = reinterpret_cast<uint32_t*>(scratch + 16);
  unsigned int* zmin = reinterpret_cast<unsigned int*>(scratch + off_tiles);
  unsigned int* zmax = zmin + n_tiles;
  int32_t* live = listed ? reinterpret_cast<int32_t*>(scratch + off_live) : nullptr;
  // the per-tile depth range (Sec. 6.2's min-max estimate) needs samples at t > 0
  const int use_range = depth_min > 0.0f ? 1 : 0;
  if (listed) {
    ash_status ls = ash_get_active_indices_async(lookup, live, lookup->capacity, live_count, stream);
    if (ls != ASH_OK) {
      cudaFreeAsync(scratch, st);
      return ls;
    }
  }
  {
    ash::TraceScope tr(ash::kKRayRange, st, 2);
    ash::launch_dependent(ash::vol::range_reset_kernel, 65, 256, st, zmin, zmax, use_range ? n_tiles : 0, occupied,
                          counter);
    ash::launch_dependent(ash::vol::block_range_kernel, grid_for(lookup->capacity * 32, launch_of(lookup, st)),
                          ash::vol::kThreads, st, lookup->kb, lookup->ks, ell, lookup->ctrl, live, lookup->capacity,
                          live_count, cam, voxel_size, width, height, tiles_x, tiles_y, use_range ? zmin : nullptr,
                          zmax, occupied);
  }
  int dev = 0;
  cudaGetDevice(&dev);
  const int64_t warps_needed = static_cast<int64_t>(n_tiles) * 2;
  // one wave of resident blocks (all variants use about the same registers)
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ash::vol::raycast_kernel<8, 4, true>, ash::vol::kThreads, 0) !=
          cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    per_sm = 4;
  }
  int64_t grid64 = static_cast<int64_t>(sm_count(dev)) * per_sm;
  if (grid64 * (ash::vol::kThreads / 32) > warps_needed) grid64 = (warps_needed + 7) / 8;
  const unsigned grid = static_cast<unsigned>(grid64 < 1 ? 1 : grid64);
  ash::TraceScope ts(ash::kKRaycast, st);
#define ASH_RAYCAST_M(E, SB, M)                                                                                     \
  ash::launch_dependent(ash::vol::raycast_kernel<E, SB, M>, static_cast<int>(grid), ash::vol::kThreads, st, tv, ltv, \
                        lvals, use_local, tsdf, weight, occupied, cap, cam, width, height, voxel_size, inv_voxel,    \
                        depth_min, step, inv_step, static_cast<int32_t>(n_steps), zmin, zmax, tiles_x, tiles_y,      \
                        use_range, counter, depth_out)
#define ASH_RAYCAST(E, SB)           \
  if (mul) ASH_RAYCAST_M(E, SB, true); \
  else ASH_RAYCAST_M(E, SB, false)
  if (ell == 8) {
    if (blocks->S == 4) { ASH_RAYCAST(8, 4); }
    else if (blocks->S == 8) { ASH_RAYCAST(8, 8); }
    else { ASH_RAYCAST(8, 16); }
  } else {
    if (blocks->S == 4) { ASH_RAYCAST(16, 4); }
    else if (blocks->S == 8) { ASH_RAYCAST(16, 8); }
    else { ASH_RAYCAST(16, 16); }
  }
#undef ASH_RAYCAST_M
#undef ASH_RAYCAST
  const ash_status s = check_launch("tsdf_raycast");
  cudaFreeAsync(scratch, st);
  return s;
}

}  // extern "C"
