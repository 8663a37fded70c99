// grid.cu -- dense bit-array packing (the paper's baseline grid) and the
// GPU builder of the VDB-style sparse grid (Sec. 3: the dense occupancy grid
// becomes a VDB tree whose uniform blocks are pruned into tiles).
//
// Kernels
//   thresholds_kernel   exact per-axis voxel boundaries X[a] (one thread per
//                       boundary, binary search over binary32 keys)
//   pack_dense_kernel   uint8 voxels -> uint32 bit words, one ballot per word
//   vdb_blocks_kernel   one warp per four 8^3 blocks in a z row (8 lanes each):
//                       the 512-bit leaf masks and the blocks'
//                       empty/partial/full states
//   vdb_nodes_kernel    one 128-thread CTA per 16^3-block node: ballots over
//                       the block states give the child and tile masks, a
//                       CTA scan gives each mask word's leaf-count prefix
//   vdb_finalize_kernel one CTA: scan of leaf counts over all nodes, global
//                       leaf prefix per mask word, leaf and tile totals
//   vdb_finish_kernel   one warp per four blocks again: partial blocks' masks
//                       into the compact leaf pool with their refinement
//                       masks, and the region map of every block (an update
//                       that changes no block's state: of the changed blocks)
// The node and finish kernels also write the refinement masks (occupied
// 32^3 and 16^3 groups per node, occupied 4^3 and 2^3 cells per leaf) that
// let hierarchical DDA cross empty space in power-of-two steps below and
// above the 8^3 leaf, in the manner of an octree (Sec. 5 suggests finer
// subdivision).  The region map flattens the refined tree for the walk: a
// ray point's region (its size and occupancy) is one 2-byte load there
// instead of a descent through node, group, block, leaf and cell masks.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>

#include "grid.cuh"

namespace hdda {
namespace {

constexpr unsigned kFull = 0xffffffffu;

__global__ void thresholds_kernel(GridDev g, float* __restrict__ thr, float* __restrict__ mthr) {
  const int64_t R1 = g.R + 1;
  int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= (int64_t)g.L * 3 * R1) return;
  const int a = (int)(idx % R1);
  const int lc = (int)(idx / R1);
  const int c = lc % 3, l = lc / 3;
  const float lo = g.lv[l].lo[c], hi = g.lv[l].hi[c], s = g.lv[l].s[c];
  float X;
  if (a == 0) {
    X = lo;
  } else if (a == g.R) {
    X = hi;
  } else if (voxel_index(hi, lo, s, g.R) < a) {
    X = hi;  // no point of the box reaches index a
  } else {
    // voxel_index is monotone in x, so the set {x : index >= a} is an upper
    // range of binary32 values; find its first element.
    uint32_t kl = float_key(lo);  // index(lo) = 0 < a
    uint32_t kh = float_key(hi);  // index(hi) >= a
    while (kh - kl > 1u) {
      uint32_t km = kl + (kh - kl) / 2u;
      if (voxel_index(key_float(km), lo, s, g.R) >= a) kh = km; else kl = km;
    }
    X = key_float(kh);
  }
  thr[idx] = X;
  // the mirrored bounds (hdda_internal.cuh)
  float* m = mthr + (int64_t)lc * mthr_stride(g.R) + g.R;
  if (a < g.R) {
    const uint32_t u = __float_as_uint(X);
    const float below = (u & 0x7fffffffu) == 0u ? __uint_as_float(0x80000001u)
                                                 : __uint_as_float((u & 0x80000000u) ? u + 1u : u - 1u);
    m[-a - 1] = -below;
  }
  if (a > 0) m[a - 1] = X;
  if (a == g.R)
    for (int j = 0; j < kNodeVox; ++j) m[g.R + j] = X;
}

__global__ void pack_dense_kernel(const uint8_t* __restrict__ dense, int L, int R, int W,
                                  uint32_t* __restrict__ bits) {
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int64_t total = (int64_t)L * W;
  const int64_t w0 = warp * 32;
  if (w0 >= total) return;  // uniform per warp
  const int64_t R3 = (int64_t)R * R * R;
  uint32_t mine = 0;
  for (int j = 0; j < 32; ++j) {
    const int64_t gw = w0 + j;
    bool on = false;
    if (gw < total) {
      const int64_t l = gw / W, w = gw % W;
      const int64_t lin = w * 32 + lane;
      if (lin < R3) on = dense[l * R3 + lin] != 0;
    }
    const uint32_t b = __ballot_sync(kFull, on);
    if (lane == j) mine = b;
  }
  if (w0 + lane < total) bits[w0 + lane] = mine;
}

// Work on blocks is laid out four blocks per warp, eight lanes per block: lane
// 4 y + j is lane y of slot j, so that the rows of four blocks side by side in z
// make whole 32-byte sectors.
struct BlockAt {
  int l, bx, by, bz;
};

__device__ __forceinline__ BlockAt block_at(uint32_t blk, int B) {  // L * B^3 <= 8 * 128^3
  BlockAt a;
  a.bz = (int)(blk % (uint32_t)B);
  blk /= (uint32_t)B;
  a.by = (int)(blk % (uint32_t)B);
  blk /= (uint32_t)B;
  a.bx = (int)(blk % (uint32_t)B);
  a.l = (int)(blk / (uint32_t)B);
  return a;
}

// Bit b of the result: byte b of the two words is not zero.
__device__ __forceinline__ uint32_t nonzero8(uint2 v) {
  const uint32_t f = ((((v.x & 0x7f7f7f7fu) + 0x7f7f7f7fu) | v.x) >> 7) & 0x01010101u;
  const uint32_t h = ((((v.y & 0x7f7f7f7fu) + 0x7f7f7f7fu) | v.y) >> 7) & 0x01010101u;
  return __dp4a(h, 0x80402010u, __dp4a(f, 0x08040201u, 0u));
}

// The 512 occupancy bits of the lane's block, voxel ((x%8)*8 + y%8)*8 + z%8 at
// bit v%32 of word v/32: lane y of the slot returns words 2 y and 2 y + 1,
// the eight z rows of x = y, one byte per row.  The lane loads the rows of its
// own y (all eight in flight together; kVec: R a multiple of 8, eight bytes
// at once), and an 8 x 8 byte transpose over the slot's lanes turns (y, x) into
// (x, y).  Voxels past the grid's edge are empty.
template <bool kVec>
__device__ __forceinline__ uint2 block_words(const uint8_t* __restrict__ dense, int R,
                                             const BlockAt& a, bool active) {
  const int lane = threadIdx.x & 31, y = lane >> 2;
  uint32_t lo = 0, hi = 0;  // bytes x = 0..3 and 4..7 of this y
  const int vy = a.by * 8 + y, vz = a.bz * 8;
  const uint8_t* row = dense + (((int64_t)a.l * R + a.bx * 8) * R + vy) * R + vz;
  if constexpr (kVec) {
    uint2 v[8];
#pragma unroll
    for (int x = 0; x < 8; ++x)
      v[x] = active ? __ldg(reinterpret_cast<const uint2*>(row + (int64_t)x * R * R))
                    : make_uint2(0u, 0u);
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      lo |= nonzero8(v[x]) << (8 * x);
      hi |= nonzero8(v[x + 4]) << (8 * x);
    }
  } else {
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      uint32_t b = 0;
      if (active && vy < R && a.bx * 8 + x < R) {
#pragma unroll
        for (int z = 0; z < 8; ++z)
          if (vz + z < R) b |= (__ldg(row + (int64_t)x * R * R + z) != 0 ? 1u : 0u) << z;
      }
      if (x < 4) lo |= b << (8 * x);
      else hi |= b << (8 * (x - 4));
    }
  }
  // transpose: halves of x against y ^ 4, then pairs against y ^ 2, then bytes against y ^ 1
  const bool u4 = y & 4, u2 = y & 2, u1 = y & 1;
  const uint32_t r4 = __shfl_xor_sync(kFull, u4 ? lo : hi, 16);
  const uint32_t A = u4 ? r4 : lo, Bq = u4 ? hi : r4;  // rows y & 3 and (y & 3) + 4
  const uint32_t k2 = __byte_perm(A, Bq, u2 ? 0x7632 : 0x5410);
  const uint32_t r2 = __shfl_xor_sync(kFull, __byte_perm(A, Bq, u2 ? 0x5410 : 0x7632), 8);
  const uint32_t own = __byte_perm(k2, r2, u1 ? 0x7531 : 0x6420);  // rows y, y+4, y^2, (y^2)+4
  const uint32_t r1 = __shfl_xor_sync(kFull, __byte_perm(k2, r2, u1 ? 0x6420 : 0x7531), 4);
  const uint32_t order = (y & 3) == 0 ? 0x3120u : (y & 3) == 1 ? 0x1302u
                         : (y & 3) == 2 ? 0x2031u : 0x0213u;
  return make_uint2(__byte_perm(__byte_perm(own, r1, 0x6420), 0u, order),
                    __byte_perm(__byte_perm(own, r1, 0x7531), 0u, order));
}

// The slot's lanes, and its block's state from the lanes' words.
__device__ __forceinline__ unsigned slot_lanes() { return 0x11111111u << (threadIdx.x & 3); }

__device__ __forceinline__ uint8_t block_state(uint2 w) {
  const unsigned m = slot_lanes();
  const bool any = (__ballot_sync(kFull, (w.x | w.y) != 0u) & m) != 0u;
  const bool all = (__ballot_sync(kFull, (w.x & w.y) == kFull) & m) == m;
  return all ? kBlockFull : any ? kBlockPartial : kBlockEmpty;
}

// The block of the lane's slot in the i-th group of four along z of a grid
// of B^3 blocks per level; false past the row's end.
__device__ __forceinline__ bool quad_block(uint32_t i, int B, BlockAt& a) {
  const uint32_t Q = ((uint32_t)B + 3) / 4;
  a.bz = (int)(i % Q) * 4 + (threadIdx.x & 3);
  i /= Q;
  a.by = (int)(i % (uint32_t)B);
  i /= (uint32_t)B;
  a.bx = (int)(i % (uint32_t)B);
  a.l = (int)(i / (uint32_t)B);
  return a.bz < B;
}

__device__ __forceinline__ uint32_t block_index(const BlockAt& a, int B) {
  return (((uint32_t)a.l * B + a.bx) * B + a.by) * B + a.bz;
}

// Bound by the occupancy bytes' read and issue (2 x 512^3: 58 us, 72 % of cycles
// issuing; reading the bytes at 6.8 TB/s takes 40).  Single-byte loads, a ballot
// per 32 voxels and a warp per block were what it replaces.
template <bool kVec>
__global__ void __launch_bounds__(256) vdb_blocks_kernel(const uint8_t* __restrict__ dense,
                                                         uint32_t quads, int R, int B,
                                                         uint32_t* __restrict__ blk_masks,
                                                         uint8_t* __restrict__ blk_state) {
  const uint32_t q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (q >= quads) return;  // uniform per warp
  BlockAt a;
  const bool active = quad_block(q, B, a);
  const uint2 w = block_words<kVec>(dense, R, a, active);
  const uint8_t st = block_state(w);
  if (!active) return;
  const uint32_t blk = block_index(a, B);
  const int y = (threadIdx.x & 31) >> 2;
  *reinterpret_cast<uint2*>(blk_masks + (size_t)blk * kLeafWords + 2 * y) = w;
  if (y == 0) blk_state[blk] = st;
}

// Exclusive CTA-wide scan of one uint32 per thread (blockDim.x <= 1024, multiple of 32).
__device__ uint32_t cta_exclusive_scan(uint32_t v, uint32_t* warp_tot, uint32_t* total_out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t inc = v;
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(kFull, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    uint32_t t = lane < nw ? warp_tot[lane] : 0u;
    uint32_t ti = t;
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(kFull, ti, o);
      if (lane >= o) ti += y;
    }
    if (lane < nw) warp_tot[lane] = ti - t;  // exclusive warp offsets
    if (lane == 31) warp_tot[32] = ti;       // CTA total
  }
  __syncthreads();
  uint32_t r = warp_tot[warp] + inc - v;
  if (total_out) *total_out = warp_tot[32];
  __syncthreads();
  return r;
}

// `gate` (null: always) lets an incremental update skip the kernel when no
// block changed between empty, partial and full; the value is the same for
// every thread of the launch.
// A cell of a node beyond the grid's edge (never stored as a block state).
constexpr uint8_t kBlockOutside = 0xff;

__global__ void vdb_nodes_kernel(int L, int B, int N, const uint8_t* __restrict__ blk_state,
                                 uint32_t* __restrict__ child, uint32_t* __restrict__ tile,
                                 uint32_t* __restrict__ local_prefix,
                                 uint32_t* __restrict__ node_leaves,
                                 uint32_t* __restrict__ node_tiles,
                                 uint32_t* __restrict__ nstate,
                                 uint32_t* __restrict__ nsuper, const unsigned* __restrict__ gate) {
  if (gate && *gate == 0u) return;
  __shared__ uint32_t warp_tot[33];
  __shared__ uint32_t s_occ[kNodeWords];  // child | tile
  __shared__ uint32_t s_g16[16];          // occupied 16^3 groups
  const int64_t N3 = (int64_t)N * N * N;
  const int64_t B3 = (int64_t)B * B * B;
  const int64_t ng = blockIdx.x;
  const int l = (int)(ng / N3);
  const int node = (int)(ng % N3);
  const int nx = node / (N * N), ny = (node / N) % N, nz = node % N;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t my_child = 0, my_tile = 0, my_in = 0;
  // all 32 block states of this warp's words first (loads in flight together), then the votes
  uint8_t st[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const int cell = (warp * 32 + j) * 32 + lane;
    const int bx = nx * 16 + (cell >> 8), by = ny * 16 + ((cell >> 4) & 15),
              bz = nz * 16 + (cell & 15);
    st[j] = kBlockOutside;
    if (bx < B && by < B && bz < B)
      st[j] = __ldg(blk_state + (int64_t)l * B3 + ((int64_t)bx * B + by) * B + bz);
  }
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const uint32_t c = __ballot_sync(kFull, st[j] == kBlockPartial);
    const uint32_t t = __ballot_sync(kFull, st[j] == kBlockFull);
    const uint32_t i = __ballot_sync(kFull, st[j] != kBlockOutside);
    if (lane == j) { my_child = c; my_tile = t; my_in = i; }
  }
  const int w = threadIdx.x;  // mask word 0..127
  child[ng * kNodeWords + w] = my_child;
  tile[ng * kNodeWords + w] = my_tile;
  uint32_t leaves = 0, tiles = 0, incells = 0;
  local_prefix[ng * kNodeWords + w] = cta_exclusive_scan(__popc(my_child), warp_tot, &leaves);
  cta_exclusive_scan(__popc(my_tile), warp_tot, &tiles);
  cta_exclusive_scan(__popc(my_in), warp_tot, &incells);
  if (threadIdx.x == 0) {
    node_leaves[ng] = leaves;
    node_tiles[ng] = tiles;
    uint32_t st = kNodeMixed;
    if (leaves == 0 && tiles == 0) st = kNodeEmpty;
    else if (leaves == 0 && tiles == incells) st = kNodeFull;
    nstate[ng] = st;
  }
  // refinement: 16^3-voxel groups are 2^3 cells, 32^3-voxel groups 2^3 of those
  s_occ[w] = my_child | my_tile;
  __syncthreads();
  for (int j = 0; j < 4; ++j) {
    const int g2 = j * kNodeWords + threadIdx.x;  // 0..511
    const int gx = g2 >> 6, gy = (g2 >> 3) & 7, gz = g2 & 7;
    bool any = false;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const int cell = ((2 * gx + (a >> 2)) * 16 + (2 * gy + ((a >> 1) & 1))) * 16 + 2 * gz + (a & 1);
      any |= (s_occ[cell >> 5] >> (cell & 31)) & 1u;
    }
    const uint32_t bal = __ballot_sync(kFull, any);
    if (lane == 0) s_g16[g2 >> 5] = bal;
  }
  __syncthreads();
  if (threadIdx.x < 64) {
    const int g4 = threadIdx.x;
    const int gx = g4 >> 4, gy = (g4 >> 2) & 3, gz = g4 & 3;
    bool any = false;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const int g2 = ((2 * gx + (a >> 2)) * 8 + (2 * gy + ((a >> 1) & 1))) * 8 + 2 * gz + (a & 1);
      any |= (s_g16[g2 >> 5] >> (g2 & 31)) & 1u;
    }
    const uint32_t bal = __ballot_sync(kFull, any);
    if (lane == 0) nsuper[ng * kSuperWords + warp] = bal;
  }
  if (threadIdx.x < 16) nsuper[ng * kSuperWords + 2 + threadIdx.x] = s_g16[threadIdx.x];
}

constexpr int kMaxNodesTotal = HDDA_MAX_LEVELS * (HDDA_MAX_RES / kNodeVox) *
                               (HDDA_MAX_RES / kNodeVox) * (HDDA_MAX_RES / kNodeVox);

__global__ void vdb_finalize_kernel(int64_t nodes, const uint32_t* __restrict__ node_leaves,
                                    const uint32_t* __restrict__ node_tiles,
                                    const uint32_t* __restrict__ local_prefix,
                                    uint32_t* __restrict__ prefix, int64_t* __restrict__ totals,
                                    const unsigned* __restrict__ gate) {
  if (gate && *gate == 0u) return;
  __shared__ uint32_t base[kMaxNodesTotal];
  __shared__ uint32_t warp_tot[33];
  uint32_t carry = 0, tiles = 0;
  for (int64_t c0 = 0; c0 < nodes; c0 += blockDim.x) {
    const int64_t i = c0 + threadIdx.x;
    const uint32_t v = i < nodes ? node_leaves[i] : 0u;
    uint32_t chunk = 0;
    const uint32_t ex = cta_exclusive_scan(v, warp_tot, &chunk);
    if (i < nodes) base[i] = carry + ex;
    carry += chunk;
    uint32_t tchunk = 0;
    cta_exclusive_scan(i < nodes ? node_tiles[i] : 0u, warp_tot, &tchunk);
    tiles += tchunk;
  }
  __syncthreads();
  for (int64_t i = threadIdx.x; i < nodes * kNodeWords; i += blockDim.x)
    prefix[i] = base[i / kNodeWords] + local_prefix[i];
  if (threadIdx.x == 0) {
    totals[0] = carry;
    totals[1] = tiles;
  }
}

// Incremental update, step 1: four listed blocks per warp (every block when
// `list` is null).  A block's mask and state are recomputed from the dense
// bytes; a mask that differs is stored and changed[i] set, and flags[0] is
// set when the block's state (empty, partial, full) changes, since the node
// masks and the leaf compaction then change too.  An index outside the grid
// is skipped and raises kDevBadIndex.
template <bool kVec>
__global__ void __launch_bounds__(256) vdb_update_blocks_kernel(
    const uint8_t* __restrict__ dense, int L, int R, int B, const int64_t* __restrict__ list,
    int64_t count, uint32_t* __restrict__ blk_masks, uint8_t* __restrict__ blk_state,
    uint8_t* __restrict__ changed, unsigned* __restrict__ flags, unsigned* __restrict__ status) {
  const int64_t i0 = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * 4;
  if (i0 >= count) return;  // uniform per warp
  const int lane = threadIdx.x & 31, y = lane >> 2;
  const int64_t i = i0 + (lane & 3);
  const int64_t blk = i < count ? (list ? list[i] : i) : -1;
  const bool active = blk >= 0 && blk < (int64_t)L * B * B * B;
  const BlockAt a = block_at(active ? (uint32_t)blk : 0u, B);
  const uint2 w = block_words<kVec>(dense, R, a, active);
  const uint8_t st = block_state(w);
  uint2* mask = reinterpret_cast<uint2*>(blk_masks + (active ? blk : 0) * kLeafWords) + y;
  const uint2 old = active ? *mask : w;
  const bool diff =
      (__ballot_sync(kFull, active && (w.x != old.x || w.y != old.y)) & slot_lanes()) != 0u;
  if (active && diff) *mask = w;
  if (y == 0 && i < count) {
    changed[i] = diff ? 1 : 0;
    if (!active) {
      atomicOr(status, kDevBadIndex);
    } else if (st != blk_state[blk]) {
      blk_state[blk] = st;
      flags[0] = 1u;
    }
  }
}

// A pattern of bits 0, 2, 4, 6 as a nibble.
__device__ __forceinline__ uint32_t nibble(uint32_t v) {
  v = (v | (v >> 1)) & 0x33u;
  return (v | (v >> 2)) & 0xfu;
}

// ORs a value over the lanes of each slot.
__device__ __forceinline__ uint32_t slot_or(uint32_t v) {
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) v |= __shfl_xor_sync(kFull, v, o);
  return v;
}

// The last step of a build or update, four blocks per warp: a partial block's
// mask goes into its slot of the compact leaf pool with the leaf's refinement
// masks (occupied 2^3 and 4^3 cells, fully occupied 2^3 cells), and the
// block's 4^3 region-map cells are written (layout in hdda_internal.cuh).
// Lane y of a slot takes the cell rows y and y + 8, row = cx * 4 + cy: four
// cells along z, one 8-byte store (kVec: R a multiple of 8).  A block that is
// not partial has one region throughout, read from its node; a partial
// block's cells follow from the bytes of four voxel rows, its 4^3 cells from
// the rows' neighbours (lanes y ^ 1 and y ^ 4).  Voxels past the grid edge are
// empty in the masks.
//
// `flags` null: every block.  Otherwise an update: every block if flags[0]
// says that some block changed its state, and only the listed blocks with
// changed[i] set if not.  Grid-stride, so that an update can launch one
// resident wave.  Bound by the map's write (2 bytes per 2^3 voxels) and issue.
// For 2 x 512^3 voxels this takes 43 us; with a thread per cell that descended the
// tree and a scatter of 16 threads per block before it, the whole rebuild took
// 499 us where it takes 113 now (1 x 128^3: 27.5 -> 21, 4 x 128^3: 42.6 -> 23; an
// in-place update of 1 % of the blocks 264 -> 67, 40 -> 24 and 52 -> 25).
template <bool kVec>
__global__ void __launch_bounds__(256) vdb_finish_kernel(
    GridDev g, uint32_t quads, const uint8_t* __restrict__ blk_state,
    const uint32_t* __restrict__ blk_masks, uint32_t* __restrict__ leaves,
    uint32_t* __restrict__ lsub, uint16_t* __restrict__ rmap, const unsigned* __restrict__ flags,
    const int64_t* __restrict__ list, int64_t count, const uint8_t* __restrict__ changed) {
  const bool all = !flags || *flags != 0u;
  const int64_t items = all ? (int64_t)quads : (count + 3) / 4;
  const int lane = threadIdx.x & 31, y = lane >> 2;
  const int B = g.B, N = g.N, C = (g.R + 1) >> 1;
  const int64_t stride = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t it = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; it < items;
       it += stride) {  // uniform per warp
    BlockAt a;
    bool active;
    if (all) {
      active = quad_block((uint32_t)it, B, a);
    } else {
      const int64_t i = it * 4 + (lane & 3);
      active = i < count && changed[i];
      a = block_at(active ? (uint32_t)(list ? list[i] : i) : 0u, B);
    }
    const uint32_t blk = active ? block_index(a, B) : 0u;
    const uint8_t st = active ? blk_state[blk] : kBlockEmpty;
    const int ng = ((a.l * N + (a.bx >> 4)) * N + (a.by >> 4)) * N + (a.bz >> 4);
    const bool part = active && st == kBlockPartial;
    uint32_t one = 0;  // the entry of a block with one region
    if (active && !part) {
      const uint32_t ns = g.nstate[ng];
      if (ns != kNodeMixed) {
        one = (kMapNodeLog2 << 8) | (ns == kNodeFull ? 0xffu : 0u);
      } else if (st == kBlockFull) {
        one = (3u << 8) | 0xffu;
      } else {
        const uint32_t* sup = g.nsuper + ng * kSuperWords;
        const int g4 = (((a.bx >> 2) & 3) * 4 + ((a.by >> 2) & 3)) * 4 + ((a.bz >> 2) & 3);
        const int g2 = (((a.bx >> 1) & 7) * 8 + ((a.by >> 1) & 7)) * 8 + ((a.bz >> 1) & 7);
        one = !((sup[g4 >> 5] >> (g4 & 31)) & 1u)         ? 5u << 8
              : !((sup[2 + (g2 >> 5)] >> (g2 & 31)) & 1u) ? 4u << 8
                                                          : 3u << 8;
      }
    }
    uint2 cells[2];  // four 16-bit entries of the rows y and y + 8
    cells[0] = cells[1] = make_uint2(one | (one << 16), one | (one << 16));
    if (__any_sync(kFull, part)) {  // uniform
      const uint8_t* bytes = reinterpret_cast<const uint8_t*>(blk_masks + (size_t)blk * kLeafWords);
      uint32_t c2[2], f2[2], c4 = 0;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int cx = 2 * h + (y >> 2), cy = y & 3;
        uint32_t v0 = 0, v1 = 0;  // rows (2 cx, 2 cy), (2 cx, 2 cy + 1); the same of 2 cx + 1
        if (part) {
          v0 = *reinterpret_cast<const uint16_t*>(bytes + 16 * cx + 2 * cy);
          v1 = *reinterpret_cast<const uint16_t*>(bytes + 16 * cx + 8 + 2 * cy);
        }
        const uint32_t p0 = v0 & 0xffu, p1 = v0 >> 8, p2 = v1 & 0xffu, p3 = v1 >> 8;
        const uint32_t o = p0 | p1 | p2 | p3, n = p0 & p1 & p2 & p3;
        const uint32_t any = (o | (o >> 1)) & 0x55u, full = n & (n >> 1) & 0x55u;
        // over the 4^3 cells: some voxel (low half), some voxel missing (high half)
        uint32_t c = any | ((~full & 0x55u) << 16);
        c |= __shfl_xor_sync(kFull, c, 4);
        c |= __shfl_xor_sync(kFull, c, 16);
        uint32_t e[4];
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          const uint32_t m = ((p0 >> (2 * z)) & 3u) | (((p1 >> (2 * z)) & 3u) << 2) |
                             (((p2 >> (2 * z)) & 3u) << 4) | (((p3 >> (2 * z)) & 3u) << 6);
          const uint32_t big = c >> (4 * (z >> 1));
          e[z] = !(big & 0x5u)            ? 2u << 8
                 : !((big >> 16) & 0x5u)  ? (2u << 8) | 0xffu
                 : m == 0u || m == 0xffu  ? (1u << 8) | m
                                          : m;
        }
        if (part) cells[h] = make_uint2(e[0] | (e[1] << 16), e[2] | (e[3] << 16));
        // the leaf's masks: cell (cx * 4 + cy) * 4 + cz, 4^3 cell ((cx/2) * 2 + cy/2) * 2 + cz/2
        c2[h] = slot_or(nibble(any) << (4 * y));
        f2[h] = slot_or(nibble(full) << (4 * y));
        c4 |= (((c & 0x5u) ? 1u : 0u) | ((c & 0x50u) ? 2u : 0u)) << (4 * h + 2 * (cy >> 1));
      }
      c4 = slot_or(c4);
      if (part) {
        const int cell = ((a.bx & 15) * 16 + (a.by & 15)) * 16 + (a.bz & 15);
        const int w = ng * kNodeWords + (cell >> 5);
        const uint32_t leaf = g.prefix[w] + __popc(g.child[w] & ((1u << (cell & 31)) - 1u));
        reinterpret_cast<uint2*>(leaves + (size_t)leaf * kLeafWords)[y] =
            reinterpret_cast<const uint2*>(bytes)[y];
        uint32_t* sub = lsub + (size_t)leaf * kLeafSubWords;
        if (y < kLeafSubWords)
          sub[y] = y == 0 ? c2[0] : y == 1 ? c2[1] : y == 2 ? c4 : y == 3 ? f2[0] : f2[1];
      }
    }
    if (!active) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int cx = 4 * a.bx + 2 * h + (y >> 2), cy = 4 * a.by + (y & 3), cz = 4 * a.bz;
      uint16_t* out = rmap + (((int64_t)a.l * C + cx) * C + cy) * C + cz;
      if constexpr (kVec) {
        *reinterpret_cast<uint2*>(out) = cells[h];
      } else if (cx < C && cy < C) {  // past the grid edge when R is no multiple of 8
#pragma unroll
        for (int z = 0; z < 4; ++z)
          if (cz + z < C)
            out[z] = (uint16_t)((z < 2 ? cells[h].x : cells[h].y) >> (16 * (z & 1)));
      }
    }
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

int validate(const uint8_t* dense, int levels, int res, const hdda_aabb* aabbs) {
  if (!dense) return set_error(HDDA_ERR_INVALID_ARG, "dense is NULL");
  if (!aabbs) return set_error(HDDA_ERR_INVALID_ARG, "aabbs is NULL");
  if (levels < 1 || levels > HDDA_MAX_LEVELS)
    return set_error(HDDA_ERR_INVALID_ARG, "levels=%d outside 1..%d", levels, HDDA_MAX_LEVELS);
  if (res < 1 || res > HDDA_MAX_RES)
    return set_error(HDDA_ERR_INVALID_ARG, "res=%d outside 1..%d", res, HDDA_MAX_RES);
  for (int l = 0; l < levels; ++l) {
    for (int c = 0; c < 3; ++c) {
      const float lo = aabbs[l].lo[c], hi = aabbs[l].hi[c];
      if (!std::isfinite(lo) || !std::isfinite(hi) || !(lo < hi))
        return set_error(HDDA_ERR_INVALID_ARG, "level %d axis %d: box [%g, %g) invalid", l, c,
                         (double)lo, (double)hi);
      const float s = (float)res / (hi - lo);
      if (!std::isfinite(s))
        return set_error(HDDA_ERR_INVALID_ARG, "level %d axis %d: scale not finite", l, c);
    }
  }
  return HDDA_OK;
}

size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

template <typename T>
void carve(char* base, size_t& off, T*& ptr, int64_t count, bool take) {
  if (take) {
    ptr = reinterpret_cast<T*>(base ? base + off : nullptr);
    off = align_up(off + sizeof(T) * (size_t)count);
  } else {
    ptr = nullptr;
  }
}

size_t layout(hdda_grid* g, char* base) {
  const bool vdb = g->kind == HDDA_GRID_VDB;
  size_t off = 0;
  carve(base, off, g->thr, g->thr_count(), true);
  carve(base, off, g->mthr, (int64_t)g->L * 3 * mthr_stride(g->R), true);
  carve(base, off, g->bits, (int64_t)g->L * g->W, !vdb);
  const int64_t nw = g->nodes_total() * kNodeWords;
  carve(base, off, g->child, nw, vdb);
  carve(base, off, g->tile, nw, vdb);
  carve(base, off, g->prefix, nw, vdb);
  carve(base, off, g->nstate, g->nodes_total(), vdb);
  carve(base, off, g->leaves, g->blocks_total() * kLeafWords, vdb);
  carve(base, off, g->nsuper, g->nodes_total() * kSuperWords, vdb);
  carve(base, off, g->lsub, g->blocks_total() * kLeafSubWords, vdb);
  carve(base, off, g->rmap, g->map_cells(), vdb);
  carve(base, off, g->blk_masks, g->blocks_total() * kLeafWords, vdb);
  carve(base, off, g->blk_state, g->blocks_total(), vdb);
  carve(base, off, g->local_prefix, nw, vdb);
  carve(base, off, g->node_leaves, g->nodes_total(), vdb);
  carve(base, off, g->node_tiles, g->nodes_total(), vdb);
  carve(base, off, g->totals, 2, vdb);
  return off;
}

unsigned blocks_for(int64_t threads, int per) { return (unsigned)((threads + per - 1) / per); }

// CTAs of the update's grid-stride kernel: eight 256-thread CTAs per SM of a 152-SM GB300,
// about one resident wave
constexpr unsigned kGatedCtas = 152 * 8;

// Groups of four blocks along z, and whether their voxel rows can be loaded
// eight bytes at a time.
uint32_t quad_count(const hdda_grid* g) {
  return (uint32_t)((int64_t)g->L * g->B * g->B * ((g->B + 3) / 4));
}

bool vec_rows(const hdda_grid* g, const uint8_t* dense) {
  return g->R % 8 == 0 && reinterpret_cast<uintptr_t>(dense) % 8 == 0;
}

int launch_build(hdda_grid* g, const uint8_t* dense, cudaStream_t s) {
  if (g->kind == HDDA_GRID_DENSE) {
    const int64_t words = (int64_t)g->L * g->W;
    KernelTimer kt("pack_dense", s);
    pack_dense_kernel<<<blocks_for(words, 256), 256, 0, s>>>(dense, g->L, g->R, g->W, g->bits);
    kt.stop();
    HDDA_CUDA_TRY(cudaGetLastError());
  } else {
    KernelTimer kt("build_vdb", s);  // the four build kernels together
    const uint32_t quads = quad_count(g);
    const unsigned ctas = blocks_for((int64_t)quads * 32, 256);
    const bool vec = vec_rows(g, dense);
    (vec ? vdb_blocks_kernel<true> : vdb_blocks_kernel<false>)<<<ctas, 256, 0, s>>>(
        dense, quads, g->R, g->B, g->blk_masks, g->blk_state);
    HDDA_CUDA_TRY(cudaGetLastError());
    vdb_nodes_kernel<<<(unsigned)g->nodes_total(), kNodeWords, 0, s>>>(
        g->L, g->B, g->N, g->blk_state, g->child, g->tile, g->local_prefix, g->node_leaves,
        g->node_tiles, g->nstate, g->nsuper, nullptr);
    HDDA_CUDA_TRY(cudaGetLastError());
    vdb_finalize_kernel<<<1, 1024, 0, s>>>(g->nodes_total(), g->node_leaves, g->node_tiles,
                                          g->local_prefix, g->prefix, g->totals, nullptr);
    HDDA_CUDA_TRY(cudaGetLastError());
    (g->R % 8 == 0 ? vdb_finish_kernel<true> : vdb_finish_kernel<false>)<<<ctas, 256, 0, s>>>(
        g->view(), quads, g->blk_state, g->blk_masks, g->leaves, g->lsub, g->rmap, nullptr, nullptr,
        0, nullptr);
    kt.stop();
    HDDA_CUDA_TRY(cudaGetLastError());
  }
  HDDA_CUDA_TRY(cudaEventRecord(g->built, s));
  return HDDA_OK;
}

int create(int kind, const uint8_t* dense, int levels, int res, const hdda_aabb* aabbs,
           hdda_grid** out, cudaStream_t s) {
  clear_error();
  if (!out) return set_error(HDDA_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  int st = validate(dense, levels, res, aabbs);
  if (st != HDDA_OK) return st;
  hdda_grid* g = new (std::nothrow) hdda_grid();
  if (!g) return set_error(HDDA_ERR_OOM, "host allocation failed");
  g->kind = kind;
  g->L = levels;
  g->R = res;
  g->B = (res + kBlockDim - 1) / kBlockDim;
  g->N = (g->B + kNodeDim - 1) / kNodeDim;
  g->W = (int)(((int64_t)res * res * res + 31) / 32);
  cudaError_t e = cudaGetDevice(&g->device);
  if (e != cudaSuccess) { delete g; return cuda_error(e, "cudaGetDevice"); }
  for (int l = 0; l < levels; ++l) {
    g->boxes[l] = aabbs[l];
    for (int c = 0; c < 3; ++c) g->scale[l][c] = (float)res / (aabbs[l].hi[c] - aabbs[l].lo[c]);
  }
  g->base_bytes = layout(g, nullptr);
  e = cudaMalloc(&g->base, g->base_bytes);
  if (e != cudaSuccess) { delete g; return cuda_error(e, "cudaMalloc(grid)"); }
  layout(g, static_cast<char*>(g->base));
  scratch_users(g->device, 1);
  e = cudaEventCreateWithFlags(&g->built, cudaEventDisableTiming);
  if (e != cudaSuccess) { hdda_grid_free(g); return cuda_error(e, "cudaEventCreate"); }
  thresholds_kernel<<<blocks_for(g->thr_count(), 128), 128, 0, s>>>(g->view(), g->thr, g->mthr);
  e = cudaGetLastError();
  if (e != cudaSuccess) { hdda_grid_free(g); return cuda_error(e, "thresholds_kernel"); }
  st = launch_build(g, dense, s);
  if (st != HDDA_OK) { hdda_grid_free(g); return st; }
  *out = g;
  return HDDA_OK;
}

int64_t structure_bytes(const hdda_grid* g, int64_t n_leaves) {
  int64_t b = (int64_t)g->L * (int64_t)sizeof(LevelDev) + g->thr_count() * 4;
  if (g->kind == HDDA_GRID_DENSE) {
    b += (int64_t)g->L * g->W * 4;
  } else {
    b += g->nodes_total() * (3 * kNodeWords * 4 + 4);
    b += n_leaves * kLeafWords * 4;
    if (g->refine) b += g->nodes_total() * kSuperWords * 4 + n_leaves * kLeafSubWords * 4;
  }
  return b;
}

}  // namespace
}  // namespace hdda

using namespace hdda;

extern "C" int hdda_pack_dense(const uint8_t* dense, int levels, int res, const hdda_aabb* aabbs,
                               hdda_grid** out, hdda_stream_t stream) {
  return create(HDDA_GRID_DENSE, dense, levels, res, aabbs, out, (cudaStream_t)stream);
}

extern "C" int hdda_build_vdb(const uint8_t* dense, int levels, int res, const hdda_aabb* aabbs,
                              hdda_grid** out, size_t* bytes_out, hdda_stream_t stream) {
  int st = create(HDDA_GRID_VDB, dense, levels, res, aabbs, out, (cudaStream_t)stream);
  if (st != HDDA_OK || !bytes_out) return st;
  hdda_grid_stats gs;
  st = hdda_grid_stats_get(*out, &gs);
  if (st != HDDA_OK) return st;
  *bytes_out = (size_t)gs.bytes;
  return HDDA_OK;
}

extern "C" int hdda_grid_rebuild(hdda_grid* grid, const uint8_t* dense, hdda_stream_t stream) {
  clear_error();
  if (!grid) return set_error(HDDA_ERR_INVALID_ARG, "grid is NULL");
  if (!dense) return set_error(HDDA_ERR_INVALID_ARG, "dense is NULL");
  return launch_build(grid, dense, (cudaStream_t)stream);
}

namespace hdda {
namespace {

// Pinned host word for the synchronous status read of an update.
struct UpdateWord {
  unsigned* p = nullptr;
  ~UpdateWord() { if (p) cudaFreeHost(p); }
};
thread_local UpdateWord t_update_word;

int update_vdb(hdda_grid* g, const uint8_t* dense, const int64_t* blocks, int64_t n_blocks,
               uint32_t* dev_status, cudaStream_t s) {
  const int64_t count = blocks ? n_blocks : g->blocks_total();
  if (count == 0) return HDDA_OK;
  unsigned* hw = nullptr;
  if (!dev_status) {
    if (!t_update_word.p) HDDA_CUDA_TRY(cudaMallocHost(&t_update_word.p, sizeof(unsigned)));
    hw = t_update_word.p;
  }
  // scratch: {flags[0] = structure changed, status}, then changed[count]
  char* scratch = nullptr;
  HDDA_CUDA_TRY(scratch_alloc(&scratch, 16 + (size_t)count, s));
  unsigned* flags = reinterpret_cast<unsigned*>(scratch);
  unsigned* status = dev_status ? dev_status : flags + 1;
  uint8_t* changed = reinterpret_cast<uint8_t*>(scratch + 16);
  int st = HDDA_OK;
  cudaError_t e = cudaMemsetAsync(scratch, 0, 16, s);
  if (e != cudaSuccess) st = cuda_error(e, "cudaMemsetAsync");
  if (st == HDDA_OK) {
    KernelTimer kt("update_vdb", s);  // the update's four kernels together
    const unsigned ctas = blocks_for((count + 3) / 4 * 32, 256);
    (vec_rows(g, dense) ? vdb_update_blocks_kernel<true>
                        : vdb_update_blocks_kernel<false>)<<<ctas, 256, 0, s>>>(
        dense, g->L, g->R, g->B, blocks, count, g->blk_masks, g->blk_state, changed, flags,
        status);
    vdb_nodes_kernel<<<(unsigned)g->nodes_total(), kNodeWords, 0, s>>>(
        g->L, g->B, g->N, g->blk_state, g->child, g->tile, g->local_prefix, g->node_leaves,
        g->node_tiles, g->nstate, g->nsuper, flags);
    vdb_finalize_kernel<<<1, 1024, 0, s>>>(g->nodes_total(), g->node_leaves, g->node_tiles,
                                          g->local_prefix, g->prefix, g->totals, flags);
    // grid-stride over at most one resident wave: it costs little when no block changed state
    const uint32_t quads = quad_count(g);
    (g->R % 8 == 0 ? vdb_finish_kernel<true> : vdb_finish_kernel<false>)<<<
        std::min(blocks_for((int64_t)quads * 32, 256), kGatedCtas), 256, 0, s>>>(
        g->view(), quads, g->blk_state, g->blk_masks, g->leaves, g->lsub, g->rmap, flags, blocks,
        count, changed);
    kt.stop();
    e = cudaGetLastError();
    if (e != cudaSuccess) st = cuda_error(e, "update kernels");
  }
  if (st == HDDA_OK && !dev_status) {
    e = cudaMemcpyAsync(hw, flags + 1, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) st = cuda_error(e, "cudaMemcpyAsync(status)");
  }
  st = scratch_free(scratch, s, st);
  if (st != HDDA_OK) return st;
  HDDA_CUDA_TRY(cudaEventRecord(g->built, s));
  if (dev_status) return HDDA_OK;
  HDDA_CUDA_TRY(cudaStreamSynchronize(s));
  if (*hw & kDevBadIndex)
    return set_error(HDDA_ERR_INVALID_ARG, "a block index lies outside the grid (skipped)");
  return HDDA_OK;
}

}  // namespace
}  // namespace hdda

extern "C" int hdda_grid_update(hdda_grid* grid, const uint8_t* dense, const int64_t* blocks,
                                int64_t n_blocks, uint32_t* dev_status, hdda_stream_t stream) {
  clear_error();
  if (!grid) return set_error(HDDA_ERR_INVALID_ARG, "grid is NULL");
  if (!dense) return set_error(HDDA_ERR_INVALID_ARG, "dense is NULL");
  if (blocks && (n_blocks < 0 || n_blocks > ((int64_t)1 << 26)))
    return set_error(HDDA_ERR_INVALID_ARG, "n_blocks=%lld outside 0..2^26", (long long)n_blocks);
  if (reinterpret_cast<uintptr_t>(dev_status) % 4 != 0)
    return set_error(HDDA_ERR_INVALID_ARG, "dev_status must be 4-byte aligned");
  int dev = 0;
  HDDA_CUDA_TRY(cudaGetDevice(&dev));
  if (dev != grid->device)
    return set_error(HDDA_ERR_INVALID_ARG, "grid lives on device %d, current is %d",
                     grid->device, dev);
  cudaStream_t s = (cudaStream_t)stream;
  if (grid->kind == HDDA_GRID_DENSE) return launch_build(grid, dense, s);  // one repack
  return update_vdb(grid, dense, blocks, n_blocks, dev_status, s);
}

extern "C" int hdda_grid_stats_get(const hdda_grid* g, hdda_grid_stats* out) {
  clear_error();
  if (!g || !out) return set_error(HDDA_ERR_INVALID_ARG, "grid or out is NULL");
  std::memset(out, 0, sizeof(*out));
  out->kind = g->kind;
  out->levels = g->L;
  out->res = g->R;
  out->blocks = g->B;
  out->nodes = g->N;
  out->dense_bytes = (int64_t)g->L * g->W * 4;
  int64_t totals[2] = {0, 0};
  if (g->kind == HDDA_GRID_VDB) {
    HDDA_CUDA_TRY(cudaEventSynchronize(g->built));
    HDDA_CUDA_TRY(cudaMemcpy(totals, g->totals, sizeof(totals), cudaMemcpyDeviceToHost));
  }
  out->n_leaves = totals[0];
  out->n_tiles = totals[1];
  out->bytes = structure_bytes(g, totals[0]);
  if (g->kind == HDDA_GRID_VDB) out->map_bytes = g->map_cells() * (int64_t)sizeof(uint16_t);
  return HDDA_OK;
}

extern "C" int hdda_grid_copy_array(const hdda_grid* g, int which, void* dst, size_t bytes,
                                    size_t* needed) {
  clear_error();
  if (!g) return set_error(HDDA_ERR_INVALID_ARG, "grid is NULL");
  const bool vdb = g->kind == HDDA_GRID_VDB;
  const void* src = nullptr;
  size_t n = 0;
  const size_t nw = (size_t)g->nodes_total() * kNodeWords * 4;
  switch (which) {
    case HDDA_ARRAY_THRESHOLDS: src = g->thr; n = (size_t)g->thr_count() * 4; break;
    case HDDA_ARRAY_DENSE_BITS: if (!vdb) { src = g->bits; n = (size_t)g->L * g->W * 4; } break;
    case HDDA_ARRAY_CHILD_MASK: if (vdb) { src = g->child; n = nw; } break;
    case HDDA_ARRAY_TILE_MASK: if (vdb) { src = g->tile; n = nw; } break;
    case HDDA_ARRAY_LEAF_PREFIX: if (vdb) { src = g->prefix; n = nw; } break;
    case HDDA_ARRAY_LEAVES:
    case HDDA_ARRAY_LEAF_SUB:
      if (vdb) {
        hdda_grid_stats gs;
        int st = hdda_grid_stats_get(g, &gs);
        if (st != HDDA_OK) return st;
        const bool sub = which == HDDA_ARRAY_LEAF_SUB;
        src = sub ? g->lsub : g->leaves;
        n = (size_t)gs.n_leaves * (sub ? kLeafSubWords : kLeafWords) * 4;
      }
      break;
    case HDDA_ARRAY_NODE_SUPER:
      if (vdb) { src = g->nsuper; n = (size_t)g->nodes_total() * kSuperWords * 4; }
      break;
    case HDDA_ARRAY_REGION_MAP:
      if (vdb) { src = g->rmap; n = (size_t)g->map_cells() * sizeof(uint16_t); }
      break;
    default: break;
  }
  if (!src) return set_error(HDDA_ERR_INVALID_ARG, "array %d not held by this grid", which);
  if (needed) *needed = n;
  if (!dst) return HDDA_OK;
  if (bytes < n) return set_error(HDDA_ERR_CAPACITY, "array needs %zu bytes, got %zu", n, bytes);
  HDDA_CUDA_TRY(cudaEventSynchronize(g->built));
  if (n) HDDA_CUDA_TRY(cudaMemcpy(dst, src, n, cudaMemcpyDeviceToHost));
  return HDDA_OK;
}

extern "C" int hdda_grid_set_refine(hdda_grid* g, int on) {
  clear_error();
  if (!g) return set_error(HDDA_ERR_INVALID_ARG, "grid is NULL");
  if (g->kind != HDDA_GRID_VDB)
    return set_error(HDDA_ERR_INVALID_ARG, "refinement applies to VDB grids");
  g->refine = on ? 1 : 0;
  return HDDA_OK;
}

extern "C" int hdda_grid_set_walk(hdda_grid* g, int variant) {
  clear_error();
  if (!g) return set_error(HDDA_ERR_INVALID_ARG, "grid is NULL");
  if (variant != HDDA_WALK_BRANCH && variant != HDDA_WALK_SKIP)
    return set_error(HDDA_ERR_INVALID_ARG, "walk variant %d unknown", variant);
  g->walk_variant = variant;
  return HDDA_OK;
}

extern "C" void hdda_grid_free(hdda_grid* g) {
  if (!g) return;
  if (g->built) {
    cudaEventSynchronize(g->built);
    cudaEventDestroy(g->built);
  }
  if (g->base) {
    cudaDeviceSynchronize();
    cudaFree(g->base);
    scratch_users(g->device, -1);
  }
  delete g;
}
