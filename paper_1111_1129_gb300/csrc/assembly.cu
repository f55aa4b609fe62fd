// Assembly of the sparse representation on the GPU (Sec. 2-3):
//   numbering scheme I(x,y,z) -> contiguous index I_c (rank of the fluid
//   cells in key order, solids dropped) -> pull adjacency with implicit
//   bounce back.
//
// The paper removes the gaps of the index with distributed run descriptors
// merged up an octree of MPI ranks (Sec. 3, "In- and outcells",
// "Contiguous index generation").  On one GPU the same result is a stream
// compaction in key order.  Instead of sorting keys, the kernels walk the
// key space itself: key k is inverted to its cell (every scheme here is a
// bijection onto a superset of the box), so a tile of consecutive keys is a
// contiguous run of the final order, and ranks come from a tile count, a
// scan of the counts and a scan within the tile.  No key array is stored.
//
// The passes over the tiles come in three kinds: lexicographic order with
// aligned flags reads 16 consecutive flags per thread; the curves (Morton,
// Hilbert) take the 16^3 cube that a tile is, reading and writing it by rows
// through shared memory, and only the cubes that meet the box (a Hilbert curve
// of 1024x256x256 visits 16 times the box); blocked order inverts each key.
// The first two are bound by bytes, the blocked pass by the arithmetic of the
// inverse.  1024x256x256 bed, count + scan + scatter against one kernel that
// walked all keys one by one: Hilbert 47.2 -> 0.64 ms, 8^3 blocked 1.03 ->
// 0.34 ms; lexicographic, cells written in order from shared memory, 0.22 ->
// 0.12 ms.
#include <cstdio>

#include "lbm_internal.cuh"

namespace lbm {

namespace {

constexpr int kTileThreads = 256;
constexpr int kTileRounds = 16;
constexpr uint64_t kTileKeys = (uint64_t)kTileThreads * kTileRounds;

__global__ void keys_kernel(KeySpace ks, uint64_t* keys, int64_t box) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= box) return;
  const int64_t x = c % ks.nx, y = (c / ks.nx) % ks.ny, z = c / (ks.nx * ks.ny);
  keys[c] = key_of(ks, x, y, z);
}

// Block sum of `mine`, on thread 0.
__device__ __forceinline__ uint32_t block_sum(uint32_t mine) {
  __shared__ uint32_t warp_sum[kTileThreads / 32];
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, o);
  if ((threadIdx.x & 31) == 0) warp_sum[threadIdx.x >> 5] = mine;
  __syncthreads();
  uint32_t s = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < kTileThreads / 32; ++w) s += warp_sum[w];
  return s;
}
// Sum of `mine` over the threads before this one; *total: over all.
__device__ __forceinline__ uint32_t block_prefix(uint32_t mine, uint32_t* total) {
  __shared__ uint32_t warp_tot[kTileThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  uint32_t before = incl - mine, all = 0;
#pragma unroll
  for (int w = 0; w < kTileThreads / 32; ++w) {
    before += w < warp ? warp_tot[w] : 0;
    all += warp_tot[w];
  }
  *total = all;
  return before;
}

// ---- any order, key by key ----------------------------------------------------
// Thread t takes keys t, t + 256, ... of its tile; all their flags are requested
// before any is used.
template <bool SMALL_BLOCKED>
__device__ __forceinline__ void tile_keys(const KeySpace& ks, const uint8_t* __restrict__ flags,
                                          uint64_t base, int32_t c[kTileRounds],
                                          uint8_t f[kTileRounds]) {
#pragma unroll
  for (int r = 0; r < kTileRounds; ++r) {
    const uint64_t k = base + (uint64_t)(r * kTileThreads) + threadIdx.x;
    if (SMALL_BLOCKED) {
      int32_t x, y, z;
      c[r] = blocked_cell(ks, (uint32_t)k, x, y, z)
                 ? x + (int32_t)ks.nx * (y + (int32_t)ks.ny * z)
                 : -1;
    } else {
      int64_t x, y, z;
      c[r] = cell_of(ks, k, x, y, z) ? (int32_t)(x + ks.nx * (y + ks.ny * z)) : -1;
    }
    f[r] = c[r] >= 0 ? flags[c[r]] : 1;
  }
}
// Whether blocked_cell serves a key space (its tiles' last keys included).
bool small_blocked(const KeySpace& ks) {
  return ks.kind == LBM_ORDER_BLOCKED && ks.size + kTileKeys < (1ull << 31);
}

// Pass 1: number of fluid cells in each tile of kTileKeys consecutive keys;
// flags other than 0/1 raise *bad.
template <bool SMALL_BLOCKED>
__global__ void __launch_bounds__(kTileThreads)
    tile_count_kernel(KeySpace ks, const uint8_t* __restrict__ flags, uint32_t* counts,
                      int* bad) {
  int32_t c[kTileRounds];
  uint8_t f[kTileRounds];
  tile_keys<SMALL_BLOCKED>(ks, flags, (uint64_t)blockIdx.x * kTileKeys, c, f);
  uint32_t mine = 0;
  bool any_bad = false;
#pragma unroll
  for (int r = 0; r < kTileRounds; ++r) {
    any_bad |= f[r] > 1;
    mine += f[r] == 0;
  }
  if (any_bad) atomicOr(bad, 1);
  mine = block_sum(mine);
  if (threadIdx.x == 0) counts[blockIdx.x] = mine;
}

// Pass 2: exclusive scan of the tile counts in spans of kScanSpan, each span by
// itself (offsets; span totals to `span`), then of the span totals by one
// block (total -> *total).  The first of tile t is offsets[t] + span[t / kScanSpan].
constexpr int kScanSpan = 4096;
__global__ void __launch_bounds__(1024)
    tile_scan_kernel(const uint32_t* __restrict__ counts, int64_t ntiles,
                     uint32_t* __restrict__ offsets, int64_t* __restrict__ span) {
  __shared__ uint32_t s[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t t = (int64_t)blockIdx.x * kScanSpan + 4 * (int64_t)threadIdx.x;
  uint32_t v[4], mine = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    v[j] = t + j < ntiles ? counts[t + j] : 0;
    mine += v[j];
  }
  uint32_t incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) s[warp] = incl;
  __syncthreads();
  uint32_t before = incl - mine, all = 0;
  for (int w = 0; w < 32; ++w) {
    before += w < warp ? s[w] : 0;
    all += s[w];
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (t + j < ntiles) offsets[t + j] = before;
    before += v[j];
  }
  if (threadIdx.x == 0) span[blockIdx.x] = all;
}
__global__ void __launch_bounds__(1024)
    span_scan_kernel(int64_t* span, int64_t nspans, int64_t* total) {
  __shared__ int64_t s[1024];
  const int t = threadIdx.x;
  const int64_t chunk = (nspans + 1023) / 1024;
  const int64_t b = (int64_t)t * chunk;
  const int64_t e = b + chunk < nspans ? b + chunk : nspans;
  int64_t mine = 0;
  for (int64_t i = b; i < e; ++i) mine += span[i];
  s[t] = mine;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    const int64_t v = t >= off ? s[t - off] : 0;
    __syncthreads();
    s[t] += v;
    __syncthreads();
  }
  int64_t run = s[t] - mine;
  for (int64_t i = b; i < e; ++i) {
    const int64_t c = span[i];
    span[i] = run;
    run += c;
  }
  if (t == 1023) *total = s[1023];
}
// The scanned counts.
struct TileRanks {
  const uint32_t* offsets;
  const int64_t* span;
  __device__ __forceinline__ int64_t first(int64_t tile) const {
    return (int64_t)offsets[tile] + span[tile / kScanSpan];
  }
};

// Pass 3: walk each tile again in key order and scatter: cells[rank] = box
// index, inv[box index] = rank (or -1 for a solid cell).
template <bool SMALL_BLOCKED>
__global__ void __launch_bounds__(kTileThreads)
    tile_scatter_kernel(KeySpace ks, const uint8_t* __restrict__ flags, TileRanks ranks,
                        int32_t* cells, int32_t* inv) {
  constexpr int kWarps = kTileThreads / 32;
  __shared__ uint32_t count[kTileRounds * kWarps];   // fluid keys of each warp's round, in key order
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t c[kTileRounds];
  uint8_t f[kTileRounds];
  tile_keys<SMALL_BLOCKED>(ks, flags, (uint64_t)blockIdx.x * kTileKeys, c, f);
  uint32_t ballot[kTileRounds];
#pragma unroll
  for (int r = 0; r < kTileRounds; ++r) {
    ballot[r] = __ballot_sync(0xffffffffu, f[r] == 0);
    if (lane == 0) count[r * kWarps + warp] = __popc(ballot[r]);
  }
  __syncthreads();
  if (warp == 0) {   // exclusive scan of the kTileRounds x kWarps = 128 counts
    uint32_t v[4], mine = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) mine += v[j] = count[4 * lane + j];
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    uint32_t before = incl - mine;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      count[4 * lane + j] = before;
      before += v[j];
    }
  }
  __syncthreads();
  const int64_t first = ranks.first(blockIdx.x);
#pragma unroll
  for (int r = 0; r < kTileRounds; ++r) {
    if (c[r] < 0) continue;
    if (f[r] == 0) {
      const int64_t rank = first + count[r * kWarps + warp] + __popc(ballot[r] & ((1u << lane) - 1u));
      cells[rank] = c[r];
      inv[c[r]] = (int32_t)rank;
    } else {
      inv[c[r]] = -1;
    }
  }
}
static_assert(kTileRounds * (kTileThreads / 32) == 128, "four counts per lane");

// ---- curves: a tile is a cube ---------------------------------------------------
// The tiles whose cubes meet the box, in no particular order: as many as there
// are aligned cubes in the box, `room`.
__global__ void active_tiles_kernel(KeySpace ks, int64_t ntiles, int64_t room, uint32_t* active,
                                    uint32_t* n_active) {
  const int64_t tile = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool meets = false;
  if (tile < ntiles) {
    int32_t p[3];
    curve_point(ks, (uint64_t)tile, 0, p);
    const int32_t low = ~((1 << ks.levels) - 1);
    meets = (p[0] & low) < ks.nx && (p[1] & low) < ks.ny && (p[2] & low) < ks.nz;
  }
  if (!meets) return;
  const uint32_t at = atomicAdd(n_active, 1u);
  if (at < room) active[at] = (uint32_t)tile;
}

constexpr int kCubeCells = 4096;   // of a cube of 16 cells per axis (smaller cubes use a part)
static_assert(kCubeCells == (int)kTileKeys, "a tile of a curve of 4 levels is one cube");

// The cube's flags by rows of 16 cells, row y + 16 z of the cube by thread
// y + 16 z (1 outside the box): w[j] holds cells 4 j .. 4 j + 3.
__device__ __forceinline__ void cube_row(const KeySpace& ks, const uint8_t* __restrict__ flags,
                                         const int32_t low[3], uint32_t w[4]) {
  const int32_t y = low[1] + (int32_t)(threadIdx.x & 15), z = low[2] + (int32_t)(threadIdx.x >> 4);
#pragma unroll
  for (int j = 0; j < 4; ++j) w[j] = 0x01010101u;
  if (y >= ks.ny || z >= ks.nz) return;
  const uint8_t* row = flags + low[0] + ks.nx * (y + ks.ny * z);
  if (low[0] + 16 <= ks.nx && reinterpret_cast<uintptr_t>(row) % 16 == 0) {
    const uint4 v = *reinterpret_cast<const uint4*>(row);
    w[0] = v.x;
    w[1] = v.y;
    w[2] = v.z;
    w[3] = v.w;
  } else {
#pragma unroll
    for (int b = 0; b < 16; ++b)
      if (low[0] + b < ks.nx)
        w[b >> 2] = (w[b >> 2] & ~(0xffu << (8 * (b & 3)))) | ((uint32_t)row[b] << (8 * (b & 3)));
  }
}

// Pass 1 of a curve: fluid cells of each active cube, which needs no order.
__global__ void __launch_bounds__(kTileThreads)
    cube_count_kernel(KeySpace ks, const uint8_t* __restrict__ flags,
                      const uint32_t* __restrict__ active, const uint32_t* __restrict__ n_active,
                      uint32_t* counts, int* bad) {
  if (blockIdx.x >= *n_active) return;
  const uint32_t tile = active[blockIdx.x];
  int32_t low[3];
  curve_point(ks, tile, 0, low);
#pragma unroll
  for (int a = 0; a < 3; ++a) low[a] &= ~15;
  uint32_t w[4], mine = 0;
  cube_row(ks, flags, low, w);
  bool any_bad = false;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    any_bad |= (w[j] & 0xfefefefeu) != 0;   // a byte other than 0 or 1
    mine += 4u - (uint32_t)__popc(w[j]);     // bytes 0/1: popc counts the solid ones
  }
  if (any_bad) atomicOr(bad, 1);
  mine = block_sum(mine);
  if (threadIdx.x == 0) counts[tile] = mine;
}

// Pass 3 of a curve: thread t takes local keys 16 t .. 16 t + 15.
__global__ void __launch_bounds__(kTileThreads)
    cube_scatter_kernel(KeySpace ks, const uint8_t* __restrict__ flags,
                        const uint32_t* __restrict__ active, const uint32_t* __restrict__ n_active,
                        TileRanks ranks, int32_t* cells, int32_t* inv) {
  if (blockIdx.x >= *n_active) return;
  __shared__ __align__(16) uint8_t flag[kCubeCells];   // by place in the cube
  __shared__ int32_t rank_of[kCubeCells];              // by place in the cube
  __shared__ int32_t cell_at[kCubeCells];              // in key order, fluid cells only
  __shared__ CurveFrame frame;
  const uint32_t tile = active[blockIdx.x];
  if (threadIdx.x < 4) {
    int32_t p[3];
    curve_point(ks, tile, (int)threadIdx.x, p);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int32_t at = __shfl_sync(0xfu, p[a], 0);
      if (threadIdx.x == 0) frame.at[a] = at;
      else frame.d[threadIdx.x - 1][a] = p[a] - at;
    }
  }
  __syncthreads();
  int32_t low[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) low[a] = frame.at[a] & ~15;
  uint32_t w[4];
  cube_row(ks, flags, low, w);
  *reinterpret_cast<uint4*>(flag + 16 * threadIdx.x) = make_uint4(w[0], w[1], w[2], w[3]);
  __syncthreads();
  uint32_t place[8], fluid = 0;   // places (12 bits) of two keys per word; bit b: key b is fluid
#pragma unroll
  for (int b = 0; b < 16; ++b) {
    const uint32_t l = 16u * threadIdx.x + b;
    uint32_t at = 0;
    if (l < (1u << (3 * ks.levels))) {
      uint32_t c[3];
      int32_t p[3];
      curve_local(ks, l, c);
      curve_cell(frame, c, p);
      at = (uint32_t)((p[0] - low[0]) + 16 * ((p[1] - low[1]) + 16 * (p[2] - low[2])));
      fluid |= (uint32_t)(flag[at] == 0) << b;
    }
    place[b >> 1] = b & 1 ? place[b >> 1] | at << 16 : at;
  }
#pragma unroll
  for (int j = 0; j < 16; ++j) rank_of[kTileThreads * j + threadIdx.x] = -1;
  uint32_t total;
  uint32_t at = block_prefix((uint32_t)__popc(fluid), &total);   // its barrier orders rank_of
  const int64_t first = ranks.first(tile);
#pragma unroll
  for (int b = 0; b < 16; ++b) {
    if (!((fluid >> b) & 1u)) continue;
    const uint32_t pl = (place[b >> 1] >> (16 * (b & 1))) & 0xffffu;
    rank_of[pl] = (int32_t)first + (int32_t)at;
    cell_at[at++] = (int32_t)((low[0] + (int32_t)(pl & 15)) +
                              ks.nx * ((low[1] + (int32_t)((pl >> 4) & 15)) +
                                       ks.ny * (low[2] + (int32_t)(pl >> 8))));
  }
  __syncthreads();
  for (uint32_t j = threadIdx.x; j < total; j += kTileThreads) cells[first + j] = cell_at[j];
#pragma unroll
  for (int j = 0; j < 16; ++j) {   // 16 threads per row of the cube
    const int32_t pl = kTileThreads * j + (int32_t)threadIdx.x;
    const int32_t x = low[0] + (pl & 15), y = low[1] + ((pl >> 4) & 15), z = low[2] + (pl >> 8);
    if (x < ks.nx && y < ks.ny && z < ks.nz) inv[x + ks.nx * (y + ks.ny * z)] = rank_of[pl];
  }
}

// ---- lexicographic order: the key is the box index --------------------------
// A tile is then kTileKeys consecutive flag bytes, and thread t takes the
// 16 at tile + 16 t with one 16-byte load (flags 16-byte aligned; the last,
// partial chunk of the box byte by byte).  The generic passes above walk
// their 16 keys one by one and were bound by those dependent rounds.
static_assert(kTileKeys == 16 * kTileThreads, "16 keys per thread");

// The 16 flags of thread t's chunk (1 past the box) and how many are inside.
__device__ __forceinline__ int lex_chunk(const uint8_t* __restrict__ flags, int64_t box,
                                         int64_t k0, uint32_t w[4]) {
  if (k0 + 16 <= box) {
    const uint4 v = *reinterpret_cast<const uint4*>(flags + k0);
    w[0] = v.x;
    w[1] = v.y;
    w[2] = v.z;
    w[3] = v.w;
    return 16;
  }
  const int valid = k0 < box ? (int)(box - k0) : 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) w[j] = 0x01010101u;
  for (int b = 0; b < valid; ++b)
    w[b >> 2] = (w[b >> 2] & ~(0xffu << (8 * (b & 3)))) | ((uint32_t)flags[k0 + b] << (8 * (b & 3)));
  return valid;
}

// Pass 1 in lexicographic order (as tile_count_kernel).
__global__ void __launch_bounds__(kTileThreads)
    tile_count_lex_kernel(const uint8_t* __restrict__ flags, int64_t box, uint32_t* counts,
                          int* bad) {
  uint32_t w[4];
  lex_chunk(flags, box, (int64_t)blockIdx.x * kTileKeys + 16 * (int64_t)threadIdx.x, w);
  uint32_t mine = 0;
  bool any_bad = false;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    any_bad |= (w[j] & 0xfefefefeu) != 0;   // a byte other than 0 or 1
    mine += 4u - (uint32_t)__popc(w[j]);     // bytes 0/1: popc counts the solid ones
  }
  if (any_bad) atomicOr(bad, 1);
  mine = block_sum(mine);
  if (threadIdx.x == 0) counts[blockIdx.x] = mine;
}

// Pass 3 in lexicographic order (as tile_scatter_kernel): each thread's
// fluid cells take consecutive ranks after those of the threads before it
// (a block scan of the per-thread counts); inv is written 16 ints at a time,
// cells from shared memory in order.
__global__ void __launch_bounds__(kTileThreads)
    tile_scatter_lex_kernel(const uint8_t* __restrict__ flags, int64_t box, TileRanks ranks,
                            int32_t* cells, int32_t* inv) {
  __shared__ int32_t cell_at[kTileKeys];
  const int64_t k0 = (int64_t)blockIdx.x * kTileKeys + 16 * (int64_t)threadIdx.x;
  uint32_t w[4];
  const int valid = lex_chunk(flags, box, k0, w);
  uint32_t mine = 0, total;
#pragma unroll
  for (int j = 0; j < 4; ++j) mine += 4u - (uint32_t)__popc(w[j]);
  uint32_t at = block_prefix(mine, &total);
  const int64_t first = ranks.first(blockIdx.x);
  int32_t out[16];
#pragma unroll
  for (int b = 0; b < 16; ++b) {
    const bool fluid = ((w[b >> 2] >> (8 * (b & 3))) & 0xffu) == 0;
    out[b] = fluid ? (int32_t)(first + at) : -1;
    if (fluid) cell_at[at++] = (int32_t)(k0 + b);
  }
  if (valid == 16) {
    int4* o = reinterpret_cast<int4*>(inv + k0);
#pragma unroll
    for (int j = 0; j < 4; ++j) o[j] = make_int4(out[4 * j], out[4 * j + 1], out[4 * j + 2], out[4 * j + 3]);
  } else {
    for (int b = 0; b < valid; ++b) inv[k0 + b] = out[b];
  }
  __syncthreads();
  for (uint32_t j = threadIdx.x; j < total; j += kTileThreads) cells[first + j] = cell_at[j];
}

// Fluid index of the upwind neighbour of box cell (x, y, z) in direction q, or
// -1: the link bounces back (Sec. 2).
__device__ __forceinline__ int32_t upwind(int q, int32_t x, int32_t y, int32_t z, int32_t nx,
                                          int32_t ny, int32_t nz, uint32_t periodic,
                                          const int32_t* __restrict__ inv) {
  int32_t sx = x - cx(q), sy = y - cy(q), sz = z - cz(q);
  bool inside = true;
  if (sx < 0 || sx >= nx) {
    if (periodic & 1u) sx = sx < 0 ? sx + nx : sx - nx; else inside = false;
  }
  if (sy < 0 || sy >= ny) {
    if (periodic & 2u) sy = sy < 0 ? sy + ny : sy - ny; else inside = false;
  }
  if (sz < 0 || sz >= nz) {
    if (periodic & 4u) sz = sz < 0 ? sz + nz : sz - nz; else inside = false;
  }
  return inside ? inv[sx + nx * (sy + ny * sz)] : -1;
}

// Pull adjacency (Sec. 2): source slot of direction i for fluid cell n, in
// rows of ld >= n entries naming slot r ld + m (ld = n: the public layout).
__global__ void adjacency_kernel(int32_t nx, int32_t ny, int32_t nz, uint32_t periodic,
                                 const int32_t* __restrict__ cells,
                                 const int32_t* __restrict__ inv, int32_t* __restrict__ adj,
                                 int32_t n, int32_t ld) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t c = cells[i];
  const int32_t x = c % nx, y = (c / nx) % ny, z = c / (nx * ny);
#pragma unroll
  for (int q = 1; q < 19; ++q) {
    const int32_t m = upwind(q, x, y, z, nx, ny, nz, periodic, inv);
    adj[(q - 1) * ld + i] = m >= 0 ? q * ld + m : opp(q) * ld + i;
  }
}

// ---- short links (lbm::Links) -------------------------------------------------
// One warp per tile of kLinkTile cells, two cells per lane.  The tile's page
// list is a hash table of kLinkPages entries in shared memory, filled by the
// lanes as they meet pages (a row of 32 links mostly meets one or two): the
// entry of the page's low bits, or the next free one.  Which entry a page gets may
// depend on the order of the lanes, the slot a link names does not.  Bound by
// instructions, ~1,200 per tile (66% of issue slots busy): 0.86 ms for the
// 1024x256x256 bed, 1.25 with the list grown by ballots.
constexpr int kLinkWarps = 8;
__device__ __forceinline__ int32_t home_entry(int32_t page) {
  const int32_t e = page & 31;
  return e - (e >= kLinkPages ? 16 : 0);
}
// The entry of `page`, put into the table if it is not there; -1: it is full.
// (Out of line: 36 copies of the loop, two cells per lane at once, missed the
// instruction cache: 1.22 against 0.86 ms on the 1024x256x256 bed.)
__device__ __noinline__ int32_t find_entry(int32_t* table, int32_t page) {
  int32_t e = home_entry(page);
  for (int tries = 0; tries < kLinkPages; ++tries) {
    int32_t have = table[e];
    if (have < 0) have = atomicCAS(&table[e], -1, page);
    if (have < 0 || have == page) return e;
    e = e + 1 == kLinkPages ? 0 : e + 1;
  }
  return -1;
}
__global__ void __launch_bounds__(32 * kLinkWarps)
    short_links_kernel(int32_t nx, int32_t ny, int32_t nz, uint32_t periodic,
                       const int32_t* __restrict__ cells, const int32_t* __restrict__ inv,
                       int32_t n, int32_t ld, uint16_t* __restrict__ code,
                       int32_t* __restrict__ pages, int32_t* overflow) {
  __shared__ int32_t table[kLinkWarps][32];
  const int lane = threadIdx.x & 31;
  const int32_t tile = (int32_t)(blockIdx.x * kLinkWarps + threadIdx.x / 32);
  if (tile >= ld / kLinkTile) return;
  volatile int32_t* mine = table[threadIdx.x / 32];
  mine[lane] = -1;
  __syncwarp();
  bool full = false;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    const int32_t j = 32 * h + lane, i = tile * kLinkTile + j;
    const int32_t c = i < n ? cells[i] : 0;
    const int32_t yz = c / nx, z = yz / ny, x = c - yz * nx, y = yz - z * ny;
    int32_t m[18];
    // no face of the box within reach: the neighbours lie at fixed distances
    const bool inner = i < n && x > 0 && x < nx - 1 && y > 0 && y < ny - 1 && z > 0 && z < nz - 1;
    if (__all_sync(0xffffffffu, inner)) {
#pragma unroll
      for (int q = 1; q < 19; ++q) m[q - 1] = inv[c - (cx(q) + nx * (cy(q) + ny * cz(q)))];
    } else {
#pragma unroll
      for (int q = 1; q < 19; ++q)
        m[q - 1] = i < n ? upwind(q, x, y, z, nx, ny, nz, periodic, inv) : -1;
    }
#pragma unroll
    for (int q = 1; q < 19; ++q) {
      const uint32_t s = (uint32_t)m[q - 1];   // 2^32 - 1: bounce back
      const int32_t page = (int32_t)(s / kLinkPage);
      int32_t e = home_entry(page);
      if (mine[e] != page && m[q - 1] >= 0) {
        e = find_entry(table[threadIdx.x / 32], page);
        full |= e < 0;
      }
      uint32_t word = (uint32_t)e * kLinkPage + s % kLinkPage;
      if (m[q - 1] < 0) word = (uint32_t)((q & 1) ? kLinkPages : kLinkPages + 1) * kLinkPage + (uint32_t)j;
      code[(q - 1) * ld + i] = (uint16_t)word;
    }
  }
  if (full) *overflow = 1;
  __syncwarp();
  const int32_t first = tile * kLinkTile;
  pages[32 * tile + lane] = lane == kLinkPages       ? first + ld
                            : lane == kLinkPages + 1 ? first - ld
                                                     : max(mine[lane], 0) * kLinkPage;
}

// The public links (rows of n, slot q n + m) from 32-bit links in rows of ld
// (slot r ld + m); grid (cells, 18 rows).
__global__ void public_wide_kernel(const int32_t* __restrict__ wide, int32_t ld, int32_t n,
                                   int32_t* __restrict__ adj) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  const int32_t r = (int32_t)blockIdx.y;
  if (i >= n) return;
  const uint32_t s = (uint32_t)wide[r * ld + i];
  const uint32_t q = s / (uint32_t)ld;
  adj[r * n + i] = (int32_t)(q * (uint32_t)n + (s - q * (uint32_t)ld));
}

// The same from short links: one warp per 32 cells, lane e holding the tile's
// page entry e.
__global__ void __launch_bounds__(256)
    public_short_kernel(const uint16_t* __restrict__ code, const int32_t* __restrict__ pages,
                        int32_t ld, int32_t n, int32_t* __restrict__ adj) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ld) return;   // whole warps
  const int32_t entry = pages[32 * (i / kLinkTile) + (int32_t)(threadIdx.x & 31)];
  uint32_t word[18];
#pragma unroll
  for (int r = 0; r < 18; ++r) word[r] = code[r * ld + i];
#pragma unroll
  for (int r = 0; r < 18; ++r) {
    const int32_t e = (int32_t)(word[r] / kLinkPage);
    const int32_t m = __shfl_sync(0xffffffffu, entry, e) + (int32_t)(word[r] % kLinkPage);
    if (i < n) adj[r * n + i] = e < kLinkPages ? (r + 1) * n + m : opp(r + 1) * n + i;
  }
}

}  // namespace

int64_t one_wave_cells() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return 4 * (int64_t)sms * kSweepThreads;
}

int make_key_space(const int32_t dims[3], const lbm_ordering& ord, bool clamp_blocks,
                   KeySpace* ks) {
  if (!dims) return fail(LBM_EINVAL, "dims is NULL");
  for (int k = 0; k < 3; ++k)
    if (dims[k] < 1) return fail(LBM_EINVAL, "dims[%d] = %d must be >= 1", k, dims[k]);
  const int64_t box = (int64_t)dims[0] * dims[1] * dims[2];
  if (box >= (int64_t)1 << 31)
    return fail(LBM_EOVERFLOW, "box of %lld cells: the bounding box must stay below 2^31 cells",
                (long long)box);
  if (ord.kind < LBM_ORDER_LEX || ord.kind > LBM_ORDER_HILBERT)
    return fail(LBM_EINVAL, "unknown ordering kind %d", ord.kind);
  if (ord.periodic > 7u) return fail(LBM_EINVAL, "periodic mask %u has bits beyond 0..2", ord.periodic);
  KeySpace s{};
  s.kind = ord.kind;
  s.nx = dims[0];
  s.ny = dims[1];
  s.nz = dims[2];
  s.bx = s.by = s.bz = 1;
  if (ord.kind == LBM_ORDER_BLOCKED) {
    for (int k = 0; k < 3; ++k)
      if (ord.block[k] < 1) return fail(LBM_EINVAL, "block[%d] = %d must be >= 1", k, ord.block[k]);
    s.bx = ord.block[0];
    s.by = ord.block[1];
    s.bz = ord.block[2];
    // A block wider than the box along an axis visits that axis
    // lexicographically either way; clamping leaves the order unchanged but
    // keeps the walked key space small.  Keys handed out keep the literal
    // blocking factors.
    if (clamp_blocks) {
      if (s.bx > s.nx) s.bx = s.nx;
      if (s.by > s.ny) s.by = s.ny;
      if (s.bz > s.nz) s.bz = s.nz;
    }
    if ((double)s.bx * (double)s.by * (double)s.bz >= 9.0e18)
      return fail(LBM_EOVERFLOW, "blocking factors too large");
  }
  s.nbx = (s.nx + s.bx - 1) / s.bx;
  s.nby = (s.ny + s.by - 1) / s.by;
  s.nbz = (s.nz + s.bz - 1) / s.bz;
  s.hbits = 1;
  while ((1LL << s.hbits) < s.nx || (1LL << s.hbits) < s.ny || (1LL << s.hbits) < s.nz) ++s.hbits;
  // curve keys keep this many bits of each coordinate (key_of); a longer axis
  // would give several cells one key
  const int32_t key_bits = ord.kind == LBM_ORDER_MORTON2 ? 20 : 21;
  if (is_curve(ord.kind) && s.hbits > key_bits)
    return fail(LBM_EOVERFLOW, "an axis of more than 2^%d cells exceeds the keys of this ordering",
                (int)key_bits);
  if (ord.kind == LBM_ORDER_BLOCKED) {
    s.size = (uint64_t)(s.nbx * s.nby * s.nbz) * (uint64_t)(s.bx * s.by * s.bz);
  } else if (ord.kind == LBM_ORDER_HILBERT) {
    // the Hilbert curve wanders through the whole enclosing cube
    s.size = 1ull << (3 * s.hbits);
  } else {
    s.size = ~0ull;
    // lexicographic and Z-curve keys are monotone in each coordinate: the
    // far corner holds the largest key
    s.size = key_of(s, s.nx - 1, s.ny - 1, s.nz - 1) + 1;
  }
  // for the walk, whose blocks are no larger than the box: literal blocks may
  // span a key space of more than 64 bits, and size is then no measure of it
  if (ord.kind == LBM_ORDER_BLOCKED && clamp_blocks && s.size < (1ull << 31)) {
    s.by_bsz = fixed_div((uint32_t)(s.bx * s.by * s.bz));
    s.by_bx = fixed_div((uint32_t)s.bx);
    s.by_bxy = fixed_div((uint32_t)(s.bx * s.by));
    s.by_nbx = fixed_div((uint32_t)s.nbx);
    s.by_nbxy = fixed_div((uint32_t)(s.nbx * s.nby));
  }
  if (is_curve(ord.kind)) {
    s.levels = ord.kind == LBM_ORDER_HILBERT && s.hbits < 4 ? s.hbits : 4;
    for (int a = 0; a < 3; ++a) {
      const uint64_t e[3] = {a == 0, a == 1, a == 2};
      s.unit[a] = ord.kind == LBM_ORDER_MORTON1   ? 1u << a
                  : ord.kind == LBM_ORDER_MORTON2 ? 1u << (2 * a)
                                                  : (uint32_t)hilbert_encode(s.levels, e[0], e[1], e[2]);
    }
  }
  *ks = s;
  return LBM_OK;
}

int public_links(const lbm_sparse* sp_c, const int32_t** out) {
  // logically const: the public links are a cached view of the steps' links
  lbm_sparse* sp = const_cast<lbm_sparse*>(sp_c);
  if (!sp->adj) {
    const cudaStream_t stream = sp->stream;
    int32_t* adj = nullptr;
    if (dev_alloc(&adj, sizeof(int32_t) * 18 * (size_t)(sp->n > 0 ? sp->n : 1), stream, true) !=
        cudaSuccess) {
      cudaGetLastError();
      return fail(LBM_ENOMEM, "public adjacency allocation failed (%lld fluid cells)",
                  (long long)sp->n);
    }
    const Links links = state_links(sp);
    if (sp->n > 0 && links.wide)
      public_wide_kernel<<<dim3((unsigned)((sp->n + 255) / 256), 18), 256, 0, stream>>>(
          links.wide, (int32_t)sp->ld, (int32_t)sp->n, adj);
    else if (sp->n > 0)
      public_short_kernel<<<(unsigned)((sp->ld + 255) / 256), 256, 0, stream>>>(
          links.code, links.pages, (int32_t)sp->ld, (int32_t)sp->n, adj);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) {
      dev_free(adj, stream, true);
      cudaStreamSynchronize(stream);
      return cuda_fail(e, "public adjacency");
    }
    sp->adj = adj;
  }
  if (out) *out = sp->adj;
  return LBM_OK;
}

}  // namespace lbm

using namespace lbm;

extern "C" int lbm_ordering_keys(const int32_t dims[3], lbm_ordering ord, uint64_t* keys_dev,
                                 void* stream) {
  clear_error();
  KeySpace ks;
  int rc = make_key_space(dims, ord, false, &ks);
  if (rc) return rc;
  if (!keys_dev) return fail(LBM_EINVAL, "keys_dev is NULL");
  const int64_t box = ks.nx * ks.ny * ks.nz;
  const int threads = 256;
  keys_kernel<<<(unsigned)((box + threads - 1) / threads), threads, 0, (cudaStream_t)stream>>>(
      ks, keys_dev, box);
  LBM_CUDA_TRY(cudaGetLastError());
  return LBM_OK;
}

extern "C" int lbm_build_sparse(const uint8_t* flags, const int32_t dims[3], lbm_ordering ord,
                                void* stream_v, lbm_sparse** out) {
  clear_error();
  if (!out) return fail(LBM_EINVAL, "out is NULL");
  *out = nullptr;
  if (!flags) return fail(LBM_EINVAL, "flags is NULL");
  KeySpace ks;
  int rc = make_key_space(dims, ord, true, &ks);
  if (rc) return rc;
  cudaStream_t stream = (cudaStream_t)stream_v;
  const int64_t box = ks.nx * ks.ny * ks.nz;
  const int64_t ntiles = (int64_t)((ks.size + kTileKeys - 1) / kTileKeys);
  if (ntiles >= (int64_t)1 << 31) return fail(LBM_EOVERFLOW, "key space too large");
  const int64_t nspans = (ntiles + kScanSpan - 1) / kScanSpan;
  // the aligned cubes a curve's tiles are, counted over the box
  const bool curve = is_curve(ks.kind);
  const int64_t cubes = ((ks.nx + 15) / 16) * ((ks.ny + 15) / 16) * ((ks.nz + 15) / 16);
  // host flags (pinned or pageable) are copied to the device first
  cudaPointerAttributes attr{};
  const cudaError_t pe = cudaPointerGetAttributes(&attr, flags);
  if (pe != cudaSuccess) return cuda_fail(pe, "cudaPointerGetAttributes(flags)");
  const bool on_host = attr.type == cudaMemoryTypeHost || attr.type == cudaMemoryTypeUnregistered;

  // scratch: tile counts, tile offsets, span totals, a curve's active tiles
  uint32_t* counts = nullptr;
  uint32_t* offsets = nullptr;
  int64_t* span = nullptr;
  uint32_t* active = nullptr;
  int64_t* scal = nullptr;  // [0] total, [1] bad-flag word, [2] short links overflow, [3] active tiles
  uint8_t* flags_copy = nullptr;
  lbm_sparse* sp = new lbm_sparse{};
  sp->magic = kMagicSparse;
  for (int k = 0; k < 3; ++k) sp->dims[k] = dims[k];
  sp->ord = ord;
  sp->stream = stream;
  auto release = [&](void* p) { dev_free(p, stream, true); };
  auto cleanup = [&](int status) {
    release(counts);
    release(offsets);
    release(span);
    release(active);
    release(scal);
    release(flags_copy);
    if (status != LBM_OK) {
      release(sp->cells);
      release(sp->inv);
      release(sp->adj);
      release(sp->adj_ld);
      release(sp->code);
      release(sp->pages);
      delete sp;
    }
    cudaStreamSynchronize(stream);
    return status;
  };
  if (dev_alloc(&counts, sizeof(uint32_t) * ntiles, stream, true) != cudaSuccess ||
      dev_alloc(&offsets, sizeof(uint32_t) * ntiles, stream, true) != cudaSuccess ||
      dev_alloc(&span, sizeof(int64_t) * nspans, stream, true) != cudaSuccess ||
      (curve && dev_alloc(&active, sizeof(uint32_t) * cubes, stream, true) != cudaSuccess) ||
      dev_alloc(&scal, sizeof(int64_t) * 4, stream, true) != cudaSuccess ||
      dev_alloc(&sp->inv, sizeof(int32_t) * box, stream, true) != cudaSuccess) {
    cudaGetLastError();
    return cleanup(fail(LBM_ENOMEM, "device allocation failed (box %lld cells)", (long long)box));
  }
  if (cudaMemsetAsync(scal, 0, sizeof(int64_t) * 4, stream) != cudaSuccess)
    return cleanup(cuda_fail(cudaGetLastError(), "cudaMemsetAsync"));
  const uint8_t* flags_dev = flags;
  if (on_host) {
    if (dev_alloc(&flags_copy, (size_t)box, stream, true) != cudaSuccess) {
      cudaGetLastError();
      return cleanup(fail(LBM_ENOMEM, "device copy of the host flags (%lld bytes) failed",
                          (long long)box));
    }
    const cudaError_t ce =
        cudaMemcpyAsync(flags_copy, flags, (size_t)box, cudaMemcpyHostToDevice, stream);
    if (ce != cudaSuccess) return cleanup(cuda_fail(ce, "cudaMemcpyAsync(flags)"));
    flags_dev = flags_copy;
  }
  // lexicographic order with 16-byte aligned flags takes the vector passes
  const bool lex_vec = ks.kind == LBM_ORDER_LEX && reinterpret_cast<uintptr_t>(flags_dev) % 16 == 0;
  if (lex_vec)
    tile_count_lex_kernel<<<(unsigned)ntiles, kTileThreads, 0, stream>>>(flags_dev, box, counts,
                                                                        (int*)(scal + 1));
  else if (curve) {
    if (cudaMemsetAsync(counts, 0, sizeof(uint32_t) * ntiles, stream) != cudaSuccess)
      return cleanup(cuda_fail(cudaGetLastError(), "cudaMemsetAsync"));
    active_tiles_kernel<<<(unsigned)((ntiles + 255) / 256), 256, 0, stream>>>(
        ks, ntiles, cubes, active, (uint32_t*)(scal + 3));
    cube_count_kernel<<<(unsigned)cubes, kTileThreads, 0, stream>>>(
        ks, flags_dev, active, (const uint32_t*)(scal + 3), counts, (int*)(scal + 1));
  } else {
    (small_blocked(ks) ? tile_count_kernel<true> : tile_count_kernel<false>)
        <<<(unsigned)ntiles, kTileThreads, 0, stream>>>(ks, flags_dev, counts, (int*)(scal + 1));
  }
  tile_scan_kernel<<<(unsigned)nspans, 1024, 0, stream>>>(counts, ntiles, offsets, span);
  span_scan_kernel<<<1, 1024, 0, stream>>>(span, nspans, scal);
  const TileRanks ranks{offsets, span};
  int64_t host_scal[2] = {0, 0};
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(host_scal, scal, sizeof(host_scal), cudaMemcpyDeviceToHost, stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) return cleanup(cuda_fail(e, "sparse assembly: tile count/scan"));
  if (host_scal[1] != 0) return cleanup(fail(LBM_EFLAGS, "flags must be 0 (fluid) or 1 (solid)"));
  const int64_t n = host_scal[0];
  const int64_t ld = row_stride(n);
  if (19 * ld >= ((int64_t)1 << 31))
    return cleanup(fail(LBM_EOVERFLOW,
                        "%lld fluid cells: 19*L PDF slots (rows of L = %lld, N rounded up to 64) "
                        "exceed the int32 adjacency range",
                        (long long)n, (long long)ld));
  sp->n = n;
  sp->ld = ld;
  const size_t nn = (size_t)(n > 0 ? n : 1);
  // Lists of more than two waves take short links.  A smaller list's steps run
  // from L2, where bytes count less than the decoding.  MFLUP/s with short /
  // 32-bit links: 29,479 cells FP64 storage 8,148 / 8,890, FP32S 17,590 /
  // 17,853, FP16S 18,730 / 18,446; 221,119 cells FP64 storage 19,623 / 21,163,
  // FP32S 37,045 / 43,126, FP16S 36,547 / 44,828;
  // 413,546 cells FP64 storage 16,411 / 14,675, FP32S 43,166 / 38,031.
  const bool brief = n > small_list_cells();
  const auto alloc_wide = [&]() {   // they are the public links when ld == n
    int32_t** links = ld == n ? &sp->adj : &sp->adj_ld;
    return dev_alloc(links, sizeof(int32_t) * 18 * (size_t)(ld > 0 ? ld : 1), stream, true);
  };
  cudaError_t ea = dev_alloc(&sp->cells, sizeof(int32_t) * nn, stream, true);
  if (brief) {
    if (ea == cudaSuccess) ea = dev_alloc(&sp->code, sizeof(uint16_t) * 18 * (size_t)ld, stream, true);
    if (ea == cudaSuccess)
      ea = dev_alloc(&sp->pages, sizeof(int32_t) * 32 * (size_t)(ld / kLinkTile), stream, true);
  } else if (ea == cudaSuccess) {
    ea = alloc_wide();
  }
  if (ea != cudaSuccess) {
    cudaGetLastError();
    return cleanup(fail(LBM_ENOMEM, "device allocation failed (%lld fluid cells)", (long long)n));
  }
  if (lex_vec)
    tile_scatter_lex_kernel<<<(unsigned)ntiles, kTileThreads, 0, stream>>>(
        flags_dev, box, ranks, sp->cells, sp->inv);
  else if (curve)
    cube_scatter_kernel<<<(unsigned)cubes, kTileThreads, 0, stream>>>(
        ks, flags_dev, active, (const uint32_t*)(scal + 3), ranks, sp->cells, sp->inv);
  else
    (small_blocked(ks) ? tile_scatter_kernel<true> : tile_scatter_kernel<false>)
        <<<(unsigned)ntiles, kTileThreads, 0, stream>>>(ks, flags_dev, ranks, sp->cells, sp->inv);
  const auto write_wide = [&]() {
    if (n == 0) return;
    adjacency_kernel<<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(
        dims[0], dims[1], dims[2], ord.periodic, sp->cells, sp->inv,
        ld == n ? sp->adj : sp->adj_ld, (int32_t)n, (int32_t)ld);
  };
  if (brief) {
    const unsigned tiles = (unsigned)(ld / kLinkTile);
    short_links_kernel<<<(tiles + kLinkWarps - 1) / kLinkWarps, 32 * kLinkWarps, 0, stream>>>(
        dims[0], dims[1], dims[2], ord.periodic, sp->cells, sp->inv, (int32_t)n, (int32_t)ld,
        sp->code, sp->pages, (int32_t*)(scal + 2));
    e = cudaMemcpyAsync(host_scal, scal + 2, sizeof(int64_t), cudaMemcpyDeviceToHost, stream);
  } else {
    write_wide();
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  if (e == cudaSuccess && brief && host_scal[0] != 0) {
    // a tile's neighbours lie in more than kLinkPages pages
    release(sp->code);
    release(sp->pages);
    sp->code = nullptr;
    sp->pages = nullptr;
    if (alloc_wide() != cudaSuccess) {
      cudaGetLastError();
      return cleanup(fail(LBM_ENOMEM, "device allocation failed (%lld fluid cells)", (long long)n));
    }
    write_wide();
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  }
  if (e != cudaSuccess) return cleanup(cuda_fail(e, "sparse assembly: scatter/links"));
  *out = sp;
  return cleanup(LBM_OK);
}

extern "C" int lbm_sparse_info(const lbm_sparse* sp, int64_t* n_fluid, const int32_t** cells_dev,
                               const int32_t** adj_dev, const int32_t** inv_dev) {
  clear_error();
  if (!sp || sp->magic != kMagicSparse) return fail(LBM_EINVAL, "not a sparse handle");
  if (n_fluid) *n_fluid = sp->n;
  if (cells_dev) *cells_dev = sp->cells;
  if (adj_dev) {
    const int rc = public_links(sp, adj_dev);
    if (rc != LBM_OK) return rc;
  }
  if (inv_dev) *inv_dev = sp->inv;
  return LBM_OK;
}
