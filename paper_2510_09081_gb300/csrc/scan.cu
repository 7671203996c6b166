// A4: per-voxel list offsets by an exclusive prefix sum over the counts of the
// voxels that receive a list (Sec. 3.3; the first half of the linearized
// layered fragment buffer it extends). Single-pass decoupled look-back scan:
// tiles take ids in launch order from an atomic counter, publish their
// aggregate, then their inclusive prefix once a warp has looked back to a
// published prefix. Every wait is bounded; a wait that gives up sets the
// timeout bit and the tile carries on with the sum it has.
//
// The same pass sums the count and occupancy fields over all voxels, which pass 2
// compares with the fragment and occupancy totals that pass 1 accumulated
// separately: a difference means that a 16-bit field overflowed.
#include "launch.h"
#include "scan_tile.cuh"

namespace vrt {

constexpr int kSpinLimit = 1 << 22;

__global__ void __launch_bounds__(kTileThreads, 8) k_scan(GridDev g, int all_visible,
                                                       unsigned long long* tile_state,
                                                       uint32_t n_tiles, int stall_tile,
                                                       int spin_limit) {
  __shared__ uint32_t s_tile;
  __shared__ uint32_t s_warp[kTileWarps];
  __shared__ uint32_t s_prefix;
  __shared__ uint32_t s_red[4][kTileWarps];
  dependency_wait();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    s_tile = atomicAdd(&g.st->scan_tile_counter, 1u);
  }
  __syncthreads();
  const uint32_t tile = s_tile;
  uint4 word[kTileRows];
  uint32_t vis = 0;  // 4 bits a row: the voxels that receive a list
#pragma unroll
  for (int q = 0; q < kTileRows; ++q) {
    const uint32_t i = tile_word(tile, q);
    word[q] = *reinterpret_cast<const uint4*>(g.word + i);
    vis |= (all_visible ? 0xfu : (g.vis[i >> 5] >> (i & 31)) & 0xfu) << (4 * q);
  }
  uint2 cnt[kTileRows];
  uint32_t sum[kTileRows], excl[kTileRows];
  uint32_t cf = 0, of = 0, occupied = 0, visible = 0, maxc = 0;  // cf, of: below 2^28 in a tile
#pragma unroll
  for (int q = 0; q < kTileRows; ++q) {
    const uint32_t w[4] = {word[q].x, word[q].y, word[q].z, word[q].w};
    cnt[q] = masked(pack_counts(word[q]), vis >> (4 * q));
    sum[q] = sum_counts(cnt[q]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t c = w[k] & 0xffffu;
      cf += c;
      of += w[k] >> 16;
      occupied += c != 0;
      visible += c != 0 && ((vis >> (4 * q + k)) & 1u);
      maxc = max(maxc, c);
    }
  }
  cf = __reduce_add_sync(0xffffffffu, cf);
  of = __reduce_add_sync(0xffffffffu, of);
  occupied = __reduce_add_sync(0xffffffffu, (visible << 16) | occupied);  // at most 512 each
  maxc = __reduce_max_sync(0xffffffffu, maxc);
  if (lane == 0) {
    s_red[0][warp] = cf; s_red[1][warp] = of; s_red[2][warp] = occupied; s_red[3][warp] = maxc;
  }
  const uint32_t warp_sum = tile_rows_exclusive(sum, excl);
  if (lane == 0) s_warp[warp] = warp_sum;
  __syncthreads();
  uint32_t warp_off = 0, agg = 0;
#pragma unroll
  for (int q = 0; q < kTileWarps; ++q) {
    const uint32_t v = s_warp[q];
    if (q < warp) warp_off += v;
    agg += v;
  }
  if (warp == 0) {
    bool gave_up;
    const unsigned long long before =
        look_back(tile_state, tile, agg, (int)tile != stall_tile, spin_limit, &gave_up);
    if (lane == 0) {
      if (gave_up) set_err(g.st, kErrTimeout);
      s_prefix = (uint32_t)before;
      if (tile == n_tiles - 1) {
        const unsigned long long total = before + agg;
        g.st->list_tail = (uint32_t)total;
        if (total > g.list_cap) set_err(g.st, kErrOverflow);
      }
    }
  }
  __syncthreads();
  const uint32_t run = s_prefix + warp_off;
#pragma unroll
  for (int q = 0; q < kTileRows; ++q) {
    const uint32_t bits = vis >> (4 * q);
    uint4 e;  // list end (pass 2 fills below it)
    e.x = run + excl[q] + (cnt[q].x & 0xffffu);
    e.y = e.x + (cnt[q].x >> 16);
    e.z = e.y + (cnt[q].y & 0xffffu);
    e.w = e.z + (cnt[q].y >> 16);
    if (!(bits & 1u)) e.x = kCulledStart;
    if (!(bits & 2u)) e.y = kCulledStart;
    if (!(bits & 4u)) e.z = kCulledStart;
    if (!(bits & 8u)) e.w = kCulledStart;
    *reinterpret_cast<uint4*>(g.cur + tile_word(tile, q)) = e;
  }

  if (tid == 0) {  // counters
    uint32_t a0 = 0, a1 = 0, a2 = 0, a3 = 0;
    for (int q = 0; q < kTileWarps; ++q) {
      a0 += s_red[0][q]; a1 += s_red[1][q]; a2 += s_red[2][q];
      a3 = max(a3, s_red[3][q]);
    }
    ScanPart& p = g.st->scan_part[tile % kScanParts];
    if (a0) atomicAdd(&p.count_field, (unsigned long long)a0);
    if (a1) atomicAdd(&p.occ_field, (unsigned long long)a1);
    if (a2) atomicAdd(&p.voxels, (unsigned long long)(a2 >> 16) << 32 | (a2 & 0xffffu));
    if (a3) atomicMax(&p.max_count, a3);
  }
}

int launch_scan(const GridDev& g, int all_visible, unsigned long long* tile_state, uint32_t n_tiles,
                int stall_tile, int spin_limit, const Queue& q) {
  launch(k_scan, n_tiles, kTileThreads, q, g, all_visible, tile_state, n_tiles, stall_tile,
                 spin_limit > 0 ? spin_limit : kSpinLimit);
  return 1;
}

}  // namespace vrt
