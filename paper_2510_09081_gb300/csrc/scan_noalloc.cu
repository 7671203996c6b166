// vrt_scan_counts_noalloc: the list-offset scan as a stand-alone entry point
// that allocates no device memory.
//
// Some callers cannot call cudaMalloc at the point where they need the scan:
// code running inside a memory pool or arena that owns all device memory of
// the process, callers that must not fragment or grow memory mid-frame, and
// real-time loops where an allocation could block on the driver. This variant
// takes the look-back scratch (one 64-bit state per tile and a tile counter)
// from a fixed file-scope device array instead of a caller or library
// allocation. The array is part of the library image, so every GPU that loads
// the library holds it (about 256 KB) until the process exits.
//
// The kernel computes the exclusive prefix sum of the per-voxel counts (low 16
// bits of each packed word) of marked voxels, and their total, over the same tiles
// and by the same look-back as the grid's scan (scan_tile.cuh). Sums are carried in
// 62 bits, so a total beyond 2^32 - 1, where the 32-bit offsets wrap, is detected
// and reported. The scratch is cleared by a kernel that this one is chained to.
// 256^3 voxels, call after call: 43.7 us with two memsets and 16 consecutive words
// to a thread, 30.6 now (136 MB, 4.4 TB/s).
#include <cooperative_groups.h>

#include <atomic>
#include <mutex>
#include <string>

#include "launch.h"
#include "scan_tile.cuh"
#include "vrt.h"

namespace vrt {
namespace {

constexpr uint32_t kNaMaxTiles = 32768;          // 134,217,728 voxels (512^3)
// Calls of up to this many tiles (a 32^3 grid) run as one cluster, the largest that
// needs no opt-in: one launch instead of two. Call after call from the host 10.8 ->
// 8.9 us, as nodes of a graph 3.2 -> 2.9 us (with two memsets and a kernel 11.3 and
// 8.2 us).
constexpr uint32_t kClusterTiles = 8;
constexpr int kNaSpinLimit = 1 << 22;
// status bits of status_out
constexpr uint32_t kNaGaveUp = 1u, kNaWrapped = 2u;

// Scratch: tile states, then the tile counter. Shared by every call.
struct NoAllocScratch {
  unsigned long long state[kNaMaxTiles];
  unsigned int tile_counter;
};
static __device__ __align__(256) NoAllocScratch g_noalloc_scratch;

// CLUSTER: the blocks are one cluster, which swaps its sums over distributed shared
// memory: no scratch, so no kernel to clear it, no ticket and no look-back. Blocks
// past the last tile (the cluster's size is a power of two) only keep the barriers.
template <bool CLUSTER>
__global__ void __launch_bounds__(kTileThreads, 6) k_scan_noalloc(
    NoAllocScratch* scratch, const uint32_t* __restrict__ words, const uint32_t* __restrict__ marks,
    uint32_t* __restrict__ offsets, uint32_t* total_out, uint32_t* status_out, uint32_t n_tiles,
    int stall_tile, int spin_limit) {
  __shared__ uint32_t s_tile;
  __shared__ uint32_t s_prefix, s_sum;
  __shared__ uint32_t s_warp[kTileWarps];
  const uint32_t zero = dependency_wait();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (!CLUSTER) {
    if (tid == 0) s_tile = atomicAdd(&scratch->tile_counter, 1u);
    __syncthreads();
  }
  // the loads of words and marks, which may be read-only ones, wait through `zero`
  const uint32_t tile = (CLUSTER ? blockIdx.x : s_tile) + zero;
  const bool some = !CLUSTER || tile < n_tiles;
  uint2 cnt[kTileRows];
  uint32_t sum[kTileRows], excl[kTileRows];
#pragma unroll
  for (int q = 0; q < kTileRows; ++q) {
    cnt[q] = make_uint2(0u, 0u);
    if (!some) continue;
    const uint32_t i = tile_word(tile, q);
    const uint32_t bits = marks ? marks[i >> 5] >> (i & 31) : 0xfu;
    cnt[q] = masked(pack_counts(*reinterpret_cast<const uint4*>(words + i)), bits);
  }
#pragma unroll
  for (int q = 0; q < kTileRows; ++q) sum[q] = sum_counts(cnt[q]);
  const uint32_t warp_sum = tile_rows_exclusive(sum, excl);
  if (lane == 0) s_warp[warp] = warp_sum;
  __syncthreads();
  uint32_t warp_off = 0, agg = 0;  // the tile's sums stay below 4096 * 65535 < 2^28
#pragma unroll
  for (int q = 0; q < kTileWarps; ++q) {
    if (q < warp) warp_off += s_warp[q];
    agg += s_warp[q];
  }
  uint32_t cluster_before = 0;  // below 2^31
  if (CLUSTER) {
    auto cluster = cooperative_groups::this_cluster();
    if (tid == 0) s_sum = agg;
    cluster.sync();
    if (warp == 0)
      cluster_before = __reduce_add_sync(
          0xffffffffu, (uint32_t)lane < tile ? *cluster.map_shared_rank(&s_sum, (unsigned)lane) : 0u);
    cluster.sync();  // no block leaves while its sum is being read
  }
  if (warp == 0) {
    bool gave_up = false;
    const unsigned long long before =
        CLUSTER ? cluster_before
                : look_back(scratch->state, tile, agg, (int)tile != stall_tile, spin_limit, &gave_up);
    if (lane == 0) {
      if (gave_up && status_out) atomicOr(status_out, kNaGaveUp);
      s_prefix = (uint32_t)before;
      if (tile == n_tiles - 1) {
        const unsigned long long total = before + agg;
        if (total_out) *total_out = (uint32_t)total;
        if (total > 0xffffffffull && status_out) atomicOr(status_out, kNaWrapped);
      }
    }
  }
  __syncthreads();
  if (!some) return;
  // offsets are the low 32 bits of the prefix sums (they wrap past 2^32 - 1)
  const uint32_t run = s_prefix + warp_off;
#pragma unroll
  for (int q = 0; q < kTileRows; ++q) {
    uint4 o;
    o.x = run + excl[q];
    o.y = o.x + (cnt[q].x & 0xffffu);
    o.z = o.y + (cnt[q].x >> 16);
    o.w = o.z + (cnt[q].y & 0xffffu);
    *reinterpret_cast<uint4*>(offsets + tile_word(tile, q)) = o;
  }
}

// Testing: the tile that skips its publish (-1: none).
std::atomic<long long> g_stall_tile{-1};

// Device address of the scratch array, looked up once per device.
constexpr int kMaxDevices = 64;
std::mutex g_setup_mutex;
void* g_scratch_addr[kMaxDevices] = {};

}  // namespace

void set_noalloc_scan_stall(long long tile) { g_stall_tile.store(tile); }

}  // namespace vrt

extern thread_local std::string g_create_error;  // message returned by vrt_last_error(NULL)

extern "C" vrt_status vrt_scan_counts_noalloc(const uint32_t* words, const uint32_t* marks,
                                              uint32_t* offsets, uint64_t n_voxels,
                                              uint32_t* total_out, uint32_t* status_out,
                                              void* cuda_stream) {
  using namespace vrt;
  auto fail = [](vrt_status s, const char* m) {
    g_create_error = m;
    return s;
  };
  if (!words || !offsets) return fail(VRT_ERR_INVALID_ARG, "words and offsets must not be NULL");
  if (n_voxels == 0 || n_voxels % kTileWords != 0)
    return fail(VRT_ERR_INVALID_ARG, "n_voxels must be a positive multiple of 4096");
  if (n_voxels > (uint64_t)kNaMaxTiles * kTileWords)
    return fail(VRT_ERR_INVALID_ARG,
                "n_voxels exceeds the no-allocation scan's fixed scratch (at most 134217728)");
  if (((uintptr_t)words | (uintptr_t)offsets) & 15u)
    return fail(VRT_ERR_INVALID_ARG, "words and offsets must be 16-byte aligned");
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
    return fail(VRT_ERR_CUDA, "cudaGetDevice failed");
  void* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_addr[dev]) {
      void* p = nullptr;
      const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess || !p) return fail(VRT_ERR_CUDA, cudaGetErrorString(e));
      g_scratch_addr[dev] = p;
    }
    scratch = g_scratch_addr[dev];
  }
  const uint32_t n_tiles = (uint32_t)(n_voxels / kTileWords);
  const Queue q = {(cudaStream_t)cuda_stream, stream_alone((cudaStream_t)cuda_stream)};
  NoAllocScratch* sc = (NoAllocScratch*)scratch;
  const long long stall = g_stall_tile.load();
  if (n_tiles <= kClusterTiles && stall < 0) {
    unsigned size = 1;
    while (size < n_tiles) size *= 2;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(size);
    c.blockDim = dim3(kTileThreads);
    c.stream = q.s;
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = size;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = q.chained ? 2 : 1;
    cudaLaunchKernelEx(&c, k_scan_noalloc<true>, sc, words, marks, offsets, total_out, status_out,
                       n_tiles, -1, 0);
  } else {
    // the states of the tiles this call uses and the tile counter start at zero
    launch_reset(reinterpret_cast<uint32_t*>(sc->state), 2 * n_tiles, &sc->tile_counter, 1, q);
    launch(k_scan_noalloc<false>, n_tiles, kTileThreads, q, sc, words, marks, offsets, total_out,
           status_out, n_tiles, stall >= 0 ? (int)stall : -1, stall >= 0 ? kSpinLimitTest : kNaSpinLimit);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(VRT_ERR_CUDA, cudaGetErrorString(e));
  return VRT_OK;
}
