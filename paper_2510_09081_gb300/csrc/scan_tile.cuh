// What the two list-offset scans (scan.cu, scan_noalloc.cu) share: the order a
// tile is read in, its sums, and the look-back over the tiles before it.
//
// A tile of 4096 words is one block's; each warp has 512 consecutive ones and
// reads them in 4 rows of 128, a lane the 16 bytes beside its neighbour's, so every
// load and store of a warp is one run of 512 bytes. (16 consecutive words to a
// thread need one warp scan instead of four, but each request touches 32 sectors
// and uses half of each.) What bounds the scan is the chain ticket - words -
// look-back - offsets that each block waits through, so the bytes in flight decide:
// counts are held two to a register, which lets 8 blocks of 256 threads be resident in
// the grid's scan and 6 in the stand-alone one (8 there spill and gain nothing).
// Together: 512^3 voxels 0.297 -> 0.199 ms (1.09 GB, 5.5 TB/s), 256^3 0.047 -> 0.033.
// Reading 64 to 256 states of the look-back at once instead of 32 was no faster
// (0.240, 0.248 against 0.234 ms): the registers cost more than the windows save.
#pragma once

#include <stdint.h>

namespace vrt {

constexpr int kTileThreads = 256;
constexpr int kTileRows = 4;                         // 16-byte loads of a thread
constexpr int kTileWords = kTileThreads * 4 * kTileRows;  // 4096
constexpr int kTileWarps = kTileThreads / 32;

// Tile state: flag (0 none, 1 aggregate, 2 inclusive prefix) in bits 62-63, the
// 62-bit sum below it.
constexpr unsigned long long kTileAgg = 1ull << 62, kTilePrefix = 2ull << 62;
constexpr unsigned long long kTileSum = (1ull << 62) - 1;

// Index of the first of the 4 words of row q of this thread.
__device__ __forceinline__ uint32_t tile_word(uint32_t tile, int q) {
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  return tile * kTileWords + warp * (kTileRows * 128) + q * 128 + lane * 4;
}

// The low 16 bits (counts) of 4 words as two registers; masked() drops those of the
// words whose bit in `bits` is clear, and the counts come back one by one below.
__device__ __forceinline__ uint2 pack_counts(uint4 w) {
  return make_uint2(__byte_perm(w.x, w.y, 0x5410), __byte_perm(w.z, w.w, 0x5410));
}
__device__ __forceinline__ uint2 masked(uint2 c, uint32_t bits) {
  return make_uint2(c.x & ((bits & 1u) * 0xffffu | (bits & 2u) * 0x7fff8000u),
                    c.y & (((bits >> 2) & 1u) * 0xffffu | ((bits >> 2) & 2u) * 0x7fff8000u));
}
__device__ __forceinline__ uint32_t sum_counts(uint2 c) {
  return (c.x & 0xffffu) + (c.x >> 16) + (c.y & 0xffffu) + (c.y >> 16);
}

// Exclusive prefix sums, within the warp's 512 words, of the thread's row sums
// (each at most 4 * 65535, so a warp's sum stays below 2^26); returns the warp's sum.
__device__ __forceinline__ uint32_t tile_rows_exclusive(const uint32_t sum[kTileRows],
                                                        uint32_t excl[kTileRows]) {
  const int lane = threadIdx.x & 31;
  uint32_t incl[kTileRows];
#pragma unroll
  for (int q = 0; q < kTileRows; ++q) incl[q] = sum[q];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1)
#pragma unroll
    for (int q = 0; q < kTileRows; ++q) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl[q], o);
      if (lane >= o) incl[q] += y;
    }
  uint32_t before = 0;
#pragma unroll
  for (int q = 0; q < kTileRows; ++q) {
    excl[q] = before + incl[q] - sum[q];
    before += __shfl_sync(0xffffffffu, incl[q], 31);
  }
  return before;
}

__device__ __forceinline__ unsigned long long load_state(const unsigned long long* p) {
  return *(volatile const unsigned long long*)p;
}

// Called by one whole warp: the sum of the tiles before `tile` (those that
// follow it, from the nearest published prefix). Publishes the tile's aggregate
// first and its inclusive prefix after. Every wait is bounded: after `spin_limit`
// polls it gives up, sets *gave_up and returns the sum it has. A tile told not to
// publish (testing) makes the waits of the tiles after it run out.
__device__ __forceinline__ unsigned long long look_back(unsigned long long* state, uint32_t tile,
                                                        uint32_t agg, bool publish, int spin_limit,
                                                        bool* gave_up) {
  const int lane = threadIdx.x & 31;
  *gave_up = false;
  if (tile == 0) {
    if (lane == 0 && publish) atomicExch(&state[0], kTilePrefix | agg);
    return 0;
  }
  if (lane == 0 && publish) atomicExch(&state[tile], kTileAgg | agg);
  unsigned long long v = 0;  // this lane's part of the sum
  int spins = 0;
  bool done = false;
  for (int j = (int)tile - 1; !done; j -= 32) {
    const int idx = j - lane;
    unsigned long long s = idx >= 0 ? load_state(&state[idx]) : kTilePrefix;
    while (__any_sync(0xffffffffu, (s >> 62) == 0)) {
      if (++spins > spin_limit) break;
      if ((s >> 62) == 0) {
        __nanosleep(20);
        s = load_state(&state[idx]);
      }
    }
    if (spins > spin_limit) {
      *gave_up = true;
      break;
    }
    const uint32_t pmask = __ballot_sync(0xffffffffu, (s >> 62) == 2);
    const int stop = pmask ? __ffs(pmask) - 1 : 31;  // nearest published prefix
    if (lane <= stop) v += s & kTileSum;
    done = pmask != 0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0 && publish) atomicExch(&state[tile], kTilePrefix | ((v + agg) & kTileSum));
  return v;
}

}  // namespace vrt
