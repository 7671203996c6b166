// Empty-space skipping for the trace and the cull march: for every 4^3 brick,
// the Chebyshev distance (in bricks, capped at kBrickDistMax) to the nearest
// brick that holds an occupied voxel (count > 0); 0 marks such a brick. A ray
// in a brick at distance k >= 1 can cross the whole cube of bricks within
// k - 1 of it in one step, since none of them holds a voxel with segments.
//
// Built after pass 1 in three separable passes: the L-infinity distance to a
// set factors over the axes, d(b) = min_k max(|k|, d_xy(b + k e_z)), and
// likewise for d_xy from d_x and d_x from the occupancy.
#include "launch.h"

namespace vrt {

// The occupancy mask of each brick, and 0 when any of its 64 voxels has a count,
// else the cap. A thread reads one x-row of a brick (16 bytes, so a warp reads
// 512 contiguous bytes) and the brick's 16 threads combine their four bits.
__global__ void __launch_bounds__(256) k_brick_occ(GridDev g, uint8_t* __restrict__ out,
                                                   uint2* __restrict__ mask) {
  const uint32_t row = blockIdx.x * blockDim.x + threadIdx.x + dependency_wait();
  const int lane = threadIdx.x & 31;
  const uint4 v = __ldg(reinterpret_cast<const uint4*>(g.word) + row);  // n^3 / 4 rows: whole blocks
  const uint32_t m = ((v.x & 0xffffu) ? 1u : 0u) | ((v.y & 0xffffu) ? 2u : 0u) |
                     ((v.z & 0xffffu) ? 4u : 0u) | ((v.w & 0xffffu) ? 8u : 0u);
  uint32_t half = m << (4 * (lane & 7));  // rows 0-7 and 8-15 of a brick: 32 bits each
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) half |= __shfl_xor_sync(0xffffffffu, half, o);
  const uint32_t hi = __shfl_down_sync(0xffffffffu, half, 8);
  if ((lane & 15) == 0) {
    const uint32_t b = row >> 4;
    mask[b] = make_uint2(half, hi);
    out[b] = (half | hi) ? 0 : (uint8_t)kBrickDistMax;
  }
}

// out(b) = min over |i| <= kBrickDistMax (inside the grid) of max(|i|, in(b + i e)),
// along axis `axis` (0 x, 1 y, 2 z).
__global__ void __launch_bounds__(256) k_brick_dist(int log2nb, int axis,
                                                    const uint8_t* __restrict__ in,
                                                    uint8_t* __restrict__ out) {
  const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x + dependency_wait();
  const uint32_t nb = 1u << (3 * log2nb);
  if (b >= nb) return;
  const int side = 1 << log2nb;
  const int shift = axis * log2nb;
  const int c = (int)((b >> shift) & (uint32_t)(side - 1));
  const uint32_t base = b - ((uint32_t)c << shift);
  int d = __ldg(&in[b]);
  for (int i = 1; i < d; ++i) {
    if (c - i >= 0) d = min(d, max(i, (int)__ldg(&in[base + ((uint32_t)(c - i) << shift)])));
    if (c + i < side) d = min(d, max(i, (int)__ldg(&in[base + ((uint32_t)(c + i) << shift)])));
  }
  out[b] = (uint8_t)d;
}

__global__ void __launch_bounds__(256) k_reset(uint32_t* a, uint32_t na, uint32_t* b, uint32_t nb) {
  dependency_wait();
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < na + nb; i += gridDim.x * blockDim.x)
    if (i < na) a[i] = 0u;
    else b[i - na] = 0u;
}

int launch_reset(uint32_t* a, uint32_t na, uint32_t* b, uint32_t nb, const Queue& q) {
  const unsigned blocks = (na + nb + 1023) / 1024;
  launch(k_reset, blocks < kSms ? blocks : kSms, 256, q, a, na, b, nb);
  return 1;
}

int launch_brick_dist_passes(int log2nb, uint8_t* tmp, uint8_t* dist, const Queue& q) {
  const uint32_t nb = 1u << (3 * log2nb);
  const int T = 256;
  const unsigned blocks = (nb + T - 1) / T;
  launch(k_brick_dist, blocks, T, q, log2nb, 0, tmp, dist);
  launch(k_brick_dist, blocks, T, q, log2nb, 1, dist, tmp);
  launch(k_brick_dist, blocks, T, q, log2nb, 2, tmp, dist);
  return 3;
}

int launch_brick_dist(const GridDev& g, uint8_t* tmp, uint8_t* dist, uint2* mask, const Queue& q) {
  const int T = 256;
  launch(k_brick_occ, (1u << (3 * g.log2nb + 4)) / T, T, q, g, tmp, mask);
  return 1 + launch_brick_dist_passes(g.log2nb, tmp, dist, q);
}

}  // namespace vrt
