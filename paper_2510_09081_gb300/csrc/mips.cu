// A2: the averaging occupancy pyramid used by cone-traced ambient occlusion
// (an averaging mipmap, Sec. 3.1; sampled by the cones of Sec. 3.4). Level 0 is
// min(1, occupancy code sum / occ_scale) per voxel, level l+1 the mean of the
// 8 children; each level is stored x-fastest (canonical) so the trace's
// trilinear samples are plain strided loads. Texels are fp32, fp16 or bf16.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "launch.h"

namespace vrt {

// Storage of a texel: fp32, or fp16 / bf16 rounded to nearest from the fp32 value
// (each level is averaged in fp32 from its stored children, then rounded once).
__device__ __forceinline__ void store_texel(float* p, float v) { *p = v; }
__device__ __forceinline__ void store_texel(__half* p, float v) { *p = __float2half_rn(v); }
__device__ __forceinline__ void store_texel(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ float load_texel(const float* p) { return *p; }
__device__ __forceinline__ float load_texel(const __half* p) { return __half2float(*p); }
__device__ __forceinline__ float load_texel(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// Level 0 and 1 together. Bound by memory (n^3 words in, n^3 and n^3 / 8 texels
// out), so the split is the one that moves whole lines: four lanes take a brick, a
// 4x2x2 part each, so a warp reads 8 bricks (2 KB in one run) by 16 bytes a load
// and writes rows of 32 level-0 and 16 level-1 texels. A level-1 texel is the mean
// of the 8 as stored (so that every level averages its stored children).
// 512^3 fp32 (1.14 GB), all levels: a thread to a level-1 texel, words and texels one
// by one, 0.309 ms; 0.188 so (0.168 at the copy rate).
template <class T, int N>
struct alignas(N * sizeof(T)) Texels {
  T v[N];
};

template <class T>
__global__ void __launch_bounds__(256) k_mip01(GridDev g, T* __restrict__ l0, T* __restrict__ l1) {
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x + dependency_wait();
  const uint32_t b = t >> 2, nb1 = (1u << g.log2nb) - 1u;
  if (b >> (3 * g.log2nb)) return;
  const uint32_t x = (b & nb1) << 2, y = (((b >> g.log2nb) & nb1) << 2) + 2 * (t & 1u),
                 z = ((b >> (2 * g.log2nb)) << 2) + (t & 2u);
  const uint4* src = reinterpret_cast<const uint4*>(g.word) + b * 16u + (t & 2u) * 4u + (t & 1u) * 2u;
  uint4 w[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) w[k] = __ldg(src + (k >> 1) * 4 + (k & 1));
  const float inv = 1.0f / g.occ_scale;
  const uint32_t n = g.n;
  float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint32_t c[4] = {w[k].x >> 16, w[k].y >> 16, w[k].z >> 16, w[k].w >> 16};
    Texels<T, 4> r;
#pragma unroll
    for (int i = 0; i < 4; ++i) store_texel(&r.v[i], fminf(1.0f, (float)c[i] * inv));
    s0 = (s0 + load_texel(&r.v[0])) + load_texel(&r.v[1]);
    s1 = (s1 + load_texel(&r.v[2])) + load_texel(&r.v[3]);
    *reinterpret_cast<Texels<T, 4>*>(&l0[((z + (k >> 1)) * n + y + (k & 1)) * n + x]) = r;
  }
  Texels<T, 2> r;
  store_texel(&r.v[0], s0 * 0.125f);
  store_texel(&r.v[1], s1 * 0.125f);
  const uint32_t m = n >> 1;
  *reinterpret_cast<Texels<T, 2>*>(&l1[((z >> 1) * m + (y >> 1)) * m + (x >> 1)]) = r;
}

template <class T>
__global__ void __launch_bounds__(256) k_mip_down(const T* __restrict__ src, T* __restrict__ dst, int m) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x + dependency_wait();
  if (t >= (long long)m * m * m) return;
  const int x = (int)(t % m), y = (int)((t / m) % m), z = (int)(t / ((long long)m * m));
  const int mp = 2 * m;
  float s = 0.0f;
#pragma unroll
  for (int dz = 0; dz < 2; ++dz)
#pragma unroll
    for (int dy = 0; dy < 2; ++dy) {
      const T* row = &src[((long long)(2 * z + dz) * mp + (2 * y + dy)) * mp + 2 * x];
      s += load_texel(row) + load_texel(row + 1);
    }
  store_texel(&dst[t], s * 0.125f);
}

template <class T>
int launch_mips_t(const GridDev& g, T* mips, const long long* lev_off, int n_levels, const Queue& q) {
  const int T_ = 256;
  long long m = g.n >> 1;
  long long cnt = m * m * m / 2;  // threads: 16 voxels each
  int launches = 1;
  launch(k_mip01<T>, (unsigned)((cnt + T_ - 1) / T_), T_, q, g, mips + lev_off[0], mips + lev_off[1]);
  for (int l = 2; l < n_levels; ++l) {
    m = g.n >> l;
    cnt = m * m * m;
    launch(k_mip_down<T>, (unsigned)((cnt + T_ - 1) / T_), T_, q, mips + lev_off[l - 1],
                   mips + lev_off[l], (int)m);
    ++launches;
  }
  return launches;
}

int launch_mips(const GridDev& g, void* mips, int fmt, const long long* lev_off, int n_levels,
                const Queue& q) {
  if (fmt == kMipsF16) return launch_mips_t(g, (__half*)mips, lev_off, n_levels, q);
  if (fmt == kMipsBF16) return launch_mips_t(g, (__nv_bfloat16*)mips, lev_off, n_levels, q);
  return launch_mips_t(g, (float*)mips, lev_off, n_levels, q);
}

}  // namespace vrt
