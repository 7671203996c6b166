// A6: voxel ray tracing (Sec. 3.5).
//
// One ray per pixel; a warp owns a tile of pixels, 4 wide and 8 tall (in the
// repair re-trace, its share of the queued pixels). Each lane walks its own ray by
// 3D-DDA (Amanatides & Woo), a 4^3 brick per round, until it reaches an occupied
// voxel; in a brick with no occupied voxel it crosses, in one step, the whole cube
// of empty bricks that the distance field built after pass 1 guarantees around
// it. The warp then numbers the entries of its lanes' pending lists one after
// another and takes them 64 at a time, so no lane idles on another lane's longer
// list; rays waiting in the same voxel share an entry's loads. A list longer than
// kShortList, or a voxel in which one ray has more hits than the warp's
// shared-memory slots hold, goes to a whole-warp path that processes one voxel
// at a time (lane l takes entries l, l+32, ...).
//
// Bound by instruction issue and latency, not memory: 20 warps an SM, 1.3 G warp
// instructions at 53% of the issue slots for 147M (ray, entry) pairs. Against a
// trace that kept all of a ray's state in registers (128, 16 warps an SM),
// stepped voxel by voxel on three loads a step, and took a pair a lane: sparse
// walks at 4K 31.0 -> 21.4 ms, 157x93 pixels at alpha 0.1 0.70 -> 0.22 ms, 10M-segment
// bundles at 1080p 3.25 -> 2.80 ms, opaque ABC at 1080p 0.57 -> 0.41 ms.
//
// For each listed segment the lane computes the first entry of the ray into
// the segment's capsule; an entry counts only if it lies in the voxel's ray
// interval [t_enter, t_exit) -- the intervals partition the ray, so each hit
// is counted once and hits come out voxel by voxel in depth order -- and both
// clip planes keep it. A cheap line-to-line distance test skips segments whose
// line passes farther than r from the ray.
//  - opaque: the minimum 64-bit key (depth bits << 32 | segment id) is the
//    voxel's nearest hit; the ray stops at the first voxel that has one.
//  - transparent, shared entries: the hits of the warp's rays are collected in
//    shared memory, ranked by key and composited by each ray's lane.
//  - transparent, whole-warp path: each lane keeps its 4 smallest keys beyond the last
//    composited one; the warp extracts keys in global (depth, id) order by
//    repeated minimum reductions -- only up to the smallest key a lane had to
//    drop, beyond which it rescans the list -- shades up to 32 of them in
//    parallel (one per lane), and accumulates them in key order,
//    C += T alpha c, T *= 1 - alpha, until T < 1e-4 (ground-truth order).
// Shading: colour = |unit tangent| per component times either cone-traced
// ambient occlusion per hit when enabled (six cones over the occupancy
// pyramid; the hits of an opaque trace are shaded by a kernel of their own at
// the end), or one trilinear sample of the voxel-space shading field at the hit
// (Sec. 3.4, built by shade.cu).
//
// Culling validation: a ray that reaches a voxel holding segments but no list
// queues the voxel (deduplicated by a bitmap), marches on as if the voxel were
// empty -- until it has queued max_queue voxels -- and finally queues its pixel
// instead of writing it; the repair round lists the queued voxels and traces
// the pixel again, so the image never depends on the culling heuristic. With
// no limit, the march queues every culled voxel before the point where it
// ends; the voxels' hits could only end the ray sooner, so the next trace
// of that pixel needs nothing more.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cmath>

#include "launch.h"
#include "pyramid.cuh"

namespace vrt {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kLaneKeys = 4;              // transparent, shared list: keys kept per lane per scan
// Transparent: hits of a round that a warp's rays share (slots are bytes), and the
// (ray, entry) pairs a round takes rays for. About 7% of the pairs of dense sets
// give hits; 128 and 768 send more rays back for another pass (bundles at
// 1080p 2.92 ms against 2.86), and a larger pool takes L1 from the lists.
constexpr uint32_t kPool = 192;
constexpr uint32_t kRoundPairs = 1536;
constexpr uint32_t kLost = 1u << 31;  // WarpMem::cnt: a hit of the ray found the pool full
// Ray::calls: the culled voxels the ray queued (bits 0-10, at most 3 n); its hits
// in the pending voxel, once counted (11-18); its walk calls (19-31). Past
// TraceArgs::max_calls, more than any walk takes, a ray is given up and vrt_sync
// reports the timeout, so that no loop of the trace can run for ever whatever the
// data. (With a register of its own for the rounds of a warp sparse walks at 4K took
// 2.6% longer, so 0.8%.)
constexpr uint32_t kQueued = 2047u, kHits = 255u << 11, kCall = 1u << 19;
// Rays that share an entry's loads. Lists are short (4 entries on average for
// sparse walks, 24 for the bundles), so larger groups leave lanes without an
// entry: groups of 32 take 0.55 ms where 4 take 0.43 on the opaque 1080p ABC
// view, and 3.37 against 3.30 on the bundles; single rays 0.46 and 3.73.
constexpr int kGroup = 4;

// Instrumented trace: mark element i of a touch bitmap.
__device__ __forceinline__ void touch(uint32_t* bits, uint32_t i) {
  if (bits) atomicOr(&bits[i >> 5], 1u << (i & 31));
}

__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(FULL, v, o);
    v = w < v ? w : v;
  }
  return v;
}

__device__ __forceinline__ float3 shfl3(float3 v, int src) {
  return make_float3(__shfl_sync(FULL, v.x, src), __shfl_sync(FULL, v.y, src),
                     __shfl_sync(FULL, v.z, src));
}

// The voxel-space shading field at P: trilinear over voxel centres, texel
// coordinates clamped to the grid. A hit accepted in voxel v reads only v and
// its neighbours, all of which the shading pass computed.
__device__ __forceinline__ float shade_at(const TraceArgs& A, float3 P) {
  const int n1 = A.g.n - 1;
  const float ux = P.x - 0.5f, uy = P.y - 0.5f, uz = P.z - 0.5f;
  const float fx0 = floorf(ux), fy0 = floorf(uy), fz0 = floorf(uz);
  const int x = (int)fx0, y = (int)fy0, z = (int)fz0;
  const float fx = ux - fx0, fy = uy - fy0, fz = uz - fz0;
  float acc = 0.0f;
#pragma unroll
  for (int dz = 0; dz < 2; ++dz)
#pragma unroll
    for (int dy = 0; dy < 2; ++dy)
#pragma unroll
      for (int dx = 0; dx < 2; ++dx) {
        const float w = (dx ? fx : 1.0f - fx) * (dy ? fy : 1.0f - fy) * (dz ? fz : 1.0f - fz);
        const int xi = min(max(x + dx, 0), n1), yi = min(max(y + dy, 0), n1), zi = min(max(z + dz, 0), n1);
        acc = fmaf(w, __ldg(&A.shade[brick_index(xi, yi, zi, A.g.log2nb)]), acc);
      }
  return acc;
}

// Shading factor of a transparent hit at P. The trace kernels are instantiated
// with AO for cone AO per hit and without it for no shading or the voxel-space
// field: a call to the AO code anywhere in a kernel costs all its rays
// registers (bundles at alpha 0.3 without AO 1% slower, small random walks 3%).
__device__ __noinline__ float field_shade(const TraceArgs& A, float3 P) { return shade_at(A, P); }
template <bool AO>
__device__ __forceinline__ float hit_shade(const TraceArgs& A, float3 P) {
  if constexpr (AO) return ao_lane(A, P);
  else return field_shade(A, P);
}

__device__ __forceinline__ float3 tangent_colour(float3 a, float3 b) {
  const float3 dv = b - a;
  const float l2 = dot3(dv, dv);
  if (!(l2 > 0.0f)) return make_float3(1.0f, 1.0f, 1.0f);
  const float il = rsqrt_normal(l2);
  return make_float3(fabsf(dv.x) * il, fabsf(dv.y) * il, fabsf(dv.z) * il);
}

// Sort key of an accepted hit at depth t of segment id, entry li of the voxel's
// list, the voxel's ray interval being [t0, t1). Default: the depth's fp32 bits
// above the id (depth order, ties by id). With A.key16 the paper's per-voxel
// key (Sec. 3.5): the depth within the voxel quantized to 16 bits above the
// 16-bit list index -- hits of equal quantized depth then follow the list's
// order -- with the id below it, for shading.
template <bool KEY16>
__device__ __forceinline__ unsigned long long hit_key(float t, uint32_t id, uint32_t li, float t0,
                                                      float t1) {
  if (!KEY16) return ((unsigned long long)__float_as_uint(t) << 32) | id;
  const float u = __fdividef(t - t0, t1 - t0);
  const uint32_t q = min(65535u, (uint32_t)fmaxf(0.0f, u * 65536.0f));
  return ((unsigned long long)((q << 16) | (li & 0xffffu)) << 32) | id;
}

// Depth of the hit a key names: stored in the default key; recomputed from the
// segment with the 16+16 key, which keeps only its quantized position.
template <bool KEY16>
__device__ __forceinline__ float hit_depth(const TraceArgs& A, unsigned long long k, float3 o,
                                           float3 d) {
  if (!KEY16) return __uint_as_float((uint32_t)(k >> 32));
  const uint32_t id = (uint32_t)(k & 0xffffffffu);
  const float4 p0 = __ldg(&A.pos[id]), p1 = __ldg(&A.pos[id + 1]);
  return capsule_entry(o, d, f3(p0), f3(p1), A.g.r * A.g.r);
}

__device__ __forceinline__ bool clip_keeps(const TraceArgs& A, float3 P, float4 p0, float4 p1,
                                           uint32_t id) {
  if (__float_as_uint(p0.w) & kClipOn) {
    const float3 n0 = f3(__ldg(&A.nrm[id]));
    if (dot3(P - f3(p0), n0) < 0.0f) return false;
  }
  if (__float_as_uint(p1.w) & kClipOn) {
    const float3 n1 = f3(__ldg(&A.nrm[id + 1]));
    if (dot3(P - f3(p1), n1) > 0.0f) return false;
  }
  return true;
}

// Key of list entry s for ray (o, d) over [t0, t1): depth bits << 32 | id, or
// ~0 when the segment gives no accepted hit there.
template <bool COUNT, bool KEY16>
__device__ __forceinline__ unsigned long long entry_key(const TraceArgs& A, uint32_t s, uint32_t beg,
                                                        float3 o, float3 d, float t0, float t1,
                                                        float r2, float rrm, unsigned& n_cap) {
  const uint32_t id = __ldg(&A.g.lists[s]);
  if (id + 1 >= A.n_vert) {
    set_err(A.g.st, kErrBounds);
    return ~0ull;
  }
  if (COUNT) {
    touch(A.touch_list, s);
    touch(A.touch_vert, id);
    touch(A.touch_vert, id + 1);
  }
  const float4 p0 = __ldg(&A.pos[id]), p1 = __ldg(&A.pos[id + 1]);
  if (!lines_may_meet(o, d, f3(p0), f3(p1), rrm)) return ~0ull;
  if (COUNT) ++n_cap;
  const float t = capsule_entry(o, d, f3(p0), f3(p1), r2);
  if (!(t >= t0 && t < t1)) return ~0ull;
  if (!clip_keeps(A, o + t * d, p0, p1, id)) return ~0ull;
  return hit_key<KEY16>(t, id, s - beg, t0, t1);
}

// One warp's shared memory. Per ray: what the line and capsule tests of other
// lanes read (origin and entry parameter, direction and exit parameter) and what
// its own lane needs only between tests (reciprocal direction, colour, first
// hit), which keeps the registers of a lane to the walk's or the test's working
// set. Transparent hits of a round go to a pool that the warp's rays share;
// opaque rays keep their nearest key.
template <bool OPAQUE, bool KEY16>
struct WarpMem {
  float4 o[32];     // origin, entry parameter of the pending voxel
  float4 d[32];     // direction, exit parameter
  float4 inv[32];   // 1 / direction per axis (0 where it is 0); first hit's id as bits
  float4 acc[32];   // colour so far; first hit's depth
  uint32_t uid[128];             // segment ids of the units of this step and the last
  uint16_t uli[KEY16 ? 128 : 2]; // their list indices (16+16 keys)
  uint16_t q[32 + 64 * kGroup];  // pairs queued for the capsule test: unit | ray << 8
  unsigned long long key[OPAQUE ? 32 : kPool];  // opaque: the ray's nearest key
  float col[OPAQUE ? 1 : 3][OPAQUE ? 1 : kPool];
  uint16_t own[OPAQUE ? 2 : kPool];    // the hit's ray | its number among the ray's hits << 8
  uint8_t slot[OPAQUE ? 4 : kPool];    // pool slots, ray after ray
  uint8_t order[OPAQUE ? 4 : kPool];   // the same, each ray's by key
  uint32_t cnt[OPAQUE ? 1 : 32];       // hits of each ray in the round
};

// Registers a lane keeps for its ray. Voxel coordinates are packed, four added
// to each (so that the fields stay positive one step outside the grid):
// (x + 4) | (y + 4) << 10 | (z + 4) << 20.
struct Ray {
  uint32_t p;
  uint2 mask;          // the current brick's occupied voxels
  int kd;              // and its distance to an occupied brick
  float tcur, t1, T;
  uint32_t pix, vox;   // pixel; pending voxel's word index
  uint32_t beg, len;   // pending voxel's list
  uint32_t calls;      // walk calls, hits in the pending voxel, culled voxels queued
  bool active, pending, missed;
};

// Work counters of a lane (instrumented trace).
struct Work {
  unsigned steps = 0, entries = 0, cap = 0, vox = 0, hits = 0, ww_vox = 0, ww_ent = 0;
  // warp cycles: DDA, shared-entry path, whole-warp path, capsule stage
  unsigned long long cyc[4] = {0, 0, 0, 0};
};

__device__ __forceinline__ uint32_t pack_pos(int x, int y, int z) {
  return (uint32_t)(x + 4) | ((uint32_t)(y + 4) << 10) | ((uint32_t)(z + 4) << 20);
}
__device__ __forceinline__ void unpack_pos(uint32_t p, int& x, int& y, int& z) {
  x = (int)(p & 1023u) - 4;
  y = (int)((p >> 10) & 1023u) - 4;
  z = (int)(p >> 20) - 4;
}
constexpr uint32_t kLocalBits = 0x00300c03u;  // the coordinates within a 4^3 brick

// Parameter where the ray leaves coordinate `b` along an axis it moves on;
// +inf when it does not move on that axis.
__device__ __forceinline__ float cross_t(float inv, float b, float ooi) {
  return inv != 0.0f ? fmaf(b, inv, -ooi) : __int_as_float(0x7f800000);
}

__device__ __forceinline__ uint32_t brick_of(const TraceArgs& A, int x, int y, int z) {
  return ((uint32_t)(z >> 2) << (2 * A.g.log2nb)) | ((uint32_t)(y >> 2) << A.g.log2nb) | (uint32_t)(x >> 2);
}

// Read the mask and empty distance of the brick the ray is in (R.p in the grid).
__device__ __forceinline__ void load_brick(const TraceArgs& A, Ray& R) {
  int x, y, z;
  unpack_pos(R.p, x, y, z);
  const uint32_t b = brick_of(A, x, y, z);
  R.mask = __ldg(&A.g.bmask[b]);
  R.kd = __ldg(&A.g.bdist[b]);
}

// Walk the lane's ray through the brick it is in: 1 when it reached an occupied
// voxel (then pending in R.vox over [o.w, d.w)), 0 when it leaves the grid, -1
// when it goes on in the next brick. In a brick without occupied voxels the ray
// crosses the whole cube of empty bricks around it. Every call moves the ray
// forward through the grid, so its walk ends.
//
// Bound by the latency of its loads: a call reads the brick's 64-bit occupancy
// mask and its empty distance, once, and steps from voxel to voxel on the mask
// in registers; the voxel's word and list end are read only for an occupied
// voxel, in the round that processes it. Reading the distance, word and list
// end at every voxel step kept a 4K trace of sparse walks in 512^3 (133 steps and
// 16 occupied voxels per ray, words far larger than L2) waiting on three loads
// per step.
template <class M, bool COUNT>
__device__ __forceinline__ int walk_brick(const TraceArgs& A, M& S, Ray& R, Work& W) {
  const int lane = threadIdx.x & 31;
  const int n = A.g.n;
  if (R.tcur > R.t1) return 0;
  int x, y, z;
  unpack_pos(R.p, x, y, z);
  const float4 inv = S.inv[lane], o = S.o[lane];
  const float3 ooi = make_float3(o.x * inv.x, o.y * inv.y, o.z * inv.z);
  if (R.kd > 0) {
    // cross the cube of empty bricks within kd - 1 of this one: low corner
    // (bx, by, bz), side w voxels
    if (COUNT) ++W.steps;
    const float4 d = S.d[lane];
    const int ext = 4 * (R.kd - 1), w = 4 + 2 * ext;
    const int bx = (x & ~3) - ext, by = (y & ~3) - ext, bz = (z & ~3) - ext;
    const float tx = cross_t(inv.x, (float)(inv.x > 0.0f ? bx + w : bx), ooi.x);
    const float ty = cross_t(inv.y, (float)(inv.y > 0.0f ? by + w : by), ooi.y);
    const float tz = cross_t(inv.z, (float)(inv.z > 0.0f ? bz + w : bz), ooi.z);
    const float tb = fminf(tx, fminf(ty, tz));
    if (tb > R.t1) return 0;
    const int cx = min(min(bx + w, n) - 1, max(max(bx, 0), (int)floorf(fmaf(tb, d.x, o.x))));
    const int cy = min(min(by + w, n) - 1, max(max(by, 0), (int)floorf(fmaf(tb, d.y, o.y))));
    const int cz = min(min(bz + w, n) - 1, max(max(bz, 0), (int)floorf(fmaf(tb, d.z, o.z))));
    if (tb == tx) {
      x = inv.x > 0.0f ? bx + w : bx - 1; y = cy; z = cz;
      if ((unsigned)x >= (unsigned)n) return 0;
    } else if (tb == ty) {
      y = inv.y > 0.0f ? by + w : by - 1; x = cx; z = cz;
      if ((unsigned)y >= (unsigned)n) return 0;
    } else {
      z = inv.z > 0.0f ? bz + w : bz - 1; x = cx; y = cy;
      if ((unsigned)z >= (unsigned)n) return 0;
    }
    R.p = pack_pos(x, y, z);
    R.tcur = fmaxf(R.tcur, tb);
    load_brick(A, R);
    return -1;
  }
  const float sx = inv.x > 0.0f ? 1.0f : -1.0f, sy = inv.y > 0.0f ? 1.0f : -1.0f,
              sz = inv.z > 0.0f ? 1.0f : -1.0f;
  float bx = (float)(inv.x > 0.0f ? x + 1 : x), by = (float)(inv.y > 0.0f ? y + 1 : y),
        bz = (float)(inv.z > 0.0f ? z + 1 : z);
  const uint32_t px = inv.x > 0.0f ? 1u : 0u - 1u, py = inv.y > 0.0f ? 1u << 10 : 0u - (1u << 10),
                 pz = inv.z > 0.0f ? 1u << 20 : 0u - (1u << 20);
  float tx = cross_t(inv.x, bx, ooi.x), ty = cross_t(inv.y, by, ooi.y), tz = cross_t(inv.z, bz, ooi.z);
  const uint32_t p0 = R.p;
  uint32_t p = p0;
  float tin = R.tcur;
  bool hit, left;
  uint32_t loc;
  float te;
  // at most 10 steps: each leaves one of the brick's 3 x 4 planes of voxels behind
  for (;;) {
    if (COUNT) ++W.steps;
    // x + 4 y + 16 z of the coordinates within the brick: three shifted copies
    // of the packed fields meet in bits 20-25
    loc = ((p & kLocalBits) * ((1u << 20) | (1u << 12) | (1u << 4)) >> 20) & 63u;
    hit = (((loc & 32u) ? R.mask.y : R.mask.x) >> (loc & 31u)) & 1u;
    te = fminf(tx, fminf(ty, tz));
    if (te == tx) {
      p += px;
      bx += sx;
      tx = fmaf(bx, inv.x, -ooi.x);
    } else if (te == ty) {
      p += py;
      by += sy;
      ty = fmaf(by, inv.y, -ooi.y);
    } else {
      p += pz;
      bz += sz;
      tz = fmaf(bz, inv.z, -ooi.z);
    }
    left = ((p ^ p0) & ~kLocalBits) != 0u;
    if (hit || left || te > R.t1) break;
    tin = te;
  }
  // the ray is past this voxel: the next call resumes after it
  R.p = p;
  R.tcur = te;
  if (hit) R.vox = (brick_of(A, x, y, z) << 6) | loc;
  bool inside = true;
  if (left) {
    unpack_pos(p, x, y, z);
    inside = (unsigned)x < (unsigned)n && (unsigned)y < (unsigned)n && (unsigned)z < (unsigned)n;
    // its load completes while the warp's other work goes on
    if (inside) load_brick(A, R);
  }
  if (hit) {
    S.o[lane].w = tin;
    S.d[lane].w = te;
    if (!inside) R.t1 = -1.0f;  // this was the last voxel; stop after it
    return 1;
  }
  return inside ? -1 : 0;
}

// Origin and unit direction of pixel (px, py)'s ray.
__device__ __forceinline__ void pixel_ray(const CamDev& c, int px, int py, float3& o, float3& d) {
  const float fx = (float)px + 0.5f, fy = (float)py + 0.5f;
  if (c.ortho) {
    o = c.o0 + fx * c.ox + fy * c.oy;
    d = c.d0;
  } else {
    o = c.o0;
    const float3 v = c.d0 + fx * c.dx + fy * c.dy;
    d = (1.0f / sqrtf(dot3(v, v))) * v;
  }
}

template <class M>
__device__ void init_ray(const TraceArgs& A, M& S, Ray& R, int px, int py, bool valid) {
  const int lane = threadIdx.x & 31;
  float3 ro, rd, ri;
  pixel_ray(A.cam, px, py, ro, rd);
  R.T = 1.0f;
  R.calls = 0;
  R.missed = false;
  R.pending = false;
  R.vox = R.beg = R.len = 0;
  R.pix = valid ? (uint32_t)(py * A.cam.width + px) : 0u;
  const float N = (float)A.g.n;
  float t0 = 0.0f, t1 = __int_as_float(0x7f800000);
  bool miss = !valid;
  auto axis = [&](float o, float d, float& inv) {
    if (d != 0.0f) {
      inv = 1.0f / d;
      float ta = (0.0f - o) * inv, tb = (N - o) * inv;
      if (ta > tb) { const float q = ta; ta = tb; tb = q; }
      t0 = fmaxf(t0, ta);
      t1 = fminf(t1, tb);
    } else {
      inv = 0.0f;
      if (o < 0.0f || o > N) miss = true;
    }
  };
  axis(ro.x, rd.x, ri.x);
  axis(ro.y, rd.y, ri.y);
  axis(ro.z, rd.z, ri.z);
  R.active = !miss && t0 <= t1;
  R.tcur = t0;
  R.t1 = t1;
  const int n = A.g.n;
  R.p = pack_pos(min(n - 1, max(0, (int)floorf(fmaf(t0, rd.x, ro.x)))),
                 min(n - 1, max(0, (int)floorf(fmaf(t0, rd.y, ro.y)))),
                 min(n - 1, max(0, (int)floorf(fmaf(t0, rd.z, ro.z)))));
  load_brick(A, R);
  S.o[lane] = make_float4(ro.x, ro.y, ro.z, 0.0f);
  S.d[lane] = make_float4(rd.x, rd.y, rd.z, 0.0f);
  S.inv[lane] = make_float4(ri.x, ri.y, ri.z, __int_as_float(-1));
  S.acc[lane] = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(0x7f800000));
}

// A re-traced ray continues from the state it had when it first met a culled
// voxel (now listed): same colour, transmittance and first hit, at that voxel
// and its entry parameter, so the result equals a trace from the start.
template <class M>
__device__ void resume_ray(const TraceArgs& A, M& S, Ray& R) {
  const int lane = threadIdx.x & 31;
  const float4 s0 = A.resume[2 * R.pix], s1 = A.resume[2 * R.pix + 1];
  S.acc[lane] = make_float4(s0.x, s0.y, s0.z, s1.y);
  S.inv[lane].w = s1.x;
  R.T = s0.w;
  int x, y, z;
  brick_coords(__float_as_uint(s1.z), A.g.log2nb, x, y, z);
  R.p = pack_pos(min(A.g.n - 1, max(0, x)), min(A.g.n - 1, max(0, y)), min(A.g.n - 1, max(0, z)));
  R.tcur = s1.w;
  load_brick(A, R);
}

// Read the pending voxel's word and list end: its list into R.beg, R.len, or,
// when the cull gave it none, the voxel into the repair queue, the ray marching
// on as if it were empty.
template <class M, bool COUNT>
__device__ __forceinline__ void resolve_list(const TraceArgs& A, M& S, Ray& R) {
  const int lane = threadIdx.x & 31;
  const uint32_t idx = R.vox;
  const uint32_t cnt = __ldg(&A.g.word[idx]) & 0xffffu;
  const uint32_t end0 = __ldg(&A.g.cur[idx]);
  if (COUNT) touch(A.touch_vox, idx);
  if (end0 >= kCulledStart) {
    // at the first culled voxel, keep the ray's state for the re-trace to resume from
    if ((R.calls & kQueued) == 0 && A.resume) {
      const float4 c = S.acc[lane];
      A.resume[2 * R.pix] = make_float4(c.x, c.y, c.z, R.T);
      A.resume[2 * R.pix + 1] = make_float4(S.inv[lane].w, c.w, __uint_as_float(idx), S.o[lane].w);
    }
    const uint32_t bm = 1u << (idx & 31);
    const uint32_t old = atomicOr(&A.need[idx >> 5], bm);
    if (!(old & bm)) {
      const uint32_t q = atomicAdd(A.vq_cnt, 1u);
      if (q < A.vq_cap) A.vq[q] = idx;
      else set_err(A.g.st, kErrOverflow);
    }
    R.missed = true;
    R.pending = false;
    if ((++R.calls & kQueued) >= A.max_queue || R.t1 < 0.0f) R.active = false;
    return;
  }
  if (end0 < cnt) {
    set_err(A.g.st, kErrBounds);
    R.pending = R.active = false;
    return;
  }
  // a list past the capacity (reported as overflow) is read only up to it
  const uint32_t end = (unsigned long long)end0 > A.g.list_cap ? (uint32_t)A.g.list_cap : end0;
  R.beg = end0 - cnt < end ? end0 - cnt : end;
  R.len = end - R.beg;
}

// An opaque ray ends at its nearest hit. With cone AO its pixel carries the hit
// (segment id and depth, kHitTag) to k_shade_hits, which writes the colour; otherwise
// it is shaded here.
constexpr uint32_t kHitTag = 0x7fc0a05cu;  // a NaN: no colour holds it
template <class M>
__device__ __forceinline__ void opaque_hit(const TraceArgs& A, M& S, Ray& R, uint32_t id, float t) {
  const int lane = threadIdx.x & 31;
  float3 c;
  if (A.ao == 1) {
    c = make_float3(__uint_as_float(id), t, __uint_as_float(kHitTag));
  } else {
    c = tangent_colour(f3(__ldg(&A.pos[id])), f3(__ldg(&A.pos[id + 1])));
    if (A.ao) c = field_shade(A, f3(S.o[lane]) + t * f3(S.d[lane])) * c;
    c = make_float3(A.alpha * c.x, A.alpha * c.y, A.alpha * c.z);
  }
  S.acc[lane] = make_float4(c.x, c.y, c.z, t);
  S.inv[lane].w = __uint_as_float(id);
  R.T *= (1.0f - A.alpha);
  R.active = false;
}

// The whole warp on one list, [beg, end), for the ray of lane L: the nearest key
// of an opaque ray.
template <bool COUNT, bool KEY16>
__device__ __noinline__ unsigned long long voxel_nearest(const TraceArgs& A, WarpMem<true, KEY16>& S, int L,
                                                         uint32_t beg, uint32_t end, unsigned& n_cap,
                                                         unsigned& n_hit) {
  const float4 o = S.o[L], d = S.d[L];
  const float r2 = A.g.r * A.g.r;
  const float rrm = (A.g.r + 1e-3f) * (A.g.r + 1e-3f);
  unsigned long long best = ~0ull;
  for (uint32_t s = beg + (threadIdx.x & 31); s < end; s += 32) {
    const unsigned long long k =
        entry_key<COUNT, KEY16>(A, s, beg, f3(o), f3(d), o.w, d.w, r2, rrm, n_cap);
    if (COUNT && k != ~0ull) ++n_hit;
    best = k < best ? k : best;
  }
  return warp_min_u64(best);
}

// The whole warp on one list, [beg, end), for the transparent ray of lane L with
// transmittance T: composites the voxel's hits into the ray's colour and first
// hit and returns its transmittance.
template <bool COUNT, bool KEY16, bool AO>
__device__ __noinline__ float voxel_composite(const TraceArgs& A, WarpMem<false, KEY16>& S, int L,
                                              uint32_t beg, uint32_t end, float T, unsigned& n_cap,
                                              unsigned& n_hit, unsigned& n_scan) {
  const int lane = threadIdx.x & 31;
  const float4 o4 = S.o[L], d4 = S.d[L];
  const float3 o = f3(o4), d = f3(d4);
  const float t0 = o4.w, t1 = d4.w;
  const float r2 = A.g.r * A.g.r;
  const float rrm = (A.g.r + 1e-3f) * (A.g.r + 1e-3f);
  const float4 acc = S.acc[L];
  float C0 = acc.x, C1 = acc.y, C2 = acc.z, ft = acc.w;
  int fid = __float_as_int(S.inv[L].w);
  const float om = 1.0f - A.alpha;
  unsigned long long last = 0ull;  // keys <= last are composited
  bool rescan = true;
  // a scan composites at least one of the list's entries
  for (uint32_t scan = beg; rescan && T >= kTStop && scan <= end; ++scan) {
    unsigned long long buf[kLaneKeys];
#pragma unroll
    for (int q = 0; q < kLaneKeys; ++q) buf[q] = ~0ull;
    bool dropped = false;
    if (COUNT) n_scan += end - beg;
    for (uint32_t s = beg + lane; s < end; s += 32) {
      const unsigned long long k = entry_key<COUNT, KEY16>(A, s, beg, o, d, t0, t1, r2, rrm, n_cap);
      if (COUNT && k != ~0ull) ++n_hit;
      if (k == ~0ull || k <= last) continue;
      if (k < buf[kLaneKeys - 1]) {
        if (buf[kLaneKeys - 1] != ~0ull) dropped = true;
        buf[kLaneKeys - 1] = k;
#pragma unroll
        for (int q = kLaneKeys - 1; q > 0; --q) {
          const unsigned long long lo = buf[q - 1] < buf[q] ? buf[q - 1] : buf[q];
          const unsigned long long hi = buf[q - 1] < buf[q] ? buf[q] : buf[q - 1];
          buf[q - 1] = lo;
          buf[q] = hi;
        }
      } else {
        dropped = true;
      }
    }
    // keys up to `lim` are complete: a lane that dropped keys kept its smallest
    const unsigned long long lim = warp_min_u64(dropped ? buf[kLaneKeys - 1] : ~0ull);
    rescan = lim != ~0ull;
    bool more = true;
    while (more && T >= kTStop) {
      // extract up to 32 keys in order; lane q receives the q-th
      unsigned long long mine = ~0ull;
      int n_out = 0;
      for (; n_out < 32; ++n_out) {
        const unsigned long long m = warp_min_u64(buf[0]);
        if (m == ~0ull || m > lim) break;
        if (buf[0] == m) {
#pragma unroll
          for (int q = 0; q < kLaneKeys - 1; ++q) buf[q] = buf[q + 1];
          buf[kLaneKeys - 1] = ~0ull;
        }
        if (lane == n_out) mine = m;
      }
      more = n_out == 32;
      if (n_out == 0) break;
      // shade in parallel
      float3 c = make_float3(0.f, 0.f, 0.f);
      float tq = 0.0f;
      if (lane < n_out) {
        const uint32_t id = (uint32_t)(mine & 0xffffffffu);
        tq = hit_depth<KEY16>(A, mine, o, d);
        c = tangent_colour(f3(__ldg(&A.pos[id])), f3(__ldg(&A.pos[id + 1])));
        if (A.ao) c = hit_shade<AO>(A, o + tq * d) * c;
      }
      // accumulate in key order
      for (int q = 0; q < n_out; ++q) {
        const float3 cq = shfl3(c, q);
        const unsigned long long kq = __shfl_sync(FULL, mine, q);
        const float tqq = KEY16 ? __shfl_sync(FULL, tq, q) : 0.0f;
        if (T < kTStop) break;
        const float w = T * A.alpha;
        C0 = fmaf(w, cq.x, C0);
        C1 = fmaf(w, cq.y, C1);
        C2 = fmaf(w, cq.z, C2);
        T *= om;
        if (fid < 0) {
          fid = (int)(kq & 0xffffffffu);
          ft = KEY16 ? tqq : __uint_as_float((uint32_t)(kq >> 32));
        }
        last = kq;
      }
    }
    // a rescan is needed only when the extraction stopped at the drop limit
    rescan = rescan && T >= kTStop && last == lim;
  }
  __syncwarp();  // every lane has read the ray's state
  if (lane == L) {
    S.acc[L] = make_float4(C0, C1, C2, ft);
    S.inv[L].w = __int_as_float(fid);
  }
  return T;
}

// The pending voxels of the warp's lanes with lists up to A.short_list
// entries, processed together. Lanes whose rays wait in the same voxel form
// groups of up to kGroup; a unit of work is one entry for one group. The units of
// all groups are numbered one after another and the warp takes 64 at a time, two
// per lane, so short lists do not wait for the longest one. A lane loads its
// units' entries (segment id and end points) and line-tests them against the rays
// of their groups; only the pairs that pass are compacted into the warp's queue,
// which gets the capsule test 32 at a time. A hit is shaded by the lane that
// found it. An opaque ray keeps its nearest key; a transparent ray's hits go to
// the warp's pool, where they are ranked by key for the ray's own lane to
// composite. Rays join a round only while their lists sum to kRoundPairs pairs. A
// ray with a hit that found the pool full keeps the number of its hits, and the
// next rounds take such rays only, as many as the pool holds the hits of: so each
// takes its voxel once more. `wait` is set for lanes whose voxel a later round takes; a
// lane left pending without it (a list past A.short_list, more hits than the pool or
// A.ray_keys) goes to the whole-warp path, which starts its voxel again from
// scratch.
//
// Where many rays have many hits in one voxel, what a full pool costs decides: 40,
// 200, 1500 and 3000 tubes through one column of voxels, and 3000 at one place,
// 640x480 pixels, alpha 0.3, took 0.31, 2.3, 24, 65 and 1329 ms with the voxel taken in
// parts of its interval whenever the pool was full; 0.20, 0.66, 3.4, 4.6 and 5.5 so.
template <bool OPAQUE, bool COUNT, bool KEY16, bool AO>
__device__ __forceinline__ void process_flat(const TraceArgs& A, WarpMem<OPAQUE, KEY16>& S, Ray& R, Work& W,
                                             bool& wait) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  bool take = R.pending && R.len <= A.short_list;
  wait = false;
  if (!OPAQUE) {
    const bool again = __any_sync(FULL, (R.calls & kHits) != 0u);
    const uint32_t need = !take ? 0u : (again ? (R.calls & kHits) >> 11 : R.len);
    const uint32_t room = again ? kPool : kRoundPairs;
    if (again || __reduce_add_sync(FULL, need) > room) {
      uint32_t sum = need;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(FULL, sum, o);
        if (lane >= o) sum += v;
      }
      // a later round's: rays whose hits are not counted yet while others' are, and
      // those past the room (the pool must hold all hits; the pairs may exceed theirs)
      wait = take && (again ? need == 0u || sum > room : sum - need >= room);
      take = take && !wait;
    }
  }
  // Lanes waiting in the same voxel (same list start) form groups of at most
  // kGroup; a group's lowest lane numbers the list's entries for it.
  const unsigned tm = __ballot_sync(FULL, take);
  const unsigned same = __match_any_sync(FULL, take ? R.beg : 0xffffffffu) & (take ? tm : 0u);
  const bool leads = take && __popc(same & lt) % kGroup == 0;
  unsigned gm = same & ~lt;  // from a leader on: its group's lanes
  {
    unsigned rest = gm;
#pragma unroll
    for (int q = 0; q < kGroup; ++q) rest &= rest - 1;
    gm ^= rest;
  }
  const uint32_t glen = leads ? R.len : 0u;
  uint32_t incl = glen;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += v;
  }
  const uint32_t total = __shfl_sync(FULL, incl, 31);
  if (OPAQUE) S.key[lane] = ~0ull;
  else S.cnt[lane] = 0u;
  __syncwarp();
  const uint32_t first = R.beg - (incl - glen);  // entry g of a group's list is lists[first + g]
  const float r2 = A.g.r * A.g.r;
  const float rrm = (A.g.r + 1e-3f) * (A.g.r + 1e-3f);
  uint32_t qn = 0, pn = 0;  // queued pairs, hits of the round (warp-uniform)
  // capsule test of queued pair q0 + lane for lanes below cnt
  auto capsule_stage = [&](uint32_t q0, uint32_t cnt) {
    const long long c0 = COUNT ? clock64() : 0;
    bool hit = false;
    unsigned long long k = 0;
    float3 c = make_float3(0.0f, 0.0f, 0.0f);
    int j = 0;
    if ((uint32_t)lane < cnt) {
      const uint32_t it = S.q[q0 + lane];
      const uint32_t id = S.uid[it & 127u];
      j = (int)(it >> 8);
      const float4 p0 = __ldg(&A.pos[id]), p1 = __ldg(&A.pos[id + 1]);
      const float4 ro = S.o[j], rd = S.d[j];
      if (COUNT) ++W.cap;
      const float t = capsule_entry(f3(ro), f3(rd), f3(p0), f3(p1), r2);
      if (t >= ro.w && t < rd.w && clip_keeps(A, f3(ro) + t * f3(rd), p0, p1, id)) {
        hit = true;
        k = hit_key<KEY16>(t, id, KEY16 ? S.uli[it & 127u] : 0u, ro.w, rd.w);
        if (COUNT) ++W.hits;
        if (!OPAQUE) {
          c = tangent_colour(f3(p0), f3(p1));
          if (A.ao) c = hit_shade<AO>(A, f3(ro) + t * f3(rd)) * c;
        }
      }
    }
    if (OPAQUE) {
      if (hit) atomicMin(&S.key[j], k);
    } else {
      const unsigned hm = __ballot_sync(FULL, hit);
      if (hit) {
        const uint32_t slot = pn + __popc(hm & lt);
        const uint32_t nth = atomicAdd(&S.cnt[j], 1u);
        if (slot < kPool) {
          S.key[slot] = k;
          S.col[0][slot] = c.x;
          S.col[1][slot] = c.y;
          S.col[2][slot] = c.z;
          S.own[slot] = (uint16_t)((uint32_t)j | (nth << 8));
        } else {
          atomicOr(&S.cnt[j], kLost);
        }
      }
      pn += __popc(hm);
    }
    if (COUNT) W.cyc[3] += (unsigned long long)(clock64() - c0);
  };
  // a unit of work: one entry and the rays of its group
  struct Unit {
    uint32_t s, id, li;
    unsigned m;
    float4 p0, p1;
  };
  auto find_unit = [&](uint32_t gq, Unit& u) {
    u.m = u.id = u.li = u.s = 0;
    if (__all_sync(FULL, gq >= total)) return;
    int j = 0;  // the leader that numbers unit gq
#pragma unroll
    for (int st = 16; st > 0; st >>= 1)
      if (__shfl_sync(FULL, incl, j + st - 1) <= gq) j += st;
    j = min(j, 31);
    u.s = __shfl_sync(FULL, first, j) + gq;
    u.m = __shfl_sync(FULL, gm, j);
    if (KEY16) u.li = u.s - __shfl_sync(FULL, R.beg, j);
    if (gq < total) u.id = __ldg(&A.g.lists[u.s]);
    else u.m = 0;
  };
  auto load_unit = [&](Unit& u) {
    if (u.m && u.id + 1 >= A.n_vert) {
      set_err(A.g.st, kErrBounds);
      u.m = 0;
    }
    u.p0 = u.p1 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (u.m) {
      u.p0 = __ldg(&A.pos[u.id]);
      u.p1 = __ldg(&A.pos[u.id + 1]);
      if (COUNT) { touch(A.touch_list, u.s); touch(A.touch_vert, u.id); touch(A.touch_vert, u.id + 1); }
    }
  };
  // line-tests the unit's entry against its rays; the rays that pass
  auto line_tests = [&](const Unit& u) {
    unsigned m = u.m, pm = 0;
    while (m) {  // two rays at a time: independent chains
      const int j0 = __ffs(m) - 1;
      m &= m - 1;
      const int j1 = m ? __ffs(m) - 1 : j0;
      m &= m - 1;
      const float4 o0 = S.o[j0], d0 = S.d[j0], o1 = S.o[j1], d1 = S.d[j1];
      const bool m0 = lines_may_meet(f3(o0), f3(d0), f3(u.p0), f3(u.p1), rrm);
      const bool m1 = lines_may_meet(f3(o1), f3(d1), f3(u.p0), f3(u.p1), rrm);
      pm |= (m0 ? 1u << j0 : 0u) | (m1 ? 1u << j1 : 0u);
    }
    return pm;
  };
  // Two units per lane and step, so that their load chains overlap; the next
  // step's segment ids are on their way while this step's pairs are tested. The
  // lanes' passing pairs go to the queue at places given by a prefix sum of
  // their numbers. The capsule test stands at one place: copies of it for each
  // unit and for the last, partial batch made the loop's code outgrow the
  // instruction cache (5 of 13 stall cycles per instruction on the bundles).
  Unit a, b;
  find_unit(lane, a);
  find_unit(32 + lane, b);
  uint32_t tab = 0;  // this step's half of the unit table
  for (uint32_t t0 = 0; t0 < total; t0 += 64) {
    const bool last = t0 + 64 >= total;
    load_unit(a);
    load_unit(b);
    S.uid[tab + lane] = a.id;
    S.uid[tab + 32 + lane] = b.id;
    if (KEY16) {
      S.uli[tab + lane] = (uint16_t)a.li;
      S.uli[tab + 32 + lane] = (uint16_t)b.li;
    }
    Unit na, nb;
    na.m = nb.m = na.id = nb.id = na.li = nb.li = na.s = nb.s = 0;
    if (!last) {
      find_unit(t0 + 64 + lane, na);
      find_unit(t0 + 96 + lane, nb);
    }
    unsigned pa = line_tests(a), pb = line_tests(b);
    const uint32_t np = __popc(pa) + __popc(pb);
    uint32_t at = np;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(FULL, at, o);
      if (lane >= o) at += v;
    }
    const uint32_t end = qn + __shfl_sync(FULL, at, 31);
    at += qn - np;
    for (; pa; pa &= pa - 1) S.q[at++] = (uint16_t)((tab + lane) | (uint32_t)(__ffs(pa) - 1) << 8);
    for (; pb; pb &= pb - 1) S.q[at++] = (uint16_t)((tab + 32 + lane) | (uint32_t)(__ffs(pb) - 1) << 8);
    __syncwarp();
    // full batches, and what is left of the last step's units: the next step
    // overwrites their half of the table
    const uint32_t must = last ? end : qn;
    uint32_t done = 0;
    while (end - done >= 32 || done < must) {
      capsule_stage(done, min(end - done, 32u));
      done = min(done + 32, end);
    }
    qn = end - done;  // below 32: to the front for the next step
    const uint16_t rest = S.q[done + min((uint32_t)lane, qn)];
    __syncwarp();
    if ((uint32_t)lane < qn) S.q[lane] = rest;
    a = na;
    b = nb;
    tab ^= 64u;
  }
  __syncwarp();
  if (OPAQUE) {
    if (!take) return;
    if (COUNT) {
      ++W.vox;
      W.entries += R.len;
    }
    const unsigned long long best = S.key[lane];
    if (best != ~0ull)
      opaque_hit(A, S, R, (uint32_t)(best & 0xffffffffu),
                 hit_depth<KEY16>(A, best, f3(S.o[lane]), f3(S.d[lane])));
    R.pending = false;
    if (R.t1 < 0.0f) R.active = false;
    return;
  }
  bool redo = false;  // the ray's voxel is not composited in this round
  if (pn) {
    const uint32_t raw = S.cnt[lane];
    redo = (raw & ~kLost) > A.ray_keys || (raw & kLost);
    if (take && redo) {
      const uint32_t mine = raw & ~kLost;
      wait = mine <= min(A.ray_keys, kPool);
      if (wait) R.calls |= mine << 11;
    }
    const uint32_t nk = redo ? 0u : raw;
    const uint32_t hits = min(pn, kPool);
    uint32_t off = lane;
    if (__any_sync(FULL, raw > 1u)) {
      // pool slots ray after ray, then each ray's by key: a hit's place is the
      // number of its ray's hits with smaller keys
      off = nk;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(FULL, off, o);
        if (lane >= o) off += v;
      }
      off -= nk;
      for (uint32_t q0 = 0; q0 < hits; q0 += 32) {
        const uint32_t q = q0 + lane;
        const uint32_t ow = q < hits ? S.own[q] : 0u;
        const uint32_t oo = __shfl_sync(FULL, off, ow & 31u), on = __shfl_sync(FULL, nk, ow & 31u);
        if (q < hits && on) S.slot[oo + (ow >> 8)] = (uint8_t)q;
      }
      __syncwarp();
      for (uint32_t q0 = 0; q0 < hits; q0 += 32) {
        const uint32_t q = q0 + lane;
        const uint32_t ow = q < hits ? S.own[q] : 0u;
        const uint32_t oo = __shfl_sync(FULL, off, ow & 31u), on = __shfl_sync(FULL, nk, ow & 31u);
        if (q < hits && on) {
          const unsigned long long k = S.key[q];
          uint32_t place = 0;
          for (uint32_t i = 0; i < on; ++i) place += S.key[S.slot[oo + i]] < k;
          S.order[oo + place] = (uint8_t)q;
        }
      }
    } else if (lane < hits) {
      S.order[S.own[lane] & 31u] = (uint8_t)lane;  // at most one hit a ray, so at most 32
    }
    __syncwarp();
    if (nk) {
      float4 acc = S.acc[lane];
      const float om = 1.0f - A.alpha;
      float T = R.T;
      for (uint32_t i = 0; i < nk && T >= kTStop; ++i) {
        const uint32_t q = S.order[off + i];
        const float w = T * A.alpha;
        acc.x = fmaf(w, S.col[0][q], acc.x);
        acc.y = fmaf(w, S.col[1][q], acc.y);
        acc.z = fmaf(w, S.col[2][q], acc.z);
        T *= om;
        if (i == 0 && __float_as_int(S.inv[lane].w) < 0) {
          const unsigned long long k = S.key[q];
          S.inv[lane].w = __uint_as_float((uint32_t)(k & 0xffffffffu));
          acc.w = hit_depth<KEY16>(A, k, f3(S.o[lane]), f3(S.d[lane]));
        }
      }
      R.T = T;
      S.acc[lane] = acc;
    }
  }
  if (!take || redo) return;
  if (COUNT) {
    ++W.vox;
    W.entries += R.len;
  }
  R.calls &= ~kHits;
  R.pending = false;
  if (R.T < kTStop || R.t1 < 0.0f) R.active = false;
}

// Warp cycles since `t` into the counter `c` (instrumented trace only).
template <bool COUNT>
__device__ __forceinline__ void lap(unsigned long long& c, long long& t) {
  if (COUNT) {
    const long long now = clock64();
    c += (unsigned long long)(now - t);
    t = now;
  }
}

// Trace the rays of the warp's lanes to their ends. Every round walks at least one
// ray on, and of the rounds over the warp's pending lists every one takes at least
// one ray's list: to its end, to the count of its hits, or to the whole-warp path.
template <bool OPAQUE, bool COUNT, bool KEY16, bool AO>
__device__ __forceinline__ void trace_warp(const TraceArgs& A, WarpMem<OPAQUE, KEY16>& S, Ray& R, Work& W) {
  const int lane = threadIdx.x & 31;
  long long t = COUNT ? clock64() : 0;
  for (;;) {
    if (R.active && !R.pending) {
      const int rc = walk_brick<WarpMem<OPAQUE, KEY16>, COUNT>(A, S, R, W);
      R.pending = rc == 1;
      R.calls += kCall;
      R.active = rc != 0 && R.calls < A.max_calls;  // past the limit: given up
    }
    // The warp walks its rays one brick (or empty cube) per round and
    // processes the waiting lists once a quarter of the rays still in flight
    // wait at one (or none can walk on): walking each ray to its next list in
    // one go leaves most lanes idle while the longest walk goes on.
    const unsigned pend = __ballot_sync(FULL, R.pending);
    const unsigned walk = __ballot_sync(FULL, R.active && !R.pending);
    if (!pend && !walk) break;
    if (walk && 4 * __popc(pend) < __popc(pend | walk)) continue;
    lap<COUNT>(W.cyc[0], t);
    if (R.pending) resolve_list<WarpMem<OPAQUE, KEY16>, COUNT>(A, S, R);
    __syncwarp();
    bool more;
    do {
      bool wait;
      process_flat<OPAQUE, COUNT, KEY16, AO>(A, S, R, W, wait);
      lap<COUNT>(W.cyc[1], t);
      // long lists: the whole warp on one list at a time
      unsigned pm = __ballot_sync(FULL, R.pending && !wait);
      while (pm) {
        const int L = __ffs(pm) - 1;
        pm &= pm - 1;
        const uint32_t beg = __shfl_sync(FULL, R.beg, L), end = beg + __shfl_sync(FULL, R.len, L);
        unsigned n_cap = 0, n_hit = 0, n_scan = 0;
        if constexpr (OPAQUE) {
          const unsigned long long best = voxel_nearest<COUNT, KEY16>(A, S, L, beg, end, n_cap, n_hit);
          n_scan = end - beg;
          if (lane == L && best != ~0ull)
            opaque_hit(A, S, R, (uint32_t)(best & 0xffffffffu),
                       hit_depth<KEY16>(A, best, f3(S.o[L]), f3(S.d[L])));
        } else {
          const float T = voxel_composite<COUNT, KEY16, AO>(A, S, L, beg, end,
                                                            __shfl_sync(FULL, R.T, L), n_cap, n_hit, n_scan);
          if (lane == L) {
            R.T = T;
            if (T < kTStop) R.active = false;
          }
        }
        __syncwarp();
        if (lane == L) {
          R.pending = false;
          if (R.t1 < 0.0f) R.active = false;
        }
        if (COUNT) {
          W.cap += n_cap;
          W.hits += n_hit;
          if (lane == L) {
            ++W.vox;
            ++W.ww_vox;
            W.entries += end - beg;
            W.ww_ent += n_scan;
          }
        }
      }
      lap<COUNT>(W.cyc[2], t);
      more = __any_sync(FULL, R.pending);
    } while (more);
  }
  if (R.calls >= A.max_calls) set_err(A.g.st, kErrTimeout);
  lap<COUNT>(W.cyc[0], t);
}

template <bool COUNT>
__device__ __forceinline__ void count_work(const TraceArgs& A, const Work& W) {
  if (!COUNT) return;
  unsigned long long v[7] = {W.entries, W.cap, W.vox, W.steps, W.hits, W.ww_vox, W.ww_ent};
  unsigned long long* out[7] = {&A.g.st->tr_entries, &A.g.st->tr_capsule, &A.g.st->tr_voxels,
                                &A.g.st->tr_steps, &A.g.st->tr_hits, &A.g.st->tr_ww_voxels,
                                &A.g.st->tr_ww_entries};
  for (int i = 0; i < 7; ++i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(FULL, v[i], o);
    if ((threadIdx.x & 31) == 0) atomicAdd(out[i], v[i]);
  }
  if ((threadIdx.x & 31) == 0)
    for (int k = 0; k < 4; ++k) atomicAdd(&A.g.st->tr_cycles[k], W.cyc[k]);
}

// Write a finished pixel (or queue it for the repair re-trace).
template <class M>
__device__ __forceinline__ void write_pixel(const TraceArgs& A, const M& S, const Ray& R) {
  const int lane = threadIdx.x & 31;
  if (R.missed) {
    const uint32_t q = atomicAdd(A.pq_cnt, 1u);
    if (q < A.pq_cap) A.pq[q] = R.pix;
    else set_err(A.g.st, kErrOverflow);
    return;
  }
  const float4 c = S.acc[lane];
  A.rgba[R.pix] = make_float4(c.x, c.y, c.z, 1.0f - R.T);
  if (A.first_id) A.first_id[R.pix] = __float_as_int(S.inv[lane].w);
  if (A.first_t) A.first_t[R.pix] = c.w;
}

// Resident blocks per SM the trace kernels are compiled for: 96 registers for
// the transparent trace, which spills 28 bytes of stores and 36 of loads at that (6
// blocks, at 80 registers, spill far more: sparse walks at 4K 25.8 ms against
// 20.8; 4 blocks 24.6), 72 for the opaque one.
template <bool OPAQUE, bool COUNT, bool AO>
constexpr int kMinBlocks = COUNT ? 1 : (OPAQUE ? 6 : (AO ? 4 : 5));

// Main trace. A warp takes one tile of A.tile_n pixels, tile_w wide, at a time,
// four neighbouring tiles (2x2) in a row to keep what their rays share in L1, and
// its lanes write their pixels together at the end. Warps take their tiles from
// a counter: the cost of a tile varies with the lists behind it, and a fixed
// tile per warp left the slots of a block's finished warps idle until its slowest
// was done. The counter hands out each number once and a number past the tiles
// ends the warp, so the passes of a launch number at most its tiles and warps. (A
// count of each warp's passes in shared memory cost 4% of a static view.)
template <bool OPAQUE, bool COUNT, bool KEY16, bool AO>
__global__ void __launch_bounds__(kTraceThreads, kMinBlocks<OPAQUE, COUNT, AO>) k_trace_tile(const __grid_constant__ TraceArgs A) {
  __shared__ WarpMem<OPAQUE, KEY16> s_mem[kTraceThreads / 32];
  const int lane = threadIdx.x & 31;
  WarpMem<OPAQUE, KEY16>& S = s_mem[threadIdx.x >> 5];
  const int tw = A.tile_w, th = A.tile_n / tw;
  const uint32_t quads_x = (uint32_t)(A.cam.width + 2 * tw - 1) / (uint32_t)(2 * tw);
  const uint32_t quads_y = (uint32_t)(A.cam.height + 2 * th - 1) / (uint32_t)(2 * th);
  const uint32_t block = blockIdx.x + dependency_wait();
  Work W;
  for (bool more = true; more; more = !OPAQUE) {
    uint32_t tile = block * (kTraceThreads / 32) + (threadIdx.x >> 5);
    if (!OPAQUE) {
      if (lane == 0) tile = atomicAdd(A.work_next, 1u);
      tile = __shfl_sync(FULL, tile, 0);
    }
    const uint32_t quad = tile >> 2;
    if (quad >= quads_x * quads_y) break;
    const int px = (int)(quad % quads_x) * 2 * tw + (int)(tile & 1u) * tw + (lane & (tw - 1));
    const int py = (int)(quad / quads_x) * 2 * th + (int)((tile >> 1) & 1u) * th + lane / tw;
    const bool valid = lane < A.tile_n && px < A.cam.width && py < A.cam.height;
    Ray R;
    init_ray(A, S, R, px, py, valid);
    __syncwarp();
    trace_warp<OPAQUE, COUNT, KEY16, AO>(A, S, R, W);
    if (valid) write_pixel(A, S, R);
    __syncwarp();
  }
  count_work<COUNT>(A, W);
}

// Repair re-trace of the queued pixels: each warp takes its share of the queue
// (one pixel each when few are queued), at most 32 at a time.
template <bool OPAQUE, bool COUNT, bool KEY16, bool AO>
__global__ void __launch_bounds__(kTraceThreads, kMinBlocks<OPAQUE, COUNT, AO>) k_trace_list(const __grid_constant__ TraceArgs A) {
  __shared__ WarpMem<OPAQUE, KEY16> s_mem[kTraceThreads / 32];
  const int lane = threadIdx.x & 31;
  WarpMem<OPAQUE, KEY16>& S = s_mem[threadIdx.x >> 5];
  dependency_wait();
  const uint32_t total = min(*A.pix_count, A.pq_cap);
  const uint32_t n_warps = gridDim.x * (blockDim.x >> 5);
  const uint32_t share = min(32u, (total + n_warps - 1) / n_warps);
  Work W;
  while (total) {
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(A.work_next, share);
    base = __shfl_sync(FULL, base, 0);
    if (base >= total) break;
    const bool valid = (uint32_t)lane < share && base + lane < total;
    const uint32_t pix = valid ? A.pix_list[base + lane] : 0u;
    Ray R;
    init_ray(A, S, R, (int)(pix % (uint32_t)A.cam.width), (int)(pix / (uint32_t)A.cam.width), valid);
    if (valid && A.resume) resume_ray(A, S, R);
    __syncwarp();
    trace_warp<OPAQUE, COUNT, KEY16, AO>(A, S, R, W);
    if (valid) write_pixel(A, S, R);
    __syncwarp();
  }
  count_work<COUNT>(A, W);
}

template <bool OPAQUE, bool COUNT, bool KEY16, bool AO>
void launch_one(const TraceArgs& a, const Queue& q) {
  if (a.pix_list) {
    launch(k_trace_list<OPAQUE, COUNT, KEY16, AO>, kSms * 4, kTraceThreads, q, a);
    return;
  }
  const int tw = a.tile_w, th = a.tile_n / tw;
  // opaque: a block per 2x2 tiles; transparent: as many blocks as the kernel is
  // compiled to keep resident
  const unsigned blocks = OPAQUE ? ((a.cam.width + 2 * tw - 1) / (2 * tw)) * ((a.cam.height + 2 * th - 1) / (2 * th))
                                 : kSms * (COUNT ? 4 : kMinBlocks<OPAQUE, COUNT, AO>);
  launch(k_trace_tile<OPAQUE, COUNT, KEY16, AO>, blocks, kTraceThreads, q, a);
}

template <bool COUNT, bool KEY16>
void launch_mode(const TraceArgs& a, int K, const Queue& q) {
  if (K == 1) launch_one<true, COUNT, KEY16, false>(a, q);  // AO: k_shade_hits
  else if (a.ao == 1) launch_one<false, COUNT, KEY16, true>(a, q);
  else launch_one<false, COUNT, KEY16, false>(a, q);
}

int launch_trace(const TraceArgs& args, int K, const Queue& q) {
  TraceArgs a = args;
  a.tile_n = 32;
  // A ray's walk calls: one a brick and one an occupied voxel on its way, at most
  // 3 n / 4 and 3 n, doubled for the voxel that a clamped crossing may step back.
  if (a.max_calls == 0) a.max_calls = 8u * (uint32_t)a.g.n + 64u;
  a.max_calls *= kCall;
  if (K > 1) {
    a.tile_n = transparent_tile_rays((long long)a.cam.width * a.cam.height);
    if (a.tile_n < 32) a.tile_w = a.tile_n == 16 ? 4 : 2;
  }
  if (a.count) {
    if (a.key16) launch_mode<true, true>(a, K, q);
    else launch_mode<true, false>(a, K, q);
  } else {
    if (a.key16) launch_mode<false, true>(a, K, q);
    else launch_mode<false, false>(a, K, q);
  }
  return 1;
}

// Cone AO of an opaque trace: the pixels hold their hits (opaque_hit), and one
// thread per pixel, 8x4 tiles to a warp, shades them after the last repair
// round. Inside the trace the rays of a warp find their hits in different
// rounds, so few of its lanes shaded at a time, at the trace's occupancy
// (95% of the trace's cycles on the 1080p ABC view); here every lane has a hit
// and neighbours share texels.
__global__ void __launch_bounds__(kTraceThreads) k_shade_hits(TraceArgs A) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int px = blockIdx.x * 16 + (warp & 1) * 8 + (lane & 7) + (int)dependency_wait();
  const int py = blockIdx.y * 8 + (warp >> 1) * 4 + (lane >> 3);
  if (px >= A.cam.width || py >= A.cam.height) return;
  float4* out = &A.rgba[(size_t)py * A.cam.width + px];
  const float4 v = *out;
  // no hit (transparent black), or a pixel that the repair left unfinished (vrt_sync
  // reports it): it holds what the caller's image held
  if (__float_as_uint(v.z) != kHitTag) return;
  const uint32_t id = __float_as_uint(v.x);
  if (id >= A.n_vert || id + 1 >= A.n_vert) return;
  float3 o, d;
  pixel_ray(A.cam, px, py, o, d);
  const float3 c = ao_lane(A, o + v.y * d) *
                   tangent_colour(f3(__ldg(&A.pos[id])), f3(__ldg(&A.pos[id + 1])));
  *out = make_float4(A.alpha * c.x, A.alpha * c.y, A.alpha * c.z, v.w);
}

int launch_shade_hits(const TraceArgs& a, const Queue& q) {
  const dim3 grid((a.cam.width + 15) / 16, (a.cam.height + 7) / 8);
  launch(k_shade_hits, grid, kTraceThreads, q, a);
  return 1;
}

// --------------------------------------------------- instrumented trace
__global__ void k_touch_count(const uint32_t* bits, size_t words, unsigned long long* out) {
  dependency_wait();
  unsigned long long c = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < words;
       i += (size_t)gridDim.x * blockDim.x)
    c += __popc(bits[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(FULL, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

int launch_touch_count(const uint32_t* list_bits, size_t list_words, const uint32_t* vert_bits,
                       size_t vert_words, const uint32_t* vox_bits, size_t vox_words,
                       DevStatus* st, const Queue& q) {
  launch(k_touch_count, kSms * 4, 256, q, list_bits, list_words, &st->tr_u_entries);
  launch(k_touch_count, kSms * 4, 256, q, vert_bits, vert_words, &st->tr_u_vertices);
  launch(k_touch_count, kSms * 4, 256, q, vox_bits, vox_words, &st->tr_u_voxels);
  return 3;
}

// ----------------------------------------------------------------- repair
__global__ void k_repair_alloc(GridDev g, const uint32_t* vq, const uint32_t* vq_cnt,
                               const uint32_t* pq_cnt, uint32_t vq_cap) {
  dependency_wait();
  const uint32_t nq = min(*vq_cnt, vq_cap);
  if (blockIdx.x == 0 && threadIdx.x == 0 && nq) {
    atomicAdd(&g.st->repair_rounds, 1u);
    atomicAdd(&g.st->repaired_voxels, nq);
    atomicAdd(&g.st->retraced_pixels, *pq_cnt);
  }
  for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += gridDim.x * blockDim.x) {
    const uint32_t idx = vq[q];
    const uint32_t cnt = g.word[idx] & 0xffffu;
    const uint32_t start = atomicAdd(&g.st->list_tail, cnt);
    if ((unsigned long long)start + cnt > g.list_cap) set_err(g.st, kErrOverflow);
    g.cur[idx] = start;
    atomicOr(&g.vis[idx >> 5], 1u << (idx & 31));
  }
}

__global__ void k_repair_clear(GridDev g, uint32_t* need, const uint32_t* vq, const uint32_t* vq_cnt,
                               uint32_t vq_cap, int next) {
  dependency_wait();
  const uint32_t nq = min(*vq_cnt, vq_cap);
  for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += gridDim.x * blockDim.x) {
    const uint32_t idx = vq[q];
    atomicAnd(&need[idx >> 5], ~(1u << (idx & 31)));
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    g.st->vq_cnt[next] = 0;
    g.st->pq_cnt[next] = 0;
  }
}

int launch_repair_alloc(const GridDev& g, const uint32_t* vq, const uint32_t* vq_cnt,
                        const uint32_t* pq_cnt, uint32_t vq_cap, const Queue& q) {
  launch(k_repair_alloc, kSms, 256, q, g, vq, vq_cnt, pq_cnt, vq_cap);
  return 1;
}

int launch_repair_clear(const GridDev& g, uint32_t* need, const uint32_t* vq,
                         const uint32_t* vq_cnt, uint32_t vq_cap, int next, const Queue& q) {
  launch(k_repair_clear, kSms, 256, q, g, need, vq, vq_cnt, vq_cap, next);
  return 1;
}

}  // namespace vrt
