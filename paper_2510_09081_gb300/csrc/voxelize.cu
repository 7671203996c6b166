// A1 / A5: the two voxelization passes of the voxelize-(cull-)scan-voxelize
// list build (Sec. 3.1, 3.3).
//
// Both passes enumerate the same candidate voxels per segment -- the
// slab-by-slab traversal of Alg. 1 along the major axis a0 of d = v1 - v0, each
// slab visiting a 2D box of minor-axis voxels around the segment -- and keep a
// voxel iff the segment lies within the list radius of the voxel's closed box.
// The minor half-extent of a slab uses the exact half-width of the tube's
// cross-section in a major-axis plane, rl * sqrt(1 + (d_ai / d_a0)^2), which is
// never below Eq. 1's projected radius. Every slab's box is indexed with the
// same width bound (the slab's extent along a minor axis is at most
// |d_ai / d_a0| + 2 * half-extent), so candidate q of a segment decodes in O(1).
//
// Work layout: each lane loads one segment (coalesced), sets up its walk and
// stores it in shared memory; the warp numbers the candidates of its 32 segments
// consecutively and takes them 32 at a time, each lane reading the record of the
// segment its candidate belongs to, so segments of different lengths do not
// leave lanes idle, and neighbouring lanes have neighbouring voxels (their atomics
// share sectors). The fp32 filter decides almost every candidate; pairs it
// cannot decide go to a queue that a separate kernel decides exactly (keeping
// the 128-bit integer path out of the hot kernels' registers).
//
// Pass 1 adds (occupancy code << 16) | 1 to the voxel's packed word with a
// 32-bit atomic (Sec. 3.1) and writes the fragment as an 8-byte record (voxel << 32 |
// segment) with its rank, the count field the atomic returned (fragments of
// the voxel added before it), beside it. A block takes record slots for all its
// walks' candidates with one atomic; each warp writes its fragments at the
// start of its share and marks the rest (candidates that were not kept)
// kNoRecord. The paper re-voxelizes in its second pass to save memory; with the
// records in HBM the second pass is a streaming scatter instead: for every
// record whose voxel received a list, write the segment id at the slot its
// rank gives below the voxel's list end (Sec. 3.3), with no atomic.
#include "launch.h"

namespace vrt {

constexpr int kPass1Warps = kPass1Threads / 32;
constexpr float kWalkEps = 1e-3f;
constexpr unsigned FULLW = 0xffffffffu;

constexpr int kBoxSlabs = 9;        // slabs whose boxes a segment's record holds
constexpr int kTableSlabs = 8;      // slabs an owner table's byte can name
constexpr uint32_t kWindow = 512;  // candidates of a warp whose owners are tabulated at a time

// One segment in shared memory. Short segments (up to kBoxSlabs slabs; nearly all)
// keep the box of each slab: x = j0 | l0 << 10 | w2 << 20 (first voxel on the two
// minor axes, width on the second), y = candidates of the segment before the slab
// | ceil(4096 / w2) << 16. Longer ones keep what slab_box needs, and index every
// slab's box with the widest slab's widths.
struct Seg {
  float4 a;   // v0; reciprocal of |d|^2 (0 for a point)
  float4 d;   // v1 - v0; largest squared distance stage 1 accepts
  float4 n0;  // clip normal at v0; m | c0 << 2 | clip flags << 12 | boxed << 14
  float4 n1;  // clip normal at v1; the segment's first candidate number
  union {
    uint2 box[kBoxSlabs];
    struct {
      float s1, s2, rho1, rho2, lo_m, hi_m, inv_w12, inv_w2;
      int w1, w2;
    } g;
  };
};
static_assert(sizeof(Seg) == 144, "records next to each other start four banks apart");

// Minor-axis voxel ranges of slab c (clamped to the grid): the axis line
// a_k + (x - a_m) s_k over the slab's part of [lo_m, hi_m], widened by rho_k.
__device__ __forceinline__ void slab_box(float am, float a1, float a2, float s1, float s2,
                                         float rho1, float rho2, float lo_m, float hi_m, int n,
                                         int c, int& j0, int& j1, int& l0, int& l1) {
  const float x0 = fmaxf((float)c, lo_m), x1 = fminf((float)(c + 1), hi_m);
  const float p1a = fmaf(x0 - am, s1, a1), p1b = fmaf(x1 - am, s1, a1);
  const float p2a = fmaf(x0 - am, s2, a2), p2b = fmaf(x1 - am, s2, a2);
  j0 = max(0, (int)floorf(fminf(p1a, p1b) - rho1));
  j1 = min(n - 1, (int)floorf(fmaxf(p1a, p1b) + rho1));
  l0 = max(0, (int)floorf(fminf(p2a, p2b) - rho2));
  l1 = min(n - 1, (int)floorf(fmaxf(p2a, p2b) + rho2));
}

// Set up the walk of segment a, b into its record (all but n0.w's flags' clip part
// and n1, which the caller fills): the numbers its candidates take, and in `voxels`
// how many of them are voxels. Approximate division and square roots serve:
// kWalkEps widens every box by far more than their error.
__device__ __forceinline__ uint32_t walk_setup(float3 a, float3 b, const GridDev& g, Seg& S,
                                               uint32_t& bits, bool& short_walk,
                                               uint32_t& voxels) {
  const float rl = g.rl;
  const int n = g.n;
  const float3 d = b - a;
  const float ax = fabsf(d.x), ay = fabsf(d.y), az = fabsf(d.z);
  const int m = (ax >= ay && ax >= az) ? 0 : (ay >= az ? 1 : 2);
  const int k1 = m == 0 ? 1 : 0, k2 = m == 2 ? 1 : 2;
  const float am = cmp3(a, m), dm = cmp3(d, m);
  const float inv = dm != 0.0f ? div_normal(1.0f, dm) : 0.0f;  // |dm| >= 2^-14
  const float s1 = cmp3(d, k1) * inv, s2 = cmp3(d, k2) * inv;
  const float q1 = fmaf(s1, s1, 1.0f), q2 = fmaf(s2, s2, 1.0f);
  const float rho1 = fmaf(rl * q1, rsqrt_normal(q1), kWalkEps);
  const float rho2 = fmaf(rl * q2, rsqrt_normal(q2), kWalkEps);
  const float lo_m = fminf(am, am + dm) - rl, hi_m = fmaxf(am, am + dm) + rl;
  const float a1 = cmp3(a, k1), a2 = cmp3(a, k2);
  const int c0 = max(0, (int)floorf(lo_m - kWalkEps));
  const int c1 = min(n - 1, (int)floorf(hi_m + kWalkEps));
  const int slabs = c1 - c0 + 1;
  const float dd = dot3(d, d);
  // Stage 1's rounding allowance: six times seg_box_tol's, at the largest local
  // coordinate a candidate of this segment can have, which covers the rounding
  // of the nearest point's parameter too (its distance along the axis from the
  // true nearest point, which would otherwise enter the lower bound).
  const float M = fmaxf(ax, fmaxf(ay, az)) + 1.5f * rl + 4.0f;
  S.a = make_float4(a.x, a.y, a.z, dd > 0.0f ? div_normal(1.0f, dd) : 0.0f);
  S.d = make_float4(d.x, d.y, d.z, fmaf(rl, rl, -2.9e-6f * M * M));
  const bool boxed = slabs <= kBoxSlabs;
  short_walk = slabs <= kTableSlabs;
  bits = (uint32_t)m | ((uint32_t)c0 << 2) | (boxed ? 1u << 14 : 0u);
  voxels = 0;
  if (slabs <= 0) return 0;
  if (boxed) {
    uint32_t total = 0;
    for (int k = 0; k < slabs; ++k) {
      int j0, j1, l0, l1;
      slab_box(am, a1, a2, s1, s2, rho1, rho2, lo_m, hi_m, n, c0 + k, j0, j1, l0, l1);
      // widths stay below 16: |s| <= 1 and the radius is at most 4
      const uint32_t w1 = (uint32_t)max(0, j1 - j0 + 1), w2 = (uint32_t)max(0, l1 - l0 + 1);
      const uint32_t wd = max(1u, w2);
      S.box[k] = make_uint2(((uint32_t)j0 & 1023u) | (((uint32_t)l0 & 1023u) << 10) | (wd << 20),
                            total | ((4095u + wd) / wd) << 16);
      total += w1 * w2;
    }
    for (int k = slabs; k < kBoxSlabs; ++k) S.box[k].y = 0xffffu;  // past every candidate
    voxels = total;
    return total;
  }
  int W1 = 1, W2 = 1;
  for (int c = c0; c <= c1; ++c) {
    int j0, j1, l0, l1;
    slab_box(am, a1, a2, s1, s2, rho1, rho2, lo_m, hi_m, n, c, j0, j1, l0, l1);
    W1 = max(W1, j1 - j0 + 1);
    W2 = max(W2, l1 - l0 + 1);
    voxels += (uint32_t)(max(0, j1 - j0 + 1) * max(0, l1 - l0 + 1));
  }
  S.g.s1 = s1; S.g.s2 = s2; S.g.rho1 = rho1; S.g.rho2 = rho2;
  S.g.lo_m = lo_m; S.g.hi_m = hi_m;
  S.g.inv_w12 = 1.0f / (float)(W1 * W2);
  S.g.inv_w2 = 1.0f / (float)W2;
  S.g.w1 = W1; S.g.w2 = W2;
  return (uint32_t)slabs * (uint32_t)(W1 * W2);
}

// Minor-axis voxels j, l of slab c to x, y, z.
__device__ __forceinline__ void place(uint32_t m, int c, int j, int l, int& x, int& y, int& z) {
  x = m == 0 ? c : j;
  y = m == 1 ? c : (m == 0 ? j : l);
  z = m == 2 ? c : l;
}

// Candidate q of a segment that is not boxed: its voxel, or false when q falls
// outside its slab's box.
__device__ __forceinline__ bool decode_long(const Seg& S, uint32_t bits, int n, uint32_t q, int& x,
                                            int& y, int& z) {
  const uint32_t m = bits & 3u;
  const float am = m == 0 ? S.a.x : (m == 1 ? S.a.y : S.a.z);
  const float a1 = m == 0 ? S.a.y : S.a.x;
  const float a2 = m == 2 ? S.a.y : S.a.z;
  // (q + 1/2) / w is at least 1/(2w) from an integer, far beyond fp32 error for
  // these small counts, so truncation gives the exact quotient
  const int slab = (int)(((float)q + 0.5f) * S.g.inv_w12);
  const int rem = (int)q - slab * (S.g.w1 * S.g.w2);
  const int c = (int)((bits >> 2) & 1023u) + slab;
  int j0, j1, l0, l1;
  slab_box(am, a1, a2, S.g.s1, S.g.s2, S.g.rho1, S.g.rho2, S.g.lo_m, S.g.hi_m, n, c, j0, j1, l0, l1);
  const int dj = (int)(((float)rem + 0.5f) * S.g.inv_w2);
  const int j = j0 + dj, l = l0 + rem - dj * S.g.w2;
  if (j > j1 || l > l1) return false;
  place(m, c, j, l, x, y, z);
  return true;
}

// Queue the (segment, voxel) pairs of the lanes with q set for the exact
// decision, one atomic per warp (all lanes call).
__device__ __forceinline__ void queue_exact(const GridDev& g, bool q, uint32_t seg, int x, int y,
                                            int z, int lane) {
  const unsigned m = __ballot_sync(FULLW, q);
  if (!m) return;
  uint32_t base = 0;
  if (lane == __ffs(m) - 1) base = atomicAdd(&g.st->xq_cnt, (uint32_t)__popc(m));
  base = __shfl_sync(FULLW, base, __ffs(m) - 1);
  if (q) {
    const uint32_t k = base + __popc(m & ((1u << lane) - 1u));
    if (k < g.xq_cap) g.xq[k] = make_uint2(seg, pack_voxel(x, y, z));
    else set_err(g.st, kErrOverflow);
  }
}

// The block's pass-1 counters into the status, three atomics per block (all
// threads of the block call).
__device__ __forceinline__ void flush_counters_block(DevStatus* st, unsigned long long F,
                                                     unsigned long long q, unsigned long long ex) {
  __shared__ unsigned long long s_c[3][8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    F += __shfl_down_sync(FULLW, F, o);
    q += __shfl_down_sync(FULLW, q, o);
    ex += __shfl_down_sync(FULLW, ex, o);
  }
  const int wid = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    s_c[0][wid] = F;
    s_c[1][wid] = q;
    s_c[2][wid] = ex;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    unsigned long long v = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) v += s_c[threadIdx.x][k];
    if (v) atomicAdd(threadIdx.x == 0 ? &st->F : (threadIdx.x == 1 ? &st->sum_q : &st->exact_decisions), v);
  }
}

__device__ __forceinline__ void flush_counters(DevStatus* st, unsigned long long F,
                                               unsigned long long q, unsigned long long ex) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    F += __shfl_down_sync(FULLW, F, o);
    q += __shfl_down_sync(FULLW, q, o);
    ex += __shfl_down_sync(FULLW, ex, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (F) atomicAdd(&st->F, F);
    if (q) atomicAdd(&st->sum_q, q);
    if (ex) atomicAdd(&st->exact_decisions, ex);
  }
}

// Candidate number at which slab q of a boxed segment ends: the next slab's start
// (slabs past the last start beyond the segment's end).
__device__ __forceinline__ uint32_t slab_end(const Seg& S, int q, uint32_t first, uint32_t end) {
  return q + 1 < kBoxSlabs ? min(end, first + (S.box[q + 1].y & 0xffffu)) : end;
}

// Occupancy code (Alg. 3 around Alg. 2, quantized) of a voxel whose centre lies at
// pa from v0, pb from v1 and at squared distance q2 from the axis.
__device__ __forceinline__ uint32_t occupancy_code(const GridDev& g, float3 pa, float3 pb, float q2,
                                                   float3 n0, float3 n1, bool en0, bool en1) {
  float s = (q2 > 0.0f ? q2 * rsqrt_normal(q2) : 0.0f) - g.r_clamp;
  if (en0) s = fmaxf(s, -dot3(pa, n0));
  if (en1) s = fmaxf(s, dot3(pb, n1));
  const float occ = fminf(1.0f, fmaxf(0.0f, 0.5f - s)) * g.corr;
  return (uint32_t)floorf(fmaf(g.occ_scale, occ, 0.5f));
}

// The packed-word increment (occupancy code << 16) | 1 of one fragment (Alg. 3
// at the voxel centre, quantized); counts it in F and sq.
__device__ __forceinline__ uint32_t fragment_word(const GridDev& g, float3 a, float3 b, float3 n0,
                                                  float3 n1, bool en0, bool en1, int x, int y,
                                                  int z, unsigned long long& F,
                                                  unsigned long long& sq) {
  const float3 o = make_float3((float)x, (float)y, (float)z);
  const float occ = capsule_occupancy(make_float3(0.5f, 0.5f, 0.5f), a - o, b - o, n0, n1, en0,
                                      en1, g.r_clamp, g.corr);
  const uint32_t q = (uint32_t)floorf(fmaf(g.occ_scale, occ, 0.5f));
  F += 1;
  sq += q;
  return (q << 16) | 1u;
}

// Adds a fragment to its voxel's packed word; returns its rank in the voxel.
__device__ __forceinline__ uint32_t add_fragment(const GridDev& g, float3 a, float3 b, float3 n0,
                                                 float3 n1, bool en0, bool en1, int x, int y,
                                                 int z, unsigned long long& F,
                                                 unsigned long long& sq) {
  return atomicAdd(&g.word[brick_index(x, y, z, g.log2nb)],
                   fragment_word(g, a, b, n0, n1, en0, en1, x, y, z, F, sq)) & 0xffffu;
}

// A record slot pass 1 took for a candidate it did not keep.
constexpr unsigned long long kNoRecord = ~0ull;

constexpr int kWarpRecords = 256;  // pass 2: culled records a warp stages per append
constexpr uint32_t kNoCopy = 0xffffffffu;  // cq_cnt: pass 2 copied no culled records

// Append a warp's staged culled records to cq (all lanes call); records past
// the queue's capacity are counted but dropped, which sends the repair rounds
// back to the full record stream.
__device__ __forceinline__ void flush_culled(const GridDev& g, unsigned long long* cq,
                                             const unsigned long long* srec, int n, int lane) {
  if (n == 0) return;
  uint32_t r0 = 0;
  if (lane == 0) r0 = atomicAdd(&g.st->cq_cnt, (uint32_t)n);
  r0 = __shfl_sync(FULLW, r0, 0);
  for (int k = lane; k < n; k += 32) {
    const uint32_t r = r0 + (uint32_t)k;
    if (r < g.xq_cap) cq[r] = srec[k];
  }
  __syncwarp();
}

// Bound by instruction issue (82% of the issue slots before and after), so a
// candidate's work is cut to what it needs: the owner and slab of a candidate come
// from a byte table the warp's lanes fill (one load instead of a search over the
// lanes and comparisons over the slabs), the slab's box and the segment's
// reciprocal length from its record, and the filter's point on the axis, its
// offset from the voxel centre and their distance serve the occupancy too (Alg. 2
// measures the same point). Records of 128 bytes put all lanes' loads on the
// same banks (72% of the shared-memory pipe); 144 bytes do not. Bundles (114M
// fragments, 256^3) 2.40 -> 1.74 ms, ABC flow (195M, 512^3) 4.71 -> 3.71 ms (1.65 and
// 3.42 with the bracketed Newton steps and pairs of floats that came after); without
// the atomics 10% less, so they are not what bounds it.
__global__ void __launch_bounds__(kPass1Threads, kPass1Blocks) k_pass1(const float4* __restrict__ pos,
                                                  const float4* __restrict__ nrm,
                                                  const uint32_t* __restrict__ order, long long V,
                                                  int segs_per_warp, GridDev g) {
  __shared__ Seg s_seg[kPass1Threads];
  __shared__ uint32_t s_id[kPass1Threads];          // segment id of each lane's record
  __shared__ uint8_t s_own[kPass1Warps][kWindow];   // candidate -> lane | slab << 5 (boxed segments)
  // Candidates the first filter stage leaves undecided (a few percent) wait in
  // a per-warp queue and get the Newton stage 32 at a time, so the warp does
  // not run it for one or two lanes per step.
  __shared__ uint2 s_uq[kPass1Warps][64];           // (owner lane, packed voxel)
  __shared__ uint32_t s_wtot[kPass1Warps];
  __shared__ unsigned long long s_rbase;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, tid = threadIdx.x;
  const long long base = ((long long)blockIdx.x * kPass1Warps + wid) * segs_per_warp;
  // slots in spatial order (nearby segments in the same and neighbouring
  // warps keep the packed-word atomics within a smaller part of the grid)
  const long long k = base + lane + dependency_wait();
  const long long i = lane < segs_per_warp && k < V ? (order ? (long long)__ldg(&order[k]) : k) : V;
  uint32_t count = 0, bits = 0, voxels = 0;
  bool short_walk = true;
  if (i + 1 < V) {
    const float4 p0 = pos[i];
    const uint32_t f0 = __float_as_uint(p0.w);
    if (!(f0 & kLast)) {
      const float4 p1 = pos[i + 1];
      const float4 m0 = nrm[i], m1 = nrm[i + 1];
      Seg& S = s_seg[tid];
      count = walk_setup(f3(p0), f3(p1), g, S, bits, short_walk, voxels);
      bits |= ((f0 & kClipOn) ? 1u << 12 : 0u) | ((__float_as_uint(p1.w) & kClipOn) ? 1u << 13 : 0u);
      S.n0 = make_float4(m0.x, m0.y, m0.z, __uint_as_float(bits));
      S.n1 = make_float4(m1.x, m1.y, m1.z, 0.0f);
      s_id[tid] = (uint32_t)i;
    }
  }
  // The warp's candidates, segment after segment, are numbered 0..total-1.
  uint32_t incl = count;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(FULLW, incl, o);
    if (lane >= o) incl += v;
  }
  const uint32_t total = __shfl_sync(FULLW, incl, 31);
  const uint32_t first = incl - count;
  const uint32_t slots = __reduce_add_sync(FULLW, voxels);  // record slots the warp needs at most
  if (count) s_seg[tid].n1.w = __uint_as_float(first);
  // record slots: one atomic per block for all its candidates, warp shares in
  // warp order (one atomic per warp on the single counter kept pass 1 waiting
  // on sets of many short segments: ABC at 1/8 of its lines 0.56 -> 0.75 ms);
  // the first window's table is filled while it is under way
  if (lane == 0) s_wtot[wid] = slots;
  __syncthreads();
  if (tid == 0) {
    uint32_t sum = 0;
    for (int q = 0; q < kPass1Warps; ++q) {
      const uint32_t t = s_wtot[q];
      s_wtot[q] = sum;
      sum += t;
    }
    s_rbase = sum ? atomicAdd(&g.st->rec_cnt, (unsigned long long)sum) : 0ull;
  }
  const bool tabled = __all_sync(FULLW, short_walk || !count);
  // owner and slab of the candidates of window [w0, w1)
  auto fill = [&](uint32_t w0, uint32_t w1) {
    if (!tabled || !count) return;
    uint32_t s0 = first;
    for (int q = 0; q < kTableSlabs && s0 < incl; ++q) {
      const uint32_t s1 = slab_end(s_seg[tid], q, first, incl);
      for (uint32_t c = max(s0, w0); c < min(s1, w1); ++c) s_own[wid][c - w0] = (uint8_t)(lane | q << 5);
      s0 = s1;
    }
  };
  fill(0u, min(total, kWindow));
  __syncthreads();
  // Past the capacity, `room` slots of the warp's share exist.
  const unsigned long long rbase = s_rbase + s_wtot[wid];
  const uint32_t room = rbase < g.rec_cap ? (uint32_t)min((unsigned long long)slots, g.rec_cap - rbase) : 0u;
  unsigned long long* rec = g.rec + min(rbase, (unsigned long long)g.rec_cap);
  uint16_t* rank = g.rank + min(rbase, (unsigned long long)g.rec_cap);
  const Seg* segs = s_seg + (tid & ~31);
  const uint32_t* ids = s_id + (tid & ~31);
  unsigned long long sq = 0;
  uint32_t sq32 = 0, ex = 0;  // a window's codes: at most 32 steps (and stage 2's) of 16 bits
  const unsigned lt = (1u << lane) - 1u;
  uint2* uq = s_uq[wid];
  uint32_t un = 0;      // queued (uniform)
  uint32_t wcount = 0;  // records this warp has written (uniform)
  // A fragment's rank is stored one emit later, so the latency of the
  // returning atomic that gives it overlaps a step of work: pend_r is the
  // record slot still waiting for its rank, the count field of the word
  // pend_old that the lane's atomic returned.
  uint32_t pend_r = ~0u, pend_old = 0;
  auto flush_rank = [&]() {  // all lanes call
    if (pend_r != ~0u) rank[pend_r] = (uint16_t)pend_old;  // low 16 bits: count
    pend_r = ~0u;
  };
  // a kept fragment: occupancy into the packed word, record written (all lanes
  // call). w: the voxel's centre seen from v0, e2: its squared distance to the axis.
  auto emit = [&](bool keep, int j, const float4& n0, float3 w, float e2, int x, int y, int z) {
    flush_rank();
    const unsigned am = __ballot_sync(FULLW, keep);
    if (keep) {
      const Seg& S = segs[j];
      const float3 pb = w - f3(S.d);
      const uint32_t clip = __float_as_uint(n0.w) >> 12;
      const uint32_t q = occupancy_code(g, w, pb, e2, f3(n0), f3(S.n1), clip & 1u, clip & 2u);
      sq32 += q;
      const uint32_t idx = brick_index(x, y, z, g.log2nb);
      pend_old = atomicAdd(&g.word[idx], (q << 16) | 1u);
      const uint32_t r = wcount + __popc(am & lt);
      if (r < room) {
        rec[r] = ((unsigned long long)idx << 32) | ids[j];
        pend_r = r;
      }
    }
    wcount += __popc(am);
  };
  // the voxel's centre seen from v0, and its squared distance to the axis at the
  // nearest point t of the segment
  auto offset = [&](const Seg& S, int x, int y, int z, float3& w, float& t, float3& e) {
    w = make_float3((float)x + 0.5f - S.a.x, (float)y + 0.5f - S.a.y, (float)z + 0.5f - S.a.z);
    t = fminf(1.0f, fmaxf(0.0f, dot3(w, f3(S.d)) * S.a.w));
    e = w - t * f3(S.d);
    return dot3(e, e);
  };
  // stage 2 for queued entries below cnt (all lanes call)
  auto stage2 = [&](uint32_t cnt) {
    int dec = 0, j = 0, x = 0, y = 0, z = 0;
    float3 w = make_float3(0.f, 0.f, 0.f), e;
    float t, e2 = 0.0f;
    float4 n0 = make_float4(0.f, 0.f, 0.f, 0.f);
    if ((uint32_t)lane < cnt) {
      const uint2 it = uq[lane];
      j = (int)it.x;
      unpack_voxel(it.y, x, y, z);
      const Seg& S = segs[j];
      n0 = S.n0;
      e2 = offset(S, x, y, z, w, t, e);
      const float3 la = make_float3(S.a.x - (float)x, S.a.y - (float)y, S.a.z - (float)z);
      dec = g.force_exact ? -1 : seg_box_stage2(la, f3(S.d), g.rl);
      if (dec < 0) ++ex;
    }
    queue_exact(g, dec < 0, ids[j], x, y, z, lane);
    emit(dec > 0, j, n0, w, e2, x, y, z);
  };
  const float rl2x2 = 2.0f * g.rl * g.rl;
  for (uint32_t w0 = 0; w0 < total; w0 += kWindow) {
    const uint32_t w1 = min(total, w0 + kWindow);
    if (w0) {
      __syncwarp();
      fill(w0, w1);
      __syncwarp();
    }
    for (uint32_t t0 = w0; t0 < w1; t0 += 32) {
      const uint32_t gq = t0 + lane;
      int j = 0, x = 0, y = 0, z = 0, dec = 0;
      bool have = gq < w1;
      float3 w = make_float3(0.f, 0.f, 0.f);
      float e2 = 0.0f;
      float4 n0 = make_float4(0.f, 0.f, 0.f, 0.f);
      if (tabled) {
        if (have) {
          const uint32_t own = s_own[wid][gq - w0];
          j = (int)(own & 31u);
          const Seg& S = segs[j];
          n0 = S.n0;
          const uint32_t b = __float_as_uint(n0.w);
          const uint2 bx = S.box[own >> 5];
          const uint32_t rem = gq - __float_as_uint(S.n1.w) - (bx.y & 0xffffu);
          // rem < 256 and a width below 16: exact (rem * (magic * width - 4096) < 4096)
          const uint32_t dj = (rem * (bx.y >> 16)) >> 12;
          place(b & 3u, (int)(((b >> 2) & 1023u) + (own >> 5)), (int)((bx.x & 1023u) + dj),
                (int)(((bx.x >> 10) & 1023u) + rem - dj * (bx.x >> 20)), x, y, z);
        }
      } else {
        // a warp with a long segment: the owner by a binary search over the
        // inclusive prefix of the candidate counts
#pragma unroll
        for (int st = 16; st > 0; st >>= 1)
          if (__shfl_sync(FULLW, incl, j + st - 1) <= gq) j += st;
        j = min(j, 31);
        if (have) {
          const Seg& S = segs[j];
          n0 = S.n0;
          const uint32_t b = __float_as_uint(n0.w), q = gq - __float_as_uint(S.n1.w);
          if (b & (1u << 14)) {
            uint32_t sl = 0;
            while (sl + 1 < (uint32_t)kBoxSlabs && slab_end(S, (int)sl, 0u, 0xffffu) <= q) ++sl;
            const uint2 bx = S.box[sl];
            const uint32_t rem = q - (bx.y & 0xffffu), dj = (rem * (bx.y >> 16)) >> 12;
            place(b & 3u, (int)(((b >> 2) & 1023u) + sl), (int)((bx.x & 1023u) + dj),
                  (int)(((bx.x >> 10) & 1023u) + rem - dj * (bx.x >> 20)), x, y, z);
          } else {
            have = decode_long(S, b, g.n, q, x, y, z);
          }
        }
      }
      if (have) {
        // Stage 1. The axis point p = v0 + t d nearest the voxel's centre lies e
        // from it: the box is within rl of p, so of the segment (accept), or it
        // lies, along e, beyond |e| - |e|_1 / (2 |e|) = u / |e| of p and so, p being
        // the nearest point, of the whole segment (reject when that squared
        // exceeds rl^2 by the allowance), or the pair is undecided.
        const Seg& S = segs[j];
        float t;
        float3 e;
        e2 = offset(S, x, y, z, w, t, e);
        const float fx = fabsf(e.x), fy = fabsf(e.y), fz = fabsf(e.z);
        const float ex_ = fmaxf(fx - 0.5f, 0.0f), ey = fmaxf(fy - 0.5f, 0.0f), ez = fmaxf(fz - 0.5f, 0.0f);
        const float up2 = ex_ * ex_ + ey * ey + ez * ez;
        const float u = fmaf(-0.5f, fx + fy + fz, e2);
        dec = up2 <= S.d.w ? 1 : (u > 0.0f && u * u > (rl2x2 - S.d.w) * e2 ? 0 : -1);
        if (g.force_exact) dec = -1;  // with the test option every pair goes on to the exact path
      }
      const unsigned um = __ballot_sync(FULLW, dec < 0);
      if (dec < 0) uq[un + __popc(um & lt)] = make_uint2((uint32_t)j, pack_voxel(x, y, z));
      un += __popc(um);
      emit(dec > 0, j, n0, w, e2, x, y, z);
      if (un >= 32) {
        __syncwarp();
        stage2(32);
        __syncwarp();
        // entries past the first 32 move to the front (reads 32.., writes ..31)
        if ((uint32_t)lane < un - 32) uq[lane] = uq[32 + lane];
        __syncwarp();
        un -= 32;
      }
    }
    sq += sq32;
    sq32 = 0;
    __syncwarp();
  }
  __syncwarp();
  if (un) stage2(un);
  sq += sq32;
  flush_rank();
  if (lane == 0 && wcount > room) set_err(g.st, kErrOverflow);
  for (uint32_t q = wcount + lane; q < room; q += 32) rec[q] = kNoRecord;  // candidates not kept
  flush_counters_block(g.st, lane == 0 ? (unsigned long long)wcount : 0ull, sq, ex);
}

// Decisions of pass 1's undecided pairs (a few in 100k): in pairs of floats, and
// what those leave (ties, or every pair with the force_exact test option) in
// 128-bit integers. The kept ones take their record slots with one atomic per
// warp. Few and long, so latency bound: a small grid starts soonest.
constexpr int kExactThreads = 128;
__global__ void __launch_bounds__(kExactThreads) k_exact1(const float4* __restrict__ pos,
                                                const float4* __restrict__ nrm, GridDev g) {
  dependency_wait();
  const uint32_t cnt = min(g.st->xq_cnt, g.xq_cap);
  const int lane = threadIdx.x & 31;
  unsigned long long F = 0, sq = 0;
  const unsigned long long step = gridDim.x * blockDim.x;
  for (unsigned long long e0 = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; e0 < cnt; e0 += step) {
    const unsigned long long e = e0 + lane;
    bool keep = false;
    uint32_t seg = 0, idx = 0, rank = 0;
    if (e < cnt) {
      const uint2 it = g.xq[e];
      seg = it.x;
      int x, y, z;
      unpack_voxel(it.y, x, y, z);
      const float4 p0 = pos[seg], p1 = pos[seg + 1];
      const float3 la = make_float3(p0.x - (float)x, p0.y - (float)y, p0.z - (float)z);
      const int dec = g.force_exact ? -1 : seg_box_stage3(la, f3(p1) - f3(p0), g.rl);
      keep = dec < 0 ? seg_exact_at(f3(p0), f3(p1), x, y, z, g.RL) : dec > 0;
      if (keep) {
        idx = brick_index(x, y, z, g.log2nb);
        rank = add_fragment(g, f3(p0), f3(p1), f3(nrm[seg]), f3(nrm[seg + 1]),
                            __float_as_uint(p0.w) & kClipOn, __float_as_uint(p1.w) & kClipOn, x, y, z,
                            F, sq);
      }
    }
    const unsigned km = __ballot_sync(FULLW, keep);
    if (!km) continue;
    unsigned long long r = 0;
    if (lane == 0) r = atomicAdd(&g.st->rec_cnt, (unsigned long long)__popc(km));
    r = __shfl_sync(FULLW, r, 0) + __popc(km & ((1u << lane) - 1u));
    if (keep) {
      if (r < g.rec_cap) {
        g.rec[r] = ((unsigned long long)idx << 32) | seg;
        g.rank[r] = (uint16_t)rank;
      } else {
        set_err(g.st, kErrOverflow);
      }
    }
  }
  unsigned long long z0 = 0;
  flush_counters(g.st, F, sq, z0);
}

__device__ __forceinline__ bool bit_set(const uint32_t* bits, uint32_t i) {
  return (bits[i >> 5] >> (i & 31)) & 1u;
}

// Pass 2: stream the fragment records; mode 0 lists every fragment, mode 1
// those whose voxel the cull marked, mode 2 (repair) those whose voxel's
// `need` bit is set. Modes 0 and 1 read the voxel's list end from the scan's
// cursor -- kCulledStart when the cull gave it no list -- and write the segment
// id at end - 1 - rank: no atomic, and the cursor carries the cull's decision, so the
// mark is not read. The repair, whose copied records carry no rank, bumps the
// cursor of each listed voxel from its list start with a returning atomic.
// Mode 1 also copies the records of unmarked voxels to the (by then unused)
// exact-path queue, warp-staged, so that the repair rounds stream only those;
// when they do not all fit, the repair streams every record. The copy is made
// only when under half of the fragments are culled: past that, a repair round
// streaming every record reads less than twice the bytes the copy would write
// in every frame, and repairs are rare (ABC pathlines at 512^3 cull 97% of their
// fragments and need none); k_scatter_culled lists the fragments of such a
// build instead.
__global__ void __launch_bounds__(256) k_scatter(GridDev g, int mode, const uint32_t* __restrict__ need,
                                                 const uint32_t* __restrict__ pending) {
  const uint32_t zero = dependency_wait();
  if (mode == 2 && pending[zero] == 0) return;
  if (mode != 2 && blockIdx.x == 0 && threadIdx.x < kScanParts) {
    // the scan's counters, and its field sums of the packed words against pass 1's
    // totals: a difference means that a 16-bit field overflowed
    DevStatus* st = g.st;
    const ScanPart p = st->scan_part[threadIdx.x + zero];
    unsigned long long c = p.count_field, o = p.occ_field, v = p.voxels;
    uint32_t mc = p.max_count;
#pragma unroll
    for (int k = kScanParts / 2; k > 0; k >>= 1) {
      c += __shfl_xor_sync((1u << kScanParts) - 1u, c, k);
      o += __shfl_xor_sync((1u << kScanParts) - 1u, o, k);
      v += __shfl_xor_sync((1u << kScanParts) - 1u, v, k);
      mc = max(mc, __shfl_xor_sync((1u << kScanParts) - 1u, mc, k));
    }
    if (threadIdx.x == 0) {
      st->sum_count_field = c;
      st->sum_occ_field = o;
      st->occupied_voxels = (uint32_t)v;
      st->visible_voxels = (uint32_t)(v >> 32);
      st->max_count = mc;
      if (c != st->F || o != st->sum_q) set_err(st, kErrOverflow);
    }
  }
  __shared__ unsigned long long s_rec[8][kWarpRecords];
  unsigned long long* cq = reinterpret_cast<unsigned long long*>(g.xq);
  bool copy = false;  // mode 1: copy the culled records (grid-uniform)
  if (mode == 1) {
    const unsigned long long F = g.st->F, culled = F - g.st->list_tail;
    copy = 2 * culled < F;
    if (!copy) return;  // k_scatter_culled's build
  }
  const bool compact = mode == 2 && g.st->cq_cnt != kNoCopy && g.st->cq_cnt <= g.xq_cap;
  const unsigned long long* src = compact ? cq : g.rec;
  const unsigned long long cnt =
      compact ? g.st->cq_cnt : min(g.st->rec_cnt, (unsigned long long)g.rec_cap);
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  unsigned long long* srec = s_rec[threadIdx.x >> 5];
  int wcount = 0;  // culled records staged by this warp (mode 1, uniform)
  unsigned long long listed = 0;
  const uint32_t warp = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) + zero;
  const uint32_t n_warps = (gridDim.x * blockDim.x) >> 5;
  for (unsigned long long e0 = warp * 32ull; e0 < cnt; e0 += n_warps * 32ull) {
    const unsigned long long e = e0 + lane;
    bool skip = true, have = false;
    unsigned long long r = 0;
    uint32_t rank = 0;
    if (e < cnt) {
      r = __ldcs(&src[e]);
      if (mode != 2) rank = __ldcs(&g.rank[e]);
    }
    if (e < cnt && r != kNoRecord) {
      have = true;
      const uint32_t idx = (uint32_t)(r >> 32);
      uint32_t slot = 0;
      if (mode != 2) {
        const uint32_t end = __ldg(&g.cur[idx]);
        skip = end >= kCulledStart;
        slot = end - 1u - rank;
      } else {
        skip = !bit_set(need, idx);
        if (!skip) slot = atomicAdd(&g.cur[idx], 1u);
      }
      if (!skip) {
        if (slot < g.list_cap) {
          g.lists[slot] = (uint32_t)r;
          ++listed;
        } else {
          set_err(g.st, kErrOverflow);
        }
      }
    }
    if (copy) {
      const bool keep = have && skip;
      const unsigned km = __ballot_sync(FULLW, keep);
      if (keep) srec[wcount + __popc(km & lt)] = r;
      wcount += __popc(km);
      if (wcount > kWarpRecords - 32) {
        __syncwarp();
        flush_culled(g, cq, srec, wcount, lane);
        wcount = 0;
      }
    }
  }
  if (copy) {
    __syncwarp();
    flush_culled(g, cq, srec, wcount, lane);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) listed += __shfl_down_sync(FULLW, listed, o);
  if (lane == 0 && listed) atomicAdd(&g.st->listed, listed);
}

// Pass 2 (mode 1) of a build whose cull dropped at least half of the
// fragments, which k_scatter leaves to it: no culled-record copy, and mostly
// reads, so a warp takes 4 x 32 consecutive records per round, each lane one
// of every 32, and loads the lane's four records, then their list ends,
// together -- four independent load chains in flight per lane (ABC pathlines
// at 512^3: pass 2 0.71 -> 0.47 ms; where most fragments are listed, four
// rounds' scattered list stores at once measured slower: bundles 0.90 -> 1.11).
__global__ void __launch_bounds__(256) k_scatter_culled(GridDev g) {
  const uint32_t zero = dependency_wait();
  const unsigned long long F = g.st->F;
  if (2 * (F - g.st->list_tail) < F) return;  // k_scatter's build
  if (blockIdx.x == 0 && threadIdx.x == 0) g.st->cq_cnt = kNoCopy;
  const unsigned long long cnt = min(g.st->rec_cnt, (unsigned long long)g.rec_cap);
  constexpr int U = 4;
  const int lane = threadIdx.x & 31;
  const uint32_t warp = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) + zero;
  const uint32_t n_warps = (gridDim.x * blockDim.x) >> 5;
  unsigned long long listed = 0;
  for (unsigned long long e0 = warp * (32ull * U); e0 < cnt; e0 += n_warps * (32ull * U)) {
    unsigned long long r[U];
    uint32_t rank[U], end[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const unsigned long long e = e0 + 32ull * u + lane;
      r[u] = e < cnt ? __ldcs(&g.rec[e]) : kNoRecord;
      rank[u] = e < cnt ? (uint32_t)__ldcs(&g.rank[e]) : 0u;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      end[u] = r[u] != kNoRecord ? __ldg(&g.cur[(uint32_t)(r[u] >> 32)]) : kCulledStart;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (end[u] >= kCulledStart) continue;  // no record, or the cull gave its voxel no list
      const uint32_t slot = end[u] - 1u - rank[u];
      if (slot < g.list_cap) {
        g.lists[slot] = (uint32_t)r[u];
        ++listed;
      } else {
        set_err(g.st, kErrOverflow);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) listed += __shfl_down_sync(FULLW, listed, o);
  if (lane == 0 && listed) atomicAdd(&g.st->listed, listed);
}

int launch_pass1(const float4* pos, const float4* nrm, const uint32_t* order, long long V,
                 const GridDev& g, const Queue& q) {
  if (V < 2) return 0;
  // One atomic per fragment at every grid side: summing the increments of the
  // lanes of a warp step that share a voxel first (a match on the voxel index)
  // measured slower at 256^3 (bundles pass 1 2.3 -> 3.5 ms) and, since pass 1's
  // atomics return the rank, at 512^3 too (ABC pathlines 4.70 -> 6.83 ms; it
  // paid there while they returned nothing, 7.8 -> 7.4 ms).
  const int spw = pass1_segments_per_warp(V);
  const long long per_block = (long long)spw * kPass1Warps;
  launch(k_pass1, (unsigned)((V + per_block - 1) / per_block), kPass1Threads, q, pos, nrm, order, V,
                 spw, g);
  launch(k_exact1, kSms * 2, kExactThreads, q, pos, nrm, g);
  return 2;
}

int launch_scatter(const GridDev& g, int mode, const uint32_t* need, const uint32_t* pending,
                   const Queue& q) {
  if (mode == 1) launch(k_scatter_culled, kSms * 8, 256, q, g);
  launch(k_scatter, kSms * 8, 256, q, g, mode, need, pending);
  return mode == 1 ? 2 : 1;
}

}  // namespace vrt
