// Host-side launch wrappers of the libvrt kernels (one translation unit each).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "vrt.h"
#include "vrt_internal.cuh"

namespace vrt {

// Where kernels are launched: a stream, and whether each may start while the one
// before it drains (launch).
struct Queue {
  cudaStream_t s;
  bool chained;
};

// The streams of the process's grids and servers. Launches are chained only while
// there is one: with frames of 128^3 to 512^3 sets on four streams at once, all
// chained, a run of the serving workload was seen to stop with the GPU busy, and
// reading showed no reason in the kernels (their waits and loops end), so chained
// launches and several streams do not meet. A grid enters the stream it takes and
// leaves it for the next; a server enters all of its streams while it lives.
void stream_enter(cudaStream_t s);
void stream_leave(cudaStream_t s);
// Whether no other stream than s is entered.
bool stream_alone(cudaStream_t s);

// Launches `kernel`; chained, so that it may start while the kernel before it on
// the stream drains: its blocks are resident, waiting in dependency_wait(), when that
// one completes, which saves most of a launch's latency (a frame of a small set is a
// chain of 11 to 33 kernels of a few microseconds). Every kernel launched here
// calls dependency_wait() before it touches memory. After a copy, a memset or
// an event the stream orders it as usual.
template <class... P, class... A>
void launch(void (*kernel)(P...), dim3 grid, unsigned threads, const Queue& q, A... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = dim3(threads);
  c.stream = q.s;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = q.chained ? 1 : 0;
  cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

// Camera as given through the C ABI, widened to fp64 on the host.
struct HostCamera {
  int width, height, ortho;
  double eye[3], target[3], up[3], fovy_deg, ortho_h;
};

// Camera in the form the trace kernel consumes (built on the host in fp64).
struct CamDev {
  float3 o0, ox, oy;  // origin: o0 (+ (px+.5) ox + (py+.5) oy when orthographic)
  float3 d0, dx, dy;  // direction: d0 + (px+.5) dx + (py+.5) dy, normalised
  int width, height, ortho;
};

struct TraceArgs {
  GridDev g;
  CamDev cam;
  const float4* pos;
  const float4* nrm;
  uint32_t n_vert;           // vertices; list entries must be < n_vert - 1
  float alpha;
  int ao;                    // per-hit shading: 0 none, 1 cone AO, 2 voxel-space field
  const void* mips;          // occupancy pyramid, texels in format mips_fmt
  int mips_fmt;              // kMipsF32, kMipsF16 or kMipsBF16
  long long lev_off[11];
  int n_levels;
  float4* rgba;
  int* first_id;
  float* first_t;
  const uint32_t* pix_list;  // trace only these pixels (repair) when non-null
  const uint32_t* pix_count; // number of entries of pix_list (device)
  uint32_t* need;            // [n^3 / 32] voxels queued for listing
  uint32_t* vq;              // out: queued voxels
  uint32_t* vq_cnt;
  uint32_t* pq;              // out: pixels to trace again
  uint32_t* pq_cnt;
  uint32_t vq_cap, pq_cap;
  uint32_t max_queue;        // culled voxels one ray may queue before it stops
  uint32_t* work_next;       // next work item (persistent warps)
  float4* resume;            // [2 * pixels] state of a ray at its first culled voxel:
                             // (C, T), (first id bits, first t, voxel index bits, entry t)
  uint32_t short_list;       // lists up to this length share the warp entry by entry
  uint32_t ray_keys;         // hits a transparent ray may have on that path
  int key16;                 // order hits by the paper's 16+16-bit per-voxel key
  int tile_w;                // warp tile width (2, 4, 8 or 16 pixels)
  int tile_n;                // rays a warp of the main trace owns (launch_trace sets it)
  uint32_t max_calls;        // walk calls after which a ray is given up (0: the
                             // grid's limit; launch_trace shifts it to Ray::calls' place)
  int count;                 // accumulate trace work counters
  uint32_t* touch_list;      // instrumented trace: bit per list entry read
  uint32_t* touch_vert;      //   bit per vertex read (segment end points)
  uint32_t* touch_vox;       //   bit per voxel whose words the DDA read
  const float* shade;        // voxel-space shading field [n^3] (brick order), or null
};

// Voxel-space shading (Sec. 3.4, Shading): per voxel, cone AO at its centre
// times 1/2 + 1/2 * the transmittance of a ray toward the light through the
// base occupancy level, for every voxel within one step (26-neighbourhood) of a
// listed voxel -- the voxels whose centres a trilinear sample at a hit reads.
struct ShadeArgs {
  GridDev g;
  const void* mips;          // occupancy pyramid (format mips_fmt)
  int mips_fmt;
  long long lev_off[11];
  int n_levels;
  int ao;                    // 1: include the cone AO
  float lx, ly, lz;          // unit direction toward the light
  float* shade;              // [n^3] shading value per voxel (brick order)
  uint32_t* mask;            // [n^3 / 32] voxels whose value is current this frame
  const uint32_t* vq;        // repair: voxels listed in this round
  const uint32_t* vq_cnt;
  uint32_t vq_cap;
};
// Every voxel next to a listed one (one block per brick); rewrites the mask.
int launch_shade(const ShadeArgs& a, const Queue& q);
// Zeroes up to two ranges of 32-bit words.
int launch_reset(uint32_t* a, uint32_t na, uint32_t* b, uint32_t nb, const Queue& q);
// Voxels next to the voxels a repair round listed, not yet shaded this frame.
int launch_shade_repair(const ShadeArgs& a, const Queue& q);

// Ingest of vertices [lo, hi) (nothing when hi <= lo).
int launch_ingest(const float* raw, const uint8_t* flags, long long lo, long long hi, float4* pos,
                  float4* nrm, DevStatus* st, const Queue& q);
constexpr int kPass1Threads = 128;
constexpr int kPass1Blocks = 9;  // resident per SM: 56 registers, 24 KB of shared memory
// Segments a warp of pass 1 takes, of a set of V vertices. They are a serial chain
// of steps over their candidates, and a step takes 32 candidates whatever their
// segments, so a small set is spread over more warps: 4.5k segments of 57
// fragments each 0.105 ms with 32 segments a warp, 0.056 with 8, 0.046 with 4; 20k
// of 7 0.050, 0.046, 0.048; at 98k it no longer pays (0.044 with 32, 0.047 with 16).
inline int pass1_segments_per_warp(long long V) {
  int n = 32;
  while (n > 4 && V / n < (long long)kSms * kPass1Blocks) n >>= 1;
  return n;
}
// Fragment records held for a list capacity of `cap` entries. Pass 1 takes record
// slots for candidates, warp by warp; a small set's warps take fewer segments, so
// more of the unused slots fall inside the capacity: room for them.
inline unsigned long long record_capacity(unsigned long long cap, long long V) {
  return cap + (pass1_segments_per_warp(V) < 32 ? std::min<unsigned long long>(4ull * cap, 1ull << 20) : 0ull);
}
// Pass 1 over the segments in the order `order` (V vertex indices, each
// polyline's vertices consecutive; a polyline's last vertex starts no
// segment), or in index order when `order` is null.
int launch_pass1(const float4* pos, const float4* nrm, const uint32_t* order, long long V,
                 const GridDev& g, const Queue& q);
// 12-bit spatial keys (Morton code of the 16^3 cell) of the vertices mid[0..P).
int launch_poly_keys(const float* raw, const uint32_t* mid, uint32_t P, int n, uint16_t* key,
                     cudaStream_t s);
// Occupancy masks and empty-brick distance field from the counts of pass 1
// (tmp: one byte per brick).
int launch_brick_dist(const GridDev& g, uint8_t* tmp, uint8_t* dist, uint2* mask, const Queue& q);
// The three distance passes from per-brick bytes in tmp (0 = occupied, else
// kBrickDistMax); tmp is overwritten.
int launch_brick_dist_passes(int log2nb, uint8_t* tmp, uint8_t* dist, const Queue& q);
// Pass 2 over the fragment records. mode 0: every occupied voxel has a list;
// 1: voxels marked by the cull; 2: repair, only voxels whose `need` bit is set
// (skipped when *pending is 0).
int launch_scatter(const GridDev& g, int mode, const uint32_t* need, const uint32_t* pending,
                   const Queue& q);
// stall_tile >= 0 (testing): that tile never publishes its look-back state,
// so the tiles after it give up their waits after spin_limit polls.
int launch_scan(const GridDev& g, int all_visible, unsigned long long* tile_state, uint32_t n_tiles,
                int stall_tile, int spin_limit, const Queue& q);
int launch_mips(const GridDev& g, void* mips, int fmt, const long long* lev_off, int n_levels,
                const Queue& q);
// Cull marks; btmp, cdist: one byte per brick (scratch; distance to a brick
// with eroded occupancy); emean: one float per brick (mean eroded occupancy);
// depth_max: estimated optical depth past which a voxel is culled (<= 0: the
// default, ln(1e4) + 3); occq: scratch for the indices of the occupied voxels
// (occq_cap entries; when fewer than n^3, every voxel's thread tests its own).
int launch_cull(const GridDev& g, const HostCamera& cam, float alpha, uint8_t* eroded,
                uint8_t* btmp, uint8_t* cdist, float* emean, float depth_max, uint32_t* occq,
                unsigned long long occq_cap, const Queue& q);
constexpr int kTraceThreads = 128;
// Rays a warp's tile of the transparent trace holds, of an image of npx pixels: 32
// in a shape of the caller's (TraceArgs::tile_w), fewer in a fixed one. A small
// image's tiles shrink until there are warps enough to fill the GPU (5 blocks an SM):
// a tile is a serial chain of rounds, and its units of work are entries, not
// rays, so few rays still fill a warp's lanes (157x93 pixels at alpha 0.1:
// 0.75 ms with 32 rays a tile, 0.46 with 16, 0.31 with 8, 0.22 with 4;
// where tiles of 32 fill the GPU, 16 cost a third more).
inline int transparent_tile_rays(long long npx) {
  int n = 32;
  while (n > 4 && npx / n < (long long)kSms * 5 * (kTraceThreads / 32)) n >>= 1;
  return n;
}
int launch_trace(const TraceArgs& a, int K, const Queue& q);
// Cone AO of the hits an opaque trace (K = 1, a.ao = 1) and its repair rounds
// left in a.rgba.
int launch_shade_hits(const TraceArgs& a, const Queue& q);
// Instrumented trace: the set bits of the three touch bitmaps into
// st->tr_u_entries, tr_u_vertices, tr_u_voxels (which the caller cleared).
int launch_touch_count(const uint32_t* list_bits, size_t list_words, const uint32_t* vert_bits,
                       size_t vert_words, const uint32_t* vox_bits, size_t vox_words,
                       DevStatus* st, const Queue& q);
// Repair round: list the voxels of vq (count *vq_cnt), pass 2 restricted to
// them, then clear their `need` bits and the next round's queue counters.
int launch_repair_alloc(const GridDev& g, const uint32_t* vq, const uint32_t* vq_cnt,
                        const uint32_t* pq_cnt, uint32_t vq_cap, const Queue& q);
int launch_repair_clear(const GridDev& g, uint32_t* need, const uint32_t* vq,
                         const uint32_t* vq_cnt, uint32_t vq_cap, int next, const Queue& q);

// Host-side checks shared by the C ABI and the serving loop: nullptr when the
// camera and render parameters are acceptable to vrt_cull and vrt_trace, else
// what is wrong.
const char* frame_args_error(const vrt_camera* cam, const vrt_render_params* p);

// Allocate every buffer a frame of `g` with these parameters sizes lazily, so
// that the frame's calls allocate nothing and can be captured into a CUDA
// graph (may synchronize the grid's stream).
vrt_status prepare_frame(vrt_grid g, const vrt_camera* cam, const vrt_render_params* p);
// Estimated device bytes of a grid of this side with n_vertices vertices, segments of
// mean length mean_len, and every buffer its frames can need.
uint64_t set_bytes(int side, float radius, uint64_t max_fragments, int64_t n_vertices, double mean_len);

// Testing hook of vrt_scan_counts_noalloc (vrt_set_option(NULL,
// VRT_OPT_TEST_SCAN_STALL, tile)): tile >= 0 makes that look-back tile skip
// its publish and shortens every wait; -1 restores the normal scan.
void set_noalloc_scan_stall(long long tile);

constexpr int kSpinLimitTest = 1 << 10;  // look-back polls while a test stalls a tile

}  // namespace vrt
