// Launchers of the ray-casting kernels (kernels.cu).
#pragma once

#include <cuda_runtime.h>

#include "fgl.h"
#include "fgl_internal.h"

namespace fgl {

// Dynamic shared memory of one block: a 64-bit hit key per thread plus the
// shared part of the traversal stacks.
size_t stack_smem_bytes(int W, int block, int sdepth);

// How a cast walks the tree: packets of this many consecutive rays of an
// environment a warp, together (16 or 32), or each ray for itself (0).  By what the
// sensor's packets are like (see sensor_packets), the scene's walk cost and the
// rays; the figures are shares of the time ray by ray, over sensors of 4 to 128
// beams and 91 to 2048 columns, rooms with one object (108 to 2,796 triangles, cost
// 5-6) to cluttered ones (300 to 1 M, 7-60) and 1,000 to 13 M rays:
//   close  0.55-0.95 from 400 k rays on in any scene; below, 0.7-1.1, but 1.0-1.4 in
//          rooms of cost 5, whose walks have little to share
//   fair   0.85-1.03 from 400 k rays on, 0.95-1.1 from 68 k to 220 k
//   narrow 0.9-1.1 from 400 k rays on, 1.0-1.25 from 68 k to 220 k
// Packets of 16 leave half of the lanes idle, but one ends sooner, which counts when
// they come to at most two for each of the 28 warps an SM holds (1 M triangles,
// 57,600 rays 42 -> 35 us, 131,072 51 -> 44; 184,320 would take 82 instead of 75).
// Fair ones gain (0.8-1.1) up to half as many rays, narrow ones (0.85-1.1) a quarter.
constexpr int64_t kSmallCastRays = 16 * 2 * 28 * 152;
inline bool small_cast(int64_t rays) { return rays <= kSmallCastRays; }

enum SensorPackets { kSpreadPackets = 0, kNarrowPackets = 1, kFairPackets = 2, kClosePackets = 3 };

// A tree's expected node visits and triangle tests (SAH), as of an 8-wide one.
inline float walk_cost(const HostBVH& b) { return (float)(b.width == 8 ? b.sah_cost : 0.8 * b.sah_cost); }

inline int cast_packets(int sensor, float cost, int64_t rays) {
  switch (sensor) {
    case kClosePackets:
      return cost < 5.5f && rays < (1 << 19) ? 0 : small_cast(rays) ? 16 : 32;
    case kFairPackets:
      return rays >= (1 << 18) ? (cost < 5.5f && rays < (1 << 19) ? 0 : 32)
                               : cost >= 5.5f && 2 * rays <= kSmallCastRays ? 16 : 0;
    case kNarrowPackets:
      return cost >= 7.f && 4 * rays <= kSmallCastRays ? 16 : 0;
    default:
      return 0;
  }
}

// The same for a batch, whose rays go through one launch.  Its other kernel hands
// fresh rays to idle lanes, which a walk in packets has to make up for, and draws
// packets one by one, which bounds it where walks are short and rays many: packets
// take 0.65-0.95 of its time from 5 M rays on, 0.75-1.05 up to 400 k, and between
// 0.75-1.05 at a cost of 8 and more (narrow ones 0.85-1.05 at 9.5), 1.0-1.2 below.
// Packets of 16 up to one a warp slot (65,536 rays 0.8-0.9, packets of 32 0.85-1.0;
// 130,000 rays 0.9-1.1 and 0.8-0.95).
inline bool batch_packets(int sensor, float cost, int64_t rays) {
  if (sensor == kSpreadPackets) return false;
  return rays <= (1 << 19) || rays >= (1 << 22) || cost >= (sensor == kNarrowPackets ? 9.5f : 8.f);
}
inline int batch_packet_rays(int64_t rays) { return 2 * rays <= kSmallCastRays ? 16 : 32; }

// The same over a GPU-built LBVH, whose other kernel walks the binary tree ray by
// ray: close and fair packets 0.4-1.0 of its time (tiny scenes up to 1.1 from 2 M
// rays on), narrow ones 0.5-1.0 up to 220 k rays, 0.9-1.3 from 800 k on.
inline int lbvh_packets(int sensor, int64_t n_tris, int64_t rays) {
  if (sensor == kSpreadPackets) return 0;
  if (sensor == kNarrowPackets) return 2 * rays <= kSmallCastRays ? 16 : rays <= (1 << 18) ? 32 : 0;
  if (n_tris < 2048 && rays > (1 << 20)) return 0;
  return small_cast(rays) ? 16 : 32;
}

// One launch over one item: a thread per ray (packet_rays 0) or a warp per packet
// of packet_rays rays, walked together before the per-ray traversal (needs
// tri_mode 0; see packets_fit).
// tri_mode 0: warp-pooled leaf tests; 1: lane-serial with postponing.
// tmin honours it.min_range (8-wide packets, not counted); status: the word that
// takes traversal errors (null: the shared one).
cudaError_t launch_plain(int W, bool count, int packet_rays, bool tmin, const ItemDesc& it, unsigned* status, int block,
                         int sdepth, int tri_mode, int postpone_pct, cudaStream_t s);

// Whether a block of this shape has room for the packet lists beside its
// stacks (large blocks with deep shared stacks do not).
bool packets_fit(int W, int block, int sdepth);

// Resident blocks per SM of the persistent kernel for this configuration.
int persistent_blocks_per_sm(int W, bool count, bool tmin, bool packets, int block, int sdepth);

// Persistent kernel over the work queue in `scratch`: a BatchHeader
// followed by n_items ItemDesc records (device memory).  tmin selects the
// instantiation that honours ItemDesc::min_range (needed when any item of
// the group has min_range > 0; otherwise min_range is taken as 0).  packets
// selects the kernel whose warps walk whole packets together (the group's
// sensors have narrow packets, tri_mode 0, refill 32).
cudaError_t launch_persistent(int W, bool count, bool tmin, bool packets, void* scratch, int grid, int block,
                              int sdepth, int refill_min, int tri_mode, int postpone_pct,
                              cudaStream_t s);

// Instance pass (see InstancePass in fgl_internal.h): one launch per item
// and instance, after the scene pass.
// All instances of an item in one launch (same width, at most kMaxFusedInstances).
cudaError_t launch_instances_fused(const InstanceSet& a, bool tmin, int block, int sdepth,
                                   cudaStream_t s);
cudaError_t launch_instance_pass(const InstancePass& a, bool tmin, int block, int sdepth,
                                 cudaStream_t s);

// World-frame return points of one item, after its scene and instance passes.
cudaError_t launch_points(const ItemDesc& it, float* out, cudaStream_t s);

// One-thread-per-ray cast over a GPU-built triangle LBVH's binary tree; the wide
// form as an item (sensor, poses, ranges and outputs to be filled in) and the
// LBVH's own status word (lbvh.cu).
cudaError_t launch_lbvh_cast(const fgl_lbvh_s* L, const void* dirs, const float* poses, int n_env,
                             int n_rays, float min_range, float max_range, float* out_range,
                             int32_t* out_tri, cudaStream_t s);
ItemDesc lbvh_item(const fgl_lbvh_s* L);
unsigned* lbvh_status(const fgl_lbvh_s* L);
bool lbvh_built(const fgl_lbvh_s* L);  // false after a build that failed: nothing to cast or export

// Debug export of world rays (beam order).
cudaError_t launch_l2_read(const void* buf, int64_t bytes, int reps, unsigned* sink, int sms,
                           cudaStream_t s);
cudaError_t launch_world_rays(const void* dirs, const float* poses, int n_env, int n_rays,
                              float* out_o, float* out_d, cudaStream_t s);

// Device-side error word (bit 0: traversal stack overflow) and work counters.
cudaError_t read_and_clear_status(unsigned* st);
cudaError_t read_and_clear_counters(unsigned long long* c);  // kWorkCounters values

}  // namespace fgl
