// Kernels and their launchers.
//
//   k_plain      : one thread per ray of a single (scene, sensor, poses) item
//                  -- the paper's "one thread per beam" form (Sec. IV-C).
//   k_persistent : a grid of (SM count x resident blocks) that drains a device
//                  work queue of ray packets spanning many items; a warp
//                  pulls a new packet when its current one is used up, and
//                  hands fresh rays to lanes whose ray has finished once
//                  enough lanes are idle, so warps stay full while the
//                  per-ray work (eq. cost(r_j)) varies.
//   k_plain_packets, k_packets : the same two for sensors of narrow packets
//                  (32 neighbouring rays of one environment): a warp walks
//                  the upper tree with all its rays together (packet_phase in
//                  trace.cuh) and only what is left ray by ray.
//   k_world_rays : debug export of the float32 rays of eq. r_j.
//   k_l2_read    : bandwidth probe, 16-byte L2 reads of a resident buffer.
#include <cuda_runtime.h>

#include "kernels.h"
#include "trace.cuh"

namespace fgl {

__device__ unsigned int g_status;  // bit 0: stack overflow; bit 1: item of another width
// count_work counters: rays, node visits, triangle tests, then the batched
// kernel's phases -- warp iterations of its main loop, active lanes summed
// over those iterations, pooled leaf-test rounds, stack entries popped by
// finish(), and refill passes (one per new ray packet a warp draws from)
__device__ unsigned long long g_counters[kWorkCounters];

namespace {

template <bool COUNT>
__device__ __forceinline__ void flush_counters(const uint32_t (&c)[kWorkCounters]) {
  if (!COUNT) return;
  const unsigned full = __activemask();
#pragma unroll
  for (int k = 0; k < kWorkCounters; ++k) {
    const unsigned long long v = __reduce_add_sync(full, c[k]);
    if ((threadIdx.x & 31) == (__ffs(full) - 1) && v) atomicAdd(&g_counters[k], v);
  }
}

__device__ __forceinline__ int postpone_threshold(int pct) {
  if (pct <= 0) return 0;
  return (__popc(__activemask()) * pct + 99) / 100;
}

// Dynamic shared memory: one 64-bit hit key per thread (pooled leaf tests
// merge into these), then the [sdepth][blockDim] stack arrays of groups
// (8 B) and of child keys (2 B per child).
template <int W>
struct Smem {
  using Keys = typename dev::KeyWords<W>::T;
  unsigned long long* keys;  // this warp's 32 hit keys
  uint2* ss;                 // this thread's group column
  Keys* sq;                  // this thread's child-key column
};
template <int W>
__device__ __forceinline__ Smem<W> smem_layout(int sdepth) {
  extern __shared__ __align__(16) unsigned long long smem_u64[];
  Smem<W> m;
  m.keys = smem_u64 + (threadIdx.x & ~31u);
  uint2* ss0 = reinterpret_cast<uint2*>(smem_u64 + blockDim.x);
  m.ss = ss0 + threadIdx.x;
  m.sq = reinterpret_cast<typename Smem<W>::Keys*>(ss0 + (size_t)sdepth * blockDim.x) + threadIdx.x;
  return m;
}

template <int W, bool COUNT>
__global__ void __maxnreg__(72) k_plain(const ItemDesc it, int sdepth, int tri_mode, int postpone_pct,
                                        unsigned* status) {
  using Keys = typename dev::KeyWords<W>::T;
  const unsigned FULL = 0xFFFFFFFFu;
  const Smem<W> sm = smem_layout<W>(sdepth);
  const int lane = threadIdx.x & 31;
  if (status == nullptr) status = &g_status;
  if (it.width != W) {  // never read nodes laid out for another width
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(status, 2u);
    return;
  }
  const int64_t total = (int64_t)it.n_env * it.n_rays;
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool done = gid >= total;
  int env = 0;
  float4 ds = make_float4(0.f, 0.f, 0.f, 0.f);
  dev::Tracer<W, COUNT> tr;
  tr.tg = make_uint2(0u, 0u);
  tr.ng = make_uint2(0u, 0u);
  if (COUNT) tr.n_nodes = tr.n_tris = tr.n_rounds = tr.n_pops = 0;
  if (!done) {
    env = (int)(gid / it.n_rays);
    const int j = (int)(gid - (int64_t)env * it.n_rays);
    ds = __ldg((const float4*)it.dirs + j);
    float ox, oy, oz, dx, dy, dz;
    dev::world_ray(it.poses + 12 * (int64_t)env, ds, ox, oy, oz, dx, dy, dz);
    dev::setup_ray(tr.r, ox, oy, oz, dx, dy, dz);
    tr.start(it.nodes, it.tris, it.min_range, it.max_range, it.n_nodes, it.n_tris);
  }
  uint2 ls[kStackLocal];
  Keys lq[kStackLocal];
  const dev::StackRefs<Keys> st{sm.ss, sm.sq, ls, lq, (int)blockDim.x, sdepth};
  if (tri_mode != 1) {
    while (__any_sync(FULL, !done)) {
      bool ok = true;
      if (!done) ok = tr.descend(st);
      dev::tri_phase_warp(tr, sm.keys, lane, status);
      if (!done) {
        if (!ok) {
          atomicOr(status, tr.fail_bits());
          done = true;
        } else {
          done = tr.finish_pooled(st);
        }
      }
    }
  } else if (!done) {
    for (;;) {
      const int pl = postpone_threshold(postpone_pct);
      if (tr.step(st, pl, status)) break;
    }
  }
  if (gid < total) {
    float rg;
    int32_t id;
    tr.result(rg, id);
    const int64_t o = (int64_t)env * it.n_rays + __float_as_int(ds.w);
    __stcs(it.out_range + o, rg);  // results are read by the host, not again here:
    __stcs(it.out_tri + o, id);     // evict-first, so they do not push the BVH out of L2
  }
  if (COUNT) {
    const uint32_t c[kWorkCounters] = {gid < total ? 1u : 0u, tr.n_nodes, tr.n_tris, 0u, 0u,
                                       tr.n_rounds, tr.n_pops, 0u};
    flush_counters<COUNT>(c);
  }
}

// Store a parked result (range bits << 32 | id) of a batched item; evict-first,
// so the results do not push the BVH out of L2.
__device__ __forceinline__ void store_parked(const ItemDesc& it, int64_t o, unsigned long long k) {
  __stcs(it.out_range + o, __uint_as_float((uint32_t)(k >> 32)));
  __stcs(it.out_tri + o, (int32_t)(uint32_t)k);
}

template <int W, bool COUNT, bool TMIN>
__global__ void __maxnreg__(TMIN ? 72 : 64) k_persistent(BatchHeader* __restrict__ hdr,
                                                    const ItemDesc* __restrict__ items, int sdepth,
                                                    int refill_min, int tri_mode, int postpone_pct) {
  using Keys = typename dev::KeyWords<W>::T;
  const unsigned FULL = 0xFFFFFFFFu;
  const Smem<W> sm = smem_layout<W>(sdepth);
  const int lane = threadIdx.x & 31;
  uint2 ls[kStackLocal];
  Keys lq[kStackLocal];
  const dev::StackRefs<Keys> st{sm.ss, sm.sq, ls, lq, (int)blockDim.x, sdepth};

  // The warp's packet cursor (item, environment, next ray, end ray) and its
  // drained flag live in shared memory between refills, and the batch header
  // is re-read at refill time: registers stay free for the traversal (the
  // kernel runs under a 64-register cap, eight 128-thread blocks an SM; the
  // t_min form keeps 72, where 64 would spill).
  __shared__ int4 s_cur[kMaxBlockWarps];
  __shared__ int s_drained[kMaxBlockWarps];
  const int wid = threadIdx.x >> 5;
  if (lane == 0) {
    s_cur[wid] = make_int4(0, 0, 0, 0);
    s_drained[wid] = 0;
  }
  __syncwarp();
  // lane state
  dev::Tracer<W, COUNT, TMIN> tr;
  tr.tg = make_uint2(0u, 0u);
  tr.ng = make_uint2(0u, 0u);
  if (COUNT) tr.n_nodes = tr.n_tris = tr.n_rounds = tr.n_pops = 0;
  bool active = false;
  // A finished lane parks its (range, id) in its own hit-key slot, which the
  // pooled leaf tests never touch while the lane is idle, and the idle lanes
  // store their parked results together at the next refill (or at exit): the
  // stores of a packet then coalesce into whole sectors, which matters most
  // when the outputs are page-locked host memory.
  bool parked = false;
  int out_item = 0;    // the lane's ray: its item and output offset
  int64_t out_o = 0;
  uint32_t c_rays = 0, c_nodes = 0, c_tris = 0, c_iters = 0, c_lane_iters = 0, c_refills = 0;

  for (;;) {
    unsigned idle = __ballot_sync(FULL, !active);
    if ((idle == FULL || __popc(idle) >= refill_min) && !s_drained[wid]) {
      if (parked) {
        store_parked(items[out_item], out_o, sm.keys[lane]);
        parked = false;
      }
      const int64_t n_packets = hdr->n_packets;
      const int n_items = hdr->n_items;
      const int P = hdr->packet_rays;
      int4 cur = s_cur[wid];
      int& pk_item = cur.x;
      int& pk_env = cur.y;
      int& pk_next = cur.z;
      int& pk_end = cur.w;
      bool drained = false;
      while (idle) {
        if (pk_next >= pk_end) {
          unsigned long long p = 0;
          if (lane == 0) p = atomicAdd(&hdr->head, 1ull);
          p = __shfl_sync(FULL, p, 0);
          if ((int64_t)p >= n_packets) {
            drained = true;
            break;
          }
          int lo = 0, hi = n_items - 1;
          while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (items[mid].pk_begin <= (int64_t)p) lo = mid;
            else hi = mid - 1;
          }
          const int64_t local = (int64_t)p - items[lo].pk_begin;
          const int ppe = items[lo].pk_per_env;
          pk_item = lo;
          pk_env = (int)(local / ppe);
          const int chunk = (int)(local - (int64_t)pk_env * ppe);
          pk_next = chunk * P;
          pk_end = min(pk_next + P, items[lo].n_rays);
          if (COUNT && lane == 0) ++c_refills;
        }
        if (items[pk_item].width != W) {  // never read nodes laid out for another width
          if (lane == 0) atomicOr(&g_status, 2u);
          pk_next = pk_end;
          continue;
        }
        const int avail = pk_end - pk_next;
        const int rank = __popc(idle & ((1u << lane) - 1u));
        if (((idle >> lane) & 1u) && rank < avail) {
          const ItemDesc& it = items[pk_item];
          const float4 ds = __ldg((const float4*)it.dirs + pk_next + rank);
          float ox, oy, oz, dx, dy, dz;
          dev::world_ray(it.poses + 12 * (int64_t)pk_env, ds, ox, oy, oz, dx, dy, dz);
          dev::setup_ray(tr.r, ox, oy, oz, dx, dy, dz);
          if (COUNT) {
            c_nodes += tr.n_nodes;
            c_tris += tr.n_tris;
            tr.n_nodes = tr.n_tris = 0;
          }
          tr.start(it.nodes, it.tris, it.min_range, it.max_range, it.n_nodes, it.n_tris);
          out_o = (int64_t)pk_env * it.n_rays + __float_as_int(ds.w);
          out_item = pk_item;
          active = true;
        }
        pk_next += min(__popc(idle), avail);
        idle = __ballot_sync(FULL, !active);
      }
      __syncwarp();
      if (lane == 0) {
        s_cur[wid] = cur;
        s_drained[wid] = drained ? 1 : 0;
      }
      __syncwarp();
    }
    const unsigned act = __ballot_sync(FULL, active);
    if (act == 0) {
      if (s_drained[wid]) {
        if (parked) store_parked(items[out_item], out_o, sm.keys[lane]);
        break;
      }
      continue;
    }
    bool fin = false;
    if (COUNT) {
      c_iters += lane == 0 ? 1u : 0u;
      c_lane_iters += active ? 1u : 0u;
    }
    if (tri_mode != 1) {
      bool ok = true;
      if (active) ok = tr.descend(st);
      dev::tri_phase_warp(tr, sm.keys, lane, &g_status);
      if (active) {
        if (!ok) {
          atomicOr(&g_status, tr.fail_bits());
          fin = true;
        } else {
          fin = tr.finish_pooled(st);
        }
      }
    } else if (active) {
      const int pl = postpone_pct > 0 ? (__popc(act) * postpone_pct + 99) / 100 : 0;
      fin = tr.step(st, pl, &g_status);
    }
    if (fin) {
      float rg;
      int32_t id;
      tr.result(rg, id);
      sm.keys[lane] = ((unsigned long long)__float_as_uint(rg) << 32) | (uint32_t)id;
      parked = true;
      active = false;
      if (COUNT) ++c_rays;
    }
  }
  if (COUNT) {
    const uint32_t c[kWorkCounters] = {c_rays, c_nodes + tr.n_nodes, c_tris + tr.n_tris, c_iters,
                                       c_lane_iters, tr.n_rounds, tr.n_pops, c_refills};
    flush_counters<COUNT>(c);
  }
}

// Shared memory of the packet kernels: that of the traversal, then one list
// slot (8 B) and one pending word a thread.
__device__ __forceinline__ dev::PacketList packet_smem(int W, int sdepth) {
  extern __shared__ __align__(16) unsigned long long smem_u64[];
  uint2* list = reinterpret_cast<uint2*>(reinterpret_cast<char*>(smem_u64) +
                                         (size_t)blockDim.x * (8 + (size_t)sdepth * (8 + 2 * W)));
  return dev::PacketList{list + (threadIdx.x & ~31u), reinterpret_cast<uint32_t*>(list + blockDim.x) + threadIdx.x};
}

// One packet: up to 32 consecutive rays (tile order) of one environment of an
// item, by one warp.  The packet phase walks the tree for all of them; the
// per-ray traversal takes what it leaves.
template <int W, bool COUNT, bool TMIN>
__device__ __forceinline__ void trace_packet(const ItemDesc& it, int env, int first, int n, const Smem<W>& sm,
                                             const dev::PacketList& pl,
                                             const dev::StackRefs<typename dev::KeyWords<W>::T>& st,
                                             unsigned* status, uint32_t (&c)[kWorkCounters]) {
  const unsigned FULL = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31;
  const bool live = lane < n;  // a lane past the end copies the first ray (and neither traces alone nor stores)
  const float4 ds = __ldg((const float4*)it.dirs + first + (live ? lane : 0));
  const int64_t o = (int64_t)env * it.n_rays + __float_as_int(ds.w);
  dev::Tracer<W, COUNT, TMIN> tr;
  dev::PacketEnd end;
  {
    float ox, oy, oz, dx, dy, dz;
    dev::world_ray(it.poses + 12 * (int64_t)env, ds, ox, oy, oz, dx, dy, dz);
    dev::setup_ray(tr.r, ox, oy, oz, dx, dy, dz);
    tr.start(it.nodes, it.tris, it.min_range, it.max_range, it.n_nodes, it.n_tris);
    if (COUNT) tr.n_rounds = tr.n_pops = 0;
    end = dev::packet_phase(tr, dx, dy, dz, (const uint4*)it.top, it.n_tris, pl, lane, live, status, c[3], c[4]);
  }
  if (end != dev::kPacketDone) {
    bool active = live && (end == dev::kPacketNone || tr.next_entry(pl));
    while (__any_sync(FULL, active)) {
      if (COUNT) {
        c[3] += lane == 0 ? 1u : 0u;
        c[4] += active ? 1u : 0u;
      }
      bool ok = true;
      if (active) ok = tr.descend(st);
      dev::tri_phase_warp(tr, sm.keys, lane, status);
      if (active) {
        if (!ok) {
          atomicOr(status, tr.fail_bits());
          active = false;
        } else {
          active = !tr.template finish_pooled<true>(st, pl);
        }
      }
    }
  }
  if (live) {
    float rg;
    int32_t id;
    tr.result(rg, id);
    __stcs(it.out_range + o, rg);  // evict-first: the results do not push the BVH out of L2
    __stcs(it.out_tri + o, id);
  }
  if (COUNT) {
    c[0] += live ? 1u : 0u;
    c[1] += tr.n_nodes;
    c[2] += tr.n_tris;
    c[5] += tr.n_rounds;
    c[6] += tr.n_pops;
  }
}

// k_plain with packet phases: warp w of the grid takes packet w of the item,
// `rays` rays (32, or 16 in a small cast; the other lanes copy the first).
template <int W, bool COUNT, bool TMIN>
__global__ void __maxnreg__(72) k_plain_packets(const ItemDesc it, int sdepth, unsigned* status, int rays) {
  using Keys = typename dev::KeyWords<W>::T;
  if (status == nullptr) status = &g_status;
  if (it.width != W) {  // never read nodes laid out for another width
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(status, 2u);
    return;
  }
  const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t env = (p >> 32) ? p / it.pk_per_env : (int64_t)((uint32_t)p / (uint32_t)it.pk_per_env);
  if (env >= it.n_env) return;
  const int first = (int)(p - env * it.pk_per_env) * rays;
  const Smem<W> sm = smem_layout<W>(sdepth);
  uint2 ls[kStackLocal];
  Keys lq[kStackLocal];
  const dev::StackRefs<Keys> st{sm.ss, sm.sq, ls, lq, (int)blockDim.x, sdepth};
  uint32_t c[kWorkCounters] = {};
  trace_packet<W, COUNT, TMIN>(it, (int)env, first, min(rays, it.n_rays - first), sm, packet_smem(W, sdepth), st, status,
                               c);
  flush_counters<COUNT>(c);
}

// k_persistent with packet phases: a warp draws packets of the queue and takes
// the rays of each 32 at a time.  Bound, like k_persistent, by instruction
// issue (0.70-0.75 of it), but with 140 instead of 224 warp instructions a ray:
// 4096 x 5760 rays on 1 M triangles of a cluttered room 4.91 -> 3.46 ms, a fleet
// of dense sensors on 3 cm triangles 1.86 -> 1.59 ms; k_plain_packets takes 35 us
// for one scan of 57,600 rays (packets of 16; 42 with 32, a call 51 -> 38 us).  Under
// the 72-register cap 52 bytes a thread spill; 64 (more spills) and 80 (fewer warps)
// are 1-5% slower, and sharing the loop with k_persistent's refill of partly idle
// warps keeps so much alive that most of the gain is lost.
//
// The queue's counter hands out a draw every 2.6 ns, which bounds cheap
// packets (368,640 on 20 k triangles took 0.99 ms), so a warp draws three at
// once while more than 16 a warp are left, then one: 0.81 ms there, 1.76 ->
// 1.72 on 1 M triangles, the same for few packets.  (Four are as good, eight or
// a smaller rest leave some warps with too many: up to 50% slower.)
constexpr unsigned long long kDrawLeft = 16;
constexpr unsigned kDrawMany = 3;

// k_packets' own shared memory, beside the launch's dynamic part.
struct PacketQueue {
  unsigned long long next[kMaxBlockWarps], end[kMaxBlockWarps];  // the warp's own packets
  unsigned long long total;  // not read again beside the counter, whose line the draws keep busy
};

template <int W, bool COUNT, bool TMIN>
__global__ void __maxnreg__(72) k_packets(BatchHeader* __restrict__ hdr, const ItemDesc* __restrict__ items,
                                           int sdepth) {
  using Keys = typename dev::KeyWords<W>::T;
  const unsigned FULL = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31;
  const Smem<W> sm = smem_layout<W>(sdepth);
  const dev::PacketList pl = packet_smem(W, sdepth);
  uint2 ls[kStackLocal];
  Keys lq[kStackLocal];
  const dev::StackRefs<Keys> st{sm.ss, sm.sq, ls, lq, (int)blockDim.x, sdepth};
  uint32_t c[kWorkCounters] = {};
  __shared__ PacketQueue q;
  const int wid = threadIdx.x >> 5;
  if (lane == 0) q.next[wid] = q.end[wid] = 0ull;
  if (threadIdx.x == 0) q.total = (unsigned long long)hdr->n_packets;
  __syncthreads();
  for (;;) {
    unsigned long long p = 0;
    if (lane == 0) {
      p = q.next[wid];
      if (p == q.end[wid]) {
        const unsigned long long total = q.total;
        const unsigned draw = p + kDrawLeft * (gridDim.x * (blockDim.x >> 5)) < total ? kDrawMany : 1u;
        p = atomicAdd(&hdr->head, (unsigned long long)draw);
        q.end[wid] = p < total ? min(p + draw, total) : p;
      }
      q.next[wid] = p + 1;
    }
    p = __shfl_sync(FULL, p, 0);
    if (p >= q.total) break;
    int lo = 0, hi = hdr->n_items - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (items[mid].pk_begin <= (int64_t)p) lo = mid;
      else hi = mid - 1;
    }
    const ItemDesc& it = items[lo];
    if (COUNT && lane == 0) ++c[7];
    if (it.width != W) {  // never read nodes laid out for another width
      if (lane == 0) atomicOr(&g_status, 2u);
      continue;
    }
    const int64_t local = (int64_t)p - it.pk_begin;
    const int ppe = it.pk_per_env;
    const int env = (local >> 32) ? (int)(local / ppe) : (int)((uint32_t)local / (uint32_t)ppe);
    const int P = hdr->packet_rays;
    int first = (int)(local - (int64_t)env * ppe) * P;
    const int end = min(first + P, it.n_rays);
    for (; first < end; first += 32)
      trace_packet<W, COUNT, TMIN>(it, env, first, min(32, end - first), sm, pl, st, &g_status, c);
  }
  flush_counters<COUNT>(c);
}

// Second pass over one item for instance k: every ray, moved into the
// instance's frame by the inverse of its rigid pose (the float32 sequence of
// fgl.h), is cast against the instance's BVH, pruned by the return found so
// far, and replaces it only when strictly nearer (ties stay with the scene
// and with lower instances).
template <int W, bool TMIN>
__global__ void __maxnreg__(72) k_instance_pass(const InstancePass a, int sdepth) {
  using Keys = typename dev::KeyWords<W>::T;
  const unsigned FULL = 0xFFFFFFFFu;
  const Smem<W> sm = smem_layout<W>(sdepth);
  const int lane = threadIdx.x & 31;
  if (a.width != W) {
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&g_status, 2u);
    return;
  }
  const int64_t total = (int64_t)a.n_env * a.n_rays;
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool done = gid >= total;
  int64_t o_idx = 0;
  float cur_t = 0.f;
  int32_t cur_id = -1;
  dev::Tracer<W, false, TMIN> tr;
  tr.tg = make_uint2(0u, 0u);
  tr.ng = make_uint2(0u, 0u);
  if (!done) {
    const int env = (int)(gid / a.n_rays);
    const int j = (int)(gid - (int64_t)env * a.n_rays);
    const float4 ds = __ldg((const float4*)a.dirs + j);
    o_idx = (int64_t)env * a.n_rays + __float_as_int(ds.w);
    float ox, oy, oz, dx, dy, dz;
    dev::world_ray(a.poses + 12 * (int64_t)env, ds, ox, oy, oz, dx, dy, dz);
    const float* P = a.inst_poses + 12 * ((int64_t)env * a.n_inst + a.k);
    float R[12];
#pragma unroll
    for (int i = 0; i < 12; ++i) R[i] = __ldg(P + i);
    const float u0 = __fsub_rn(ox, R[3]), u1 = __fsub_rn(oy, R[7]), u2 = __fsub_rn(oz, R[11]);
    // o' = R^T u, d' = R^T d: column i of R against (u0, u1, u2)
    float lo[3], ld[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      lo[i] = __fadd_rn(__fadd_rn(__fmul_rn(R[i], u0), __fmul_rn(R[4 + i], u1)), __fmul_rn(R[8 + i], u2));
      ld[i] = __fadd_rn(__fadd_rn(__fmul_rn(R[i], dx), __fmul_rn(R[4 + i], dy)), __fmul_rn(R[8 + i], dz));
    }
    cur_t = a.out_range[o_idx];
    cur_id = a.out_tri[o_idx];
    dev::setup_ray(tr.r, lo[0], lo[1], lo[2], ld[0], ld[1], ld[2]);
    tr.start(a.nodes, a.tris, a.min_range, cur_t, a.n_nodes, a.n_tris);
  }
  uint2 ls[kStackLocal];
  Keys lq[kStackLocal];
  const dev::StackRefs<Keys> st{sm.ss, sm.sq, ls, lq, (int)blockDim.x, sdepth};
  while (__any_sync(FULL, !done)) {
    bool ok = true;
    if (!done) ok = tr.descend(st);
    dev::tri_phase_warp(tr, sm.keys, lane, &g_status);
    if (!done) {
      if (!ok) {
        atomicOr(&g_status, tr.fail_bits());
        done = true;
      } else {
        done = tr.finish_pooled(st);
      }
    }
  }
  if (gid < total) {
    const bool take = tr.best_id != dev::kNoHit && (cur_id < 0 || tr.best_t < cur_t);
    if (take) {
      a.out_range[o_idx] = tr.best_t;
      a.out_tri[o_idx] = tr.best_id;
      if (a.out_inst) a.out_inst[o_idx] = a.k;
    } else if (a.k == 0 && a.out_inst) {
      a.out_inst[o_idx] = -1;
    }
  }
}

// Ray gid of an item as (environment, tile-order ray), by a 32-bit division
// where it fits.
__device__ __forceinline__ void ray_of(int64_t gid, int n_rays, int64_t& env, int& j) {
  env = (gid >> 32) ? gid / n_rays : (int64_t)((uint32_t)gid / (uint32_t)n_rays);
  j = (int)(gid - env * n_rays);
}

// World-frame return point: p_i = o_i + (t * d_i) (two roundings), NaN on a miss.
__device__ __forceinline__ void store_point(float* out, int64_t o, bool hit, float t, float ox, float oy, float oz,
                                            float dx, float dy, float dz) {
  const float nan = __int_as_float(0x7FC00000);
  __stcs(out + 3 * o + 0, hit ? __fadd_rn(ox, __fmul_rn(t, dx)) : nan);
  __stcs(out + 3 * o + 1, hit ? __fadd_rn(oy, __fmul_rn(t, dy)) : nan);
  __stcs(out + 3 * o + 2, hit ? __fadd_rn(oz, __fmul_rn(t, dz)) : nan);
}

// Every instance of an item in one pass (all of one width): a ray's world
// ray and its return so far stay in registers while it is moved into each
// instance's frame in turn (instance order) and cast there, pruned by that
// return, replacing it only when strictly nearer -- the per-instance passes'
// result, bit for bit, with the ray's record read and written once and its
// return point beside it.  Bound by issue, at part of the lanes: 5.9 M rays and
// four objects 0.41 ms, 0.44 with the points in a pass of their own.  (Walking
// an object's upper tree a packet at a time, as the scene's, was slower: by 7%
// of the whole cast where eight or more rays are left.)
template <int W, bool TMIN>
__global__ void __maxnreg__(72) k_instances_fused(const InstanceSet a, int sdepth) {
  using Keys = typename dev::KeyWords<W>::T;
  const unsigned FULL = 0xFFFFFFFFu;
  const Smem<W> sm = smem_layout<W>(sdepth);
  const int lane = threadIdx.x & 31;
  const InstancePass& b = a.base;
  if (b.width != W) {
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&g_status, 2u);
    return;
  }
  const int64_t total = (int64_t)b.n_env * b.n_rays;
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = gid < total;
  int64_t o_idx = 0, env = 0;
  float ox = 0.f, oy = 0.f, oz = 0.f, dx = 0.f, dy = 0.f, dz = 1.f;
  float cur_t = 0.f;
  int32_t cur_id = -1, cur_k = -1;
  if (live) {
    int j;
    ray_of(gid, b.n_rays, env, j);
    const float4 ds = __ldg((const float4*)b.dirs + j);
    o_idx = env * b.n_rays + __float_as_int(ds.w);
    dev::world_ray(b.poses + 12 * env, ds, ox, oy, oz, dx, dy, dz);
    cur_t = b.out_range[o_idx];
    cur_id = b.out_tri[o_idx];
  }
  uint2 ls[kStackLocal];
  Keys lq[kStackLocal];
  const dev::StackRefs<Keys> st{sm.ss, sm.sq, ls, lq, (int)blockDim.x, sdepth};
  for (int k = 0; k < b.n_inst; ++k) {
    dev::Tracer<W, false, TMIN> tr;
    tr.tg = make_uint2(0u, 0u);
    tr.ng = make_uint2(0u, 0u);
    bool done = !live;
    if (live) {
      const float* P = b.inst_poses + 12 * (env * b.n_inst + k);
      float R[12];
#pragma unroll
      for (int i = 0; i < 12; ++i) R[i] = __ldg(P + i);
      // cull with the instance's bounding sphere moved into the world: skip
      // when the ray line misses it, it lies behind the origin or wholly
      // beyond the return so far.  A margin of 1e-4 of its distance covers the
      // float32 error of these few products many times over, and the miss
      // test adds 1e-6 dist^2 for the cancellation in dist^2 - tca^2
      // (at most a few units of 2^-23 dist^2).
      const float* sp = a.sphere[k];
      const float cx = R[0] * sp[0] + R[1] * sp[1] + R[2] * sp[2] + R[3] - ox;
      const float cy = R[4] * sp[0] + R[5] * sp[1] + R[6] * sp[2] + R[7] - oy;
      const float cz = R[8] * sp[0] + R[9] * sp[1] + R[10] * sp[2] + R[11] - oz;
      const float dist2 = cx * cx + cy * cy + cz * cz;
      const float tca = cx * dx + cy * dy + cz * dz;
      const float rr = sp[3] + 1e-4f * (sqrtf(dist2) + sp[3]) + 1e-5f;
      const float perp2 = dist2 - tca * tca;
      const bool outside = dist2 > rr * rr;
      done = outside && (perp2 > rr * rr + 1e-6f * dist2 || tca < -rr || tca - rr > cur_t);
      if (!done) {
        const float u0 = __fsub_rn(ox, R[3]), u1 = __fsub_rn(oy, R[7]), u2 = __fsub_rn(oz, R[11]);
        float lo[3], ld[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          lo[i] = __fadd_rn(__fadd_rn(__fmul_rn(R[i], u0), __fmul_rn(R[4 + i], u1)), __fmul_rn(R[8 + i], u2));
          ld[i] = __fadd_rn(__fadd_rn(__fmul_rn(R[i], dx), __fmul_rn(R[4 + i], dy)), __fmul_rn(R[8 + i], dz));
        }
        dev::setup_ray(tr.r, lo[0], lo[1], lo[2], ld[0], ld[1], ld[2]);
        tr.start(a.nodes[k], a.tris[k], b.min_range, cur_t, a.n_nodes[k], a.n_tris[k]);
      } else {
        tr.best_id = dev::kNoHit;
      }
    }
    while (__any_sync(FULL, !done)) {
      bool ok = true;
      if (!done) ok = tr.descend(st);
      dev::tri_phase_warp(tr, sm.keys, lane, &g_status);
      if (!done) {
        if (!ok) {
          atomicOr(&g_status, tr.fail_bits());
          done = true;
        } else {
          done = tr.finish_pooled(st);
        }
      }
    }
    if (live && tr.best_id != dev::kNoHit && (cur_id < 0 || tr.best_t < cur_t)) {
      cur_t = tr.best_t;
      cur_id = tr.best_id;
      cur_k = k;
    }
  }
  if (live) {
    __stcs(b.out_range + o_idx, cur_t);
    __stcs(b.out_tri + o_idx, cur_id);
    if (b.out_inst) __stcs(b.out_inst + o_idx, cur_k);
    if (a.out_points) store_point(a.out_points, o_idx, cur_id >= 0, cur_t, ox, oy, oz, dx, dy, dz);
  }
}

// The return points of an item whose instances were not cast in one pass.
__global__ void k_points(const float4* __restrict__ dirs, const float* __restrict__ poses,
                         int n_env, int n_rays, const float* __restrict__ range,
                         const int32_t* __restrict__ tri, float* __restrict__ out) {
  const int64_t total = (int64_t)n_env * n_rays;
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= total) return;
  int64_t env;
  int j;
  ray_of(gid, n_rays, env, j);
  const float4 ds = __ldg(dirs + j);
  const int64_t o = env * n_rays + __float_as_int(ds.w);
  float ox, oy, oz, dx, dy, dz;
  dev::world_ray(poses + 12 * env, ds, ox, oy, oz, dx, dy, dz);
  store_point(out, o, tri[o] >= 0, range[o], ox, oy, oz, dx, dy, dz);
}

// Every thread reads 16-byte words of `buf` (L2 only: ld.global.cg) in a
// grid-stride loop, `reps` times over, and folds them into one word so the
// loads cannot be dropped; block 0's thread 0 publishes the fold of its own
// reads only when it is a value no read can produce alone (never, in
// practice), keeping the store off the timed path.
__global__ void k_l2_read(const uint4* __restrict__ buf, int64_t n16, int reps,
                          unsigned* __restrict__ sink) {
  uint32_t acc = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int r = 0; r < reps; ++r) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + 3 * stride < n16; i += 4 * stride) {  // four independent loads in flight
      const uint4 a = __ldcg(buf + i), b = __ldcg(buf + i + stride);
      const uint4 c = __ldcg(buf + i + 2 * stride), d = __ldcg(buf + i + 3 * stride);
      acc ^= (a.x ^ a.y ^ a.z ^ a.w) ^ (b.x ^ b.y ^ b.z ^ b.w) ^ (c.x ^ c.y ^ c.z ^ c.w) ^
             (d.x ^ d.y ^ d.z ^ d.w);
    }
    for (; i < n16; i += stride) {
      const uint4 v = __ldcg(buf + i);
      acc ^= v.x ^ v.y ^ v.z ^ v.w;
    }
  }
  if (acc == 0x5A17C0DEu) atomicXor(sink, acc);
}

__global__ void k_world_rays(const float4* __restrict__ dirs, const float* __restrict__ poses,
                             int n_env, int n_rays, float* __restrict__ out_o,
                             float* __restrict__ out_d) {
  const int64_t total = (int64_t)n_env * n_rays;
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= total) return;
  const int env = (int)(gid / n_rays);
  const int j = (int)(gid - (int64_t)env * n_rays);
  const float4 ds = dirs[j];
  float ox, oy, oz, dx, dy, dz;
  dev::world_ray(poses + 12 * (int64_t)env, ds, ox, oy, oz, dx, dy, dz);
  const int64_t o = 3 * ((int64_t)env * n_rays + __float_as_int(ds.w));
  out_o[o] = ox;
  out_o[o + 1] = oy;
  out_o[o + 2] = oz;
  out_d[o] = dx;
  out_d[o + 1] = dy;
  out_d[o + 2] = dz;
}

template <int W, bool COUNT, bool TMIN>
void* packets_fn() {
  return (void*)k_packets<W, COUNT, TMIN>;
}
template <int W>
void* pick_packets_w(bool count, bool tmin) {
  if (tmin) return count ? packets_fn<W, true, true>() : packets_fn<W, false, true>();
  return count ? packets_fn<W, true, false>() : packets_fn<W, false, false>();
}
void* pick_packets(int W, bool count, bool tmin) {
  return W == 8 ? pick_packets_w<8>(count, tmin) : pick_packets_w<4>(count, tmin);
}

template <int W, bool COUNT, bool TMIN>
void* persistent_fn() {
  return (void*)k_persistent<W, COUNT, TMIN>;
}

void* pick_plain(int W, bool count) {
  if (W == 8) return count ? (void*)k_plain<8, true> : (void*)k_plain<8, false>;
  return count ? (void*)k_plain<4, true> : (void*)k_plain<4, false>;
}
// A minimum range comes with a GPU-built hierarchy only (8-wide, not counted).
void* pick_plain_packets(int W, bool count, bool tmin) {
  if (W == 8 && tmin) return (void*)k_plain_packets<8, false, true>;
  if (W == 8) return count ? (void*)k_plain_packets<8, true, false> : (void*)k_plain_packets<8, false, false>;
  return count ? (void*)k_plain_packets<4, true, false> : (void*)k_plain_packets<4, false, false>;
}
template <int W>
void* pick_persistent_w(bool count, bool tmin) {
  if (tmin) return count ? persistent_fn<W, true, true>() : persistent_fn<W, false, true>();
  return count ? persistent_fn<W, true, false>() : persistent_fn<W, false, false>();
}
void* pick_persistent(int W, bool count, bool tmin) {
  return W == 8 ? pick_persistent_w<8>(count, tmin) : pick_persistent_w<4>(count, tmin);
}

}  // namespace

size_t stack_smem_bytes(int W, int block, int sdepth) {
  return (size_t)block * sizeof(unsigned long long) +
         (size_t)block * (size_t)sdepth * (sizeof(uint2) + 2 * (size_t)W);
}

static size_t packets_smem_bytes(int W, int block, int sdepth) {
  return stack_smem_bytes(W, block, sdepth) + (size_t)block * (sizeof(uint2) + sizeof(uint32_t));
}

// The limits hold for a kernel's dynamic and static shared memory together;
// kStaticSmem covers the static part of every traversal kernel (at most 320 B).
constexpr size_t kStaticSmem = 512;
static_assert(sizeof(PacketQueue) + 16 <= kStaticSmem, "static shared memory");

bool packets_fit(int W, int block, int sdepth) {
  const size_t smem = packets_smem_bytes(W, block, sdepth) + kStaticSmem;
  if (smem <= 48 * 1024) return true;  // any block's: no need to ask the device
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return false;
  return smem <= (size_t)optin;
}

static cudaError_t allow_smem(void* fn, size_t smem) {
  if (smem + kStaticSmem <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

cudaError_t launch_plain(int W, bool count, int packet_rays, bool tmin, const ItemDesc& it, unsigned* status, int block,
                         int sdepth, int tri_mode, int postpone_pct, cudaStream_t s) {
  const int64_t total = (int64_t)it.n_env * it.n_rays;
  if (total == 0) return cudaSuccess;
  if (tmin && (W != 8 || count || !packet_rays)) return cudaErrorInvalidValue;  // no such form
  ItemDesc arg = it;
  int rays = packet_rays;
  if (rays) arg.pk_per_env = (it.n_rays + rays - 1) / rays;
  const int64_t threads = rays ? (int64_t)it.n_env * arg.pk_per_env * 32 : total;
  const int64_t grid = (threads + block - 1) / block;
  const size_t smem = rays ? packets_smem_bytes(W, block, sdepth) : stack_smem_bytes(W, block, sdepth);
  void* fn = rays ? pick_plain_packets(W, count, tmin) : pick_plain(W, count);
  const cudaError_t e = allow_smem(fn, smem);
  if (e != cudaSuccess) return e;
  void* plain_args[] = {&arg, &sdepth, &tri_mode, &postpone_pct, &status};
  void* packet_args[] = {&arg, &sdepth, &status, &rays};
  return cudaLaunchKernel(fn, dim3((unsigned)grid), dim3(block), rays ? packet_args : plain_args, smem, s);
}

int persistent_blocks_per_sm(int W, bool count, bool tmin, bool packets, int block, int sdepth) {
  void* fn = packets ? pick_packets(W, count, tmin) : pick_persistent(W, count, tmin);
  const size_t smem = packets ? packets_smem_bytes(W, block, sdepth) : stack_smem_bytes(W, block, sdepth);
  allow_smem(fn, smem);
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, block, smem) != cudaSuccess) return 1;
  return n > 0 ? n : 1;
}

cudaError_t launch_persistent(int W, bool count, bool tmin, bool packets, void* scratch, int grid, int block,
                              int sdepth, int refill_min, int tri_mode, int postpone_pct,
                              cudaStream_t s) {
  void* fn = packets ? pick_packets(W, count, tmin) : pick_persistent(W, count, tmin);
  const size_t smem = packets ? packets_smem_bytes(W, block, sdepth) : stack_smem_bytes(W, block, sdepth);
  const cudaError_t e = allow_smem(fn, smem);
  if (e != cudaSuccess) return e;
  BatchHeader* hdr = (BatchHeader*)scratch;
  const ItemDesc* items = (const ItemDesc*)((char*)scratch + sizeof(BatchHeader));
  void* args[] = {&hdr, &items, &sdepth, &refill_min, &tri_mode, &postpone_pct};
  return cudaLaunchKernel(fn, dim3(grid), dim3(block), args, smem, s);
}

cudaError_t launch_instance_pass(const InstancePass& a, bool tmin, int block, int sdepth,
                                 cudaStream_t s) {
  const int64_t total = (int64_t)a.n_env * a.n_rays;
  if (total == 0) return cudaSuccess;
  void* fn;
  if (a.width == 8) fn = tmin ? (void*)k_instance_pass<8, true> : (void*)k_instance_pass<8, false>;
  else fn = tmin ? (void*)k_instance_pass<4, true> : (void*)k_instance_pass<4, false>;
  const size_t smem = stack_smem_bytes(a.width, block, sdepth);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  InstancePass arg = a;
  void* args[] = {&arg, &sdepth};
  return cudaLaunchKernel(fn, dim3((unsigned)((total + block - 1) / block)), dim3(block), args, smem, s);
}

cudaError_t launch_instances_fused(const InstanceSet& a, bool tmin, int block, int sdepth,
                                   cudaStream_t s) {
  const int64_t total = (int64_t)a.base.n_env * a.base.n_rays;
  if (total == 0 || a.base.n_inst == 0) return cudaSuccess;
  void* fn;
  if (a.base.width == 8) fn = tmin ? (void*)k_instances_fused<8, true> : (void*)k_instances_fused<8, false>;
  else fn = tmin ? (void*)k_instances_fused<4, true> : (void*)k_instances_fused<4, false>;
  const size_t smem = stack_smem_bytes(a.base.width, block, sdepth);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  InstanceSet arg = a;
  void* args[] = {&arg, &sdepth};
  return cudaLaunchKernel(fn, dim3((unsigned)((total + block - 1) / block)), dim3(block), args, smem, s);
}

cudaError_t launch_points(const ItemDesc& it, float* out, cudaStream_t s) {
  const int64_t total = (int64_t)it.n_env * it.n_rays;
  if (total == 0) return cudaSuccess;
  k_points<<<(unsigned)((total + 255) / 256), 256, 0, s>>>((const float4*)it.dirs, it.poses, it.n_env,
                                                          it.n_rays, it.out_range, it.out_tri, out);
  return cudaGetLastError();
}

cudaError_t launch_l2_read(const void* buf, int64_t bytes, int reps, unsigned* sink, int sms,
                           cudaStream_t s) {
  if (bytes < 16 || reps < 1) return cudaSuccess;
  k_l2_read<<<sms * 4, 512, 0, s>>>((const uint4*)buf, bytes / 16, reps, sink);
  return cudaGetLastError();
}

cudaError_t launch_world_rays(const void* dirs, const float* poses, int n_env, int n_rays,
                              float* out_o, float* out_d, cudaStream_t s) {
  const int64_t total = (int64_t)n_env * n_rays;
  if (total == 0) return cudaSuccess;
  const int block = 256;
  k_world_rays<<<(unsigned)((total + block - 1) / block), block, 0, s>>>(
      (const float4*)dirs, poses, n_env, n_rays, out_o, out_d);
  return cudaGetLastError();
}

cudaError_t read_and_clear_status(unsigned* st) {
  cudaError_t e = cudaMemcpyFromSymbol(st, g_status, sizeof(unsigned));
  if (e != cudaSuccess) return e;
  if (*st) {
    unsigned z = 0;
    e = cudaMemcpyToSymbol(g_status, &z, sizeof(unsigned));
  }
  return e;
}

cudaError_t read_and_clear_counters(unsigned long long* c) {
  cudaError_t e = cudaMemcpyFromSymbol(c, g_counters, kWorkCounters * sizeof(unsigned long long));
  if (e != cudaSuccess) return e;
  unsigned long long z[kWorkCounters] = {};
  return cudaMemcpyToSymbol(g_counters, z, sizeof(z));
}

}  // namespace fgl
