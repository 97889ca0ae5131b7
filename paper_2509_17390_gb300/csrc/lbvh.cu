// Triangle LBVH built on the GPU: the paper's own structure for LiDAR ray
// casting (Sec. IV-C: a triangle LBVH from the LBVH routine of Sec. IV-A,
// eqs. u_i, m_i and LCP, after Karras 2012), kept beside the host-built wide SAH BVH for scenes that change every frame
// and as the baseline of the build-time / traversal-speed trade-off.
//
// Build (all on one stream): triangle boxes and centroids -> scene bounds ->
// 30-bit Morton codes of the centroids in the centroid box (eq. u_i, m_i)
// -> stable radix sort (sort.cu) -> triangles gathered in Morton order ->
// one thread per internal node finds its key range and split from the longest
// common prefixes of neighbouring codes (eq. LCP; equal codes are told apart
// by their positions) -> boxes bottom up, the second child to arrive at a
// node building it (within a block's leaves in shared memory) -> the binary
// tree opened into 8-wide nodes.  Leaves hold one triangle; every leaf box is
// grown by the margin 2^-17 max(1, max |coord|), which covers the float32
// rounding of the slab tests, so culling never drops a triangle the ray meets.
//
// Cast: the wide nodes are the host-built BVH's record, so packets of rays go
// through the same kernels; rays walked one by one go through the binary tree.
// The triangle test and the (t, id) rule are the same everywhere, so all give
// bitwise identical returns.  2.9 M rays on 500 k triangles: 0.76 ms (the binary
// tree: 0.96), and the build that makes the wide nodes takes 0.30 ms (without
// them, before its climb moved to shared memory: 0.40).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <string>

#include "fgl.h"
#include "fgl_internal.h"
#include "nvtx_range.h"
#include "sort.h"
#include "trace.cuh"


using namespace fgl;

struct fgl_lbvh_s {
  int device = -1;
  int64_t nt = 0;
  bool built = false;          // the arrays hold the tree of the last build, which succeeded
  int64_t n_wide = 0;
  unsigned* status = nullptr;  // device word: bit 0 = a cast's stack overflowed, bit 2 = an
                               // index out of range (checked library)
  void* nodes = nullptr;   // (nt - 1) x 64 B
  void* tris = nullptr;    // nt x 48 B, Morton order
  void* wnodes = nullptr;  // wide_capacity(nt) x 256 B, n_wide of them made: what packets walk
                           // (null: no room for it)
  void* wtris = nullptr;   // nt x 48 B, the wide nodes' leaf runs
  void* work = nullptr;    // build scratch
  size_t work_cap = 0;
  float margin = 0.f;
  float lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
  float build_ms = 0.f;
  int32_t depth = 0;
};

namespace {

// Internal node, 64 bytes: the boxes of both children and their references
// (>= 0: internal node; < 0: ~(leaf = triangle position in Morton order)).
struct LbvhNode {
  float4 a;  // left lo xyz, left hi x
  float4 b;  // left hi yz, right lo xy
  float4 c;  // right lo z, right hi xyz
  int4 d;    // left ref, right ref, parent, 0
};
static_assert(sizeof(LbvhNode) == 64, "LbvhNode layout");

// float <-> int order-preserving map for atomic min / max
__device__ __forceinline__ int ford(float f) {
  const int i = __float_as_int(f);
  return i >= 0 ? i : i ^ 0x7FFFFFFF;
}
__host__ __device__ __forceinline__ float iord(int i) {
#ifdef __CUDA_ARCH__
  return __int_as_float(i >= 0 ? i : i ^ 0x7FFFFFFF);
#else
  int j = i >= 0 ? i : i ^ 0x7FFFFFFF;
  float f;
  std::memcpy(&f, &j, 4);
  return f;
#endif
}

__global__ void k_lbvh_boxes(const float* __restrict__ V, int64_t nv, const int32_t* __restrict__ T,
                             int64_t nt, float4* __restrict__ tbox, int* __restrict__ bounds,
                             int32_t* __restrict__ status) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  float clo[3] = {INFINITY, INFINITY, INFINITY}, chi[3] = {-INFINITY, -INFINITY, -INFINITY};
  float amax = 0.f;
  if (i < nt) {
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    bool ok = true;
    for (int v = 0; v < 3; ++v) {
      const int32_t vi = T[3 * i + v];
      if (vi < 0 || vi >= nv) {
        ok = false;
        continue;
      }
      for (int a = 0; a < 3; ++a) {
        const float x = V[3 * (int64_t)vi + a];
        if (!isfinite(x)) ok = false;
        lo[a] = fminf(lo[a], x);
        hi[a] = fmaxf(hi[a], x);
        amax = fmaxf(amax, fabsf(x));
      }
    }
    if (!ok) {
      atomicExch(status, 1);
      for (int a = 0; a < 3; ++a) lo[a] = hi[a] = 0.f;
      amax = 0.f;
    }
    tbox[2 * i] = make_float4(lo[0], lo[1], lo[2], 0.f);
    tbox[2 * i + 1] = make_float4(hi[0], hi[1], hi[2], 0.f);
    for (int a = 0; a < 3; ++a) {
      const float c = 0.5f * lo[a] + 0.5f * hi[a];
      clo[a] = c;
      chi[a] = c;
    }
  }
  // block reduction (on the order-preserving integers: one reduction
  // instruction a quantity), then one atomic per block and quantity -- an
  // atomic a warp serialised on the seven words (73 us at 500 k triangles)
  __shared__ int s_red[8][7];
  const int w = threadIdx.x >> 5;
  int v[7];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    v[q] = __reduce_min_sync(0xFFFFFFFFu, ford(clo[q]));
    v[3 + q] = __reduce_max_sync(0xFFFFFFFFu, ford(chi[q]));
  }
  v[6] = __reduce_max_sync(0xFFFFFFFFu, ford(amax));
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int q = 0; q < 7; ++q) s_red[w][q] = v[q];
  __syncthreads();
  if (threadIdx.x < 7) {
    const int q = threadIdx.x;
    int r = s_red[0][q];
    for (int k = 1; k < 8; ++k) r = q < 3 ? min(r, s_red[k][q]) : max(r, s_red[k][q]);
    if (q < 3) atomicMin(&bounds[q], r);
    else atomicMax(&bounds[q], r);
  }
}

__device__ __forceinline__ uint32_t spread10(uint32_t x) {
  x &= 0x3FFu;
  x = (x | (x << 16)) & 0x030000FFu;
  x = (x | (x << 8)) & 0x0300F00Fu;
  x = (x | (x << 4)) & 0x030C30C3u;
  x = (x | (x << 2)) & 0x09249249u;
  return x;
}

// eq. u_i, m_i: centroids quantised to 10 bits per axis inside the centroid
// box, bits interleaved (x highest).
__global__ void k_lbvh_morton(const float4* __restrict__ tbox, int64_t nt, const int* __restrict__ bounds,
                              uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nt) return;
  const float4 lo = tbox[2 * i], hi = tbox[2 * i + 1];
  const float c[3] = {0.5f * lo.x + 0.5f * hi.x, 0.5f * lo.y + 0.5f * hi.y, 0.5f * lo.z + 0.5f * hi.z};
  uint32_t u[3];
  for (int a = 0; a < 3; ++a) {
    const float b0 = iord(bounds[a]), b1 = iord(bounds[3 + a]);
    const float ext = b1 - b0;
    float q = ext > 0.f ? (c[a] - b0) / ext * 1024.f : 0.f;
    q = fminf(fmaxf(q, 0.f), 1023.f);
    u[a] = (uint32_t)q;
  }
  keys[i] = (spread10(u[0]) << 2) | (spread10(u[1]) << 1) | spread10(u[2]);
  vals[i] = (uint32_t)i;
}

// Triangles in Morton order (the 48-byte leaf record of the wide BVH) and the
// leaf boxes grown by the margin.
__global__ void k_lbvh_gather(const float* __restrict__ V, const int32_t* __restrict__ T,
                              int64_t nv, const uint32_t* __restrict__ order,
                              const float4* __restrict__ tbox, int64_t nt, const int* __restrict__ bounds,
                              float4* __restrict__ tris, float4* __restrict__ lbox) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nt) return;
  const uint32_t t = order[k];
  const float m = ldexpf(fmaxf(1.f, iord(bounds[6])), -17);
  for (int v = 0; v < 3; ++v) {
    int32_t vi = T[3 * (int64_t)t + v];
    if (vi < 0 || vi >= nv) vi = 0;
    const float* p = V + 3 * (int64_t)vi;
    tris[3 * k + v] = make_float4(p[0], p[1], p[2], v == 0 ? __int_as_float((int)t) : 0.f);
  }
  const float4 lo = tbox[2 * t], hi = tbox[2 * t + 1];
  lbox[2 * k] = make_float4(lo.x - m, lo.y - m, lo.z - m, 0.f);
  lbox[2 * k + 1] = make_float4(hi.x + m, hi.y + m, hi.z + m, 0.f);
}

// The codes, those of the block's leaves from shared memory (most of a node's
// search stays there).
struct Codes {
  const uint32_t* key;
  const uint32_t* near;  // key[b0 ..]
  int n, b0, width;
  __device__ __forceinline__ uint32_t at(int j) const {
    const unsigned k = (unsigned)(j - b0);
    return k < (unsigned)width ? near[k] : __ldg(key + j);
  }
};

// eq. LCP with positions breaking ties between equal codes
__device__ __forceinline__ int lcp(const Codes& c, uint32_t a, int i, int j) {
  if (j < 0 || j >= c.n) return -1;
  const uint32_t b = c.at(j);
  if (a != b) return __clz(a ^ b);
  return 32 + __clz((uint32_t)i ^ (uint32_t)j);
}

// Union of two boxes held as (lo xyz, hi xyz).
struct Box {
  float v[6];
};
__device__ __forceinline__ Box merge(const Box& a, const Box& b) {
  Box r;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    r.v[q] = fminf(a.v[q], b.v[q]);
    r.v[3 + q] = fmaxf(a.v[3 + q], b.v[3 + q]);
  }
  return r;
}
__device__ __forceinline__ void write_children(LbvhNode* nd, const Box& l, const Box& r) {
  nd->a = make_float4(l.v[0], l.v[1], l.v[2], l.v[3]);
  nd->b = make_float4(l.v[4], l.v[5], r.v[0], r.v[1]);
  nd->c = make_float4(r.v[2], r.v[3], r.v[4], r.v[5]);
}

// The hierarchy, and the boxes of the subtrees that lie within one block's
// leaves.  Thread i finds node i's key range, split and children (Karras
// 2012) and publishes the parent links.  Node i sits at one end of its range,
// so a node whose range lies within the block's leaves has its children and
// their links in the block: those subtrees (95% of the nodes) are climbed
// bottom up in shared memory -- the second child to arrive builds the node,
// an arrival being atomicMax(flag, height << 1 | 1).  The roots of the block's
// subtrees (their parents span blocks) go to a list with their boxes and
// heights for k_lbvh_top.  Leaves hold one triangle; leaf boxes come grown.
// Bound by the latency of the searches that leave the block's codes: 46 us at
// 500 k triangles; every node climbed in global memory took 29 + 100 us.
// (Searching eight ways at once: 54 us, so the search's loads are not it
// alone; blocks of 512: the same.)
constexpr int kLbvhBlock = 256;

__global__ void __launch_bounds__(kLbvhBlock) k_lbvh_karras(const uint32_t* __restrict__ key, int64_t n,
                                                            LbvhNode* __restrict__ nodes,
                                                            int32_t* __restrict__ leaf_parent, int32_t* __restrict__ split,
                                                            const float4* __restrict__ lbox, float4* __restrict__ nbox,
                                                            int2* __restrict__ roots, int* __restrict__ n_roots) {
  __shared__ int s_leaf_par[kLbvhBlock], s_node_par[kLbvhBlock], s_left[kLbvhBlock], s_right[kLbvhBlock];
  __shared__ unsigned s_flag[kLbvhBlock];
  __shared__ Box s_leaf[kLbvhBlock], s_node[kLbvhBlock];
  __shared__ uint32_t s_key[kLbvhBlock];
  __shared__ int2 s_roots[kLbvhBlock];  // at most one a leaf
  __shared__ int s_n_roots, s_base;
  const int t = threadIdx.x;
  const int64_t b0 = (int64_t)blockIdx.x * kLbvhBlock, i = b0 + t, bend = min(b0 + kLbvhBlock, n);
  s_leaf_par[t] = s_node_par[t] = -1;
  s_flag[t] = 0u;
  if (t == 0) s_n_roots = 0;
  if (i < n) {
    const float4 lo = lbox[2 * i], hi = lbox[2 * i + 1];
    s_leaf[t] = Box{{lo.x, lo.y, lo.z, hi.x, hi.y, hi.z}};
    s_key[t] = key[i];
  }
  __syncthreads();
  if (i < n - 1) {
    const Codes c{key, s_key, (int)n, (int)b0, (int)(bend - b0)};
    const uint32_t own = s_key[t];
    const int me = (int)i;  // n < 2^30: every index below fits 32 bits
    const int d = (lcp(c, own, me, me + 1) - lcp(c, own, me, me - 1)) >= 0 ? 1 : -1;
    const int dmin = lcp(c, own, me, me - d);
    int lmax = 2;
    while (lcp(c, own, me, me + lmax * d) > dmin) lmax <<= 1;
    int l = 0;
    for (int t = lmax >> 1; t >= 1; t >>= 1)
      if (lcp(c, own, me, me + (l + t) * d) > dmin) l += t;
    const int j = me + l * d;
    const int dnode = lcp(c, own, me, j);
    int s = 0;
    for (int div = 2;; div <<= 1) {
      const int t = (l + div - 1) / div;
      if (lcp(c, own, me, me + (s + t) * d) > dnode) s += t;
      if (t <= 1) break;
    }
    const int g = me + s * d + (d < 0 ? -1 : 0);
    const int lo = min(me, j), hi = max(me, j);
    const bool local = lo >= b0 && hi < bend;
    int left, right;
    if (lo == g) {
      left = ~(int)g;
      leaf_parent[g] = (int)i;
      if (local) s_leaf_par[g - b0] = t;
    } else {
      left = (int)g;
      nodes[g].d.z = (int)i;
      if (local) s_node_par[g - b0] = t;
    }
    if (hi == g + 1) {
      right = ~(int)(g + 1);
      leaf_parent[g + 1] = (int)i;
      if (local) s_leaf_par[g + 1 - b0] = t;
    } else {
      right = (int)(g + 1);
      nodes[g + 1].d.z = (int)i;
      if (local) s_node_par[g + 1 - b0] = t;
    }
    nodes[i].d.x = left;
    nodes[i].d.y = right;
    nodes[i].d.w = -1;
    if (i == 0) nodes[0].d.z = -1;
    split[i] = (int)(g - lo + 1);  // leaves of the left child
    s_left[t] = left;
    s_right[t] = right;
  }
  __syncthreads();
  if (i < n) {
    int p = s_leaf_par[t], height = 1, self = ~(int)i;
    Box box = s_leaf[t];
    bool done = false;  // the other child of a node was not there yet
    while (p >= 0) {
      __threadfence_block();
      const unsigned old = atomicMax(&s_flag[p], ((unsigned)height << 1) | 1u);
      if (old == 0u) {
        done = true;
        break;
      }
      __threadfence_block();
      height = max(height, (int)(old >> 1)) + 1;
      const int l = s_left[p], r = s_right[p];
      const Box bl = l < 0 ? s_leaf[~l - b0] : s_node[l - b0], br = r < 0 ? s_leaf[~r - b0] : s_node[r - b0];
      write_children(nodes + b0 + p, bl, br);
      box = merge(bl, br);
      s_node[p] = box;
      self = (int)(b0 + p);
      p = s_node_par[p];
    }
    if (!done) {
      if (self >= 0) {
        nbox[2 * (int64_t)self] = make_float4(box.v[0], box.v[1], box.v[2], 0.f);
        nbox[2 * (int64_t)self + 1] = make_float4(box.v[3], box.v[4], box.v[5], 0.f);
      }
      s_roots[atomicAdd(&s_n_roots, 1)] = make_int2(self, height);
    }
  }
  __syncthreads();
  if (t == 0) s_base = atomicAdd(n_roots, s_n_roots);
  __syncthreads();
  if (t < s_n_roots) roots[s_base + t] = s_roots[t];
}

// A child's box: leaves from an earlier launch, internal nodes perhaps written
// in this launch by another thread (read past L1, after the fence).
__device__ __forceinline__ Box child_box(const float4* nbox, const float4* lbox, int ref) {
  const float4* p = ref < 0 ? lbox + 2 * (int64_t)(~ref) : nbox + 2 * (int64_t)ref;
  const float4 lo = __ldcg(p), hi = __ldcg(p + 1);
  return Box{{lo.x, lo.y, lo.z, hi.x, hi.y, hi.z}};
}

// The nodes that span blocks, bottom up from the blocks' subtree roots: the
// second child to reach a node writes both children's boxes into it and its
// own box, and climbs on.  A child arrives with atomicMax(flags,
// height << 1 | 1): the first sees 0 and stops, the second reads the other
// subtree's height, so the root's climb carries the tree's exact height (a
// leaf counts 1).  A chain of dependent round trips to L2 a level: 40 us at
// 500 k triangles (20 k roots), with the next node's links read while the
// boxes merge (57 without).
__global__ void k_lbvh_top(LbvhNode* nodes, const int32_t* __restrict__ leaf_parent, uint32_t* flags, float4* nbox,
                           const float4* __restrict__ lbox, const int2* __restrict__ roots,
                           const int* __restrict__ n_roots, int32_t* depth) {
  const int n = *n_roots;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int2 r0 = roots[k];
    int self = r0.x, height = r0.y;
    int p = self < 0 ? leaf_parent[~self] : nodes[self].d.z;
    Box box = child_box(nbox, lbox, self);
    int4 D = p >= 0 ? __ldcg(&nodes[p].d) : make_int4(0, 0, 0, 0);  // links: written by an earlier launch
    bool done = false;
    while (p >= 0) {
      // releases this subtree's boxes and acquires the other's
      uint32_t old;
      asm volatile("atom.acq_rel.gpu.global.max.u32 %0, [%1], %2;"
                   : "=r"(old)
                   : "l"(flags + p), "r"(((uint32_t)height << 1) | 1u)
                   : "memory");
      if (old == 0u) {  // the other child is not done yet
        done = true;
        break;
      }
      height = max(height, (int)(old >> 1)) + 1;
      const bool is_left = D.x == self;
      const Box other = child_box(nbox, lbox, is_left ? D.y : D.x);
      const int up = D.z;
      if (up >= 0) D = __ldcg(&nodes[up].d);
      write_children(nodes + p, is_left ? box : other, is_left ? other : box);
      box = merge(box, other);
      nbox[2 * (int64_t)p] = make_float4(box.v[0], box.v[1], box.v[2], 0.f);
      nbox[2 * (int64_t)p + 1] = make_float4(box.v[3], box.v[4], box.v[5], 0.f);
      self = p;
      p = up;
    }
    if (!done) atomicMax(depth, height);
  }
}

// ---------------------------------------------------------------------------
// the wide form the casts walk: 8-wide nodes (the record of the host-built
// BVH) opened from the binary tree top down, largest box first
// ---------------------------------------------------------------------------

// Wide nodes of a tree over n triangles, at most.  A node of fewer than eight
// children holds leaf runs only (nothing left to open) and more than three
// triangles, so there are at most n / 4 + 1 of those; a full node adds seven
// children net, which bounds the full ones by (n - 1 - others) / 7.
int64_t wide_capacity(int64_t n) { return n * 5 / 14 + 8; }

struct WideArgs {
  const LbvhNode* nodes;
  const int32_t* split;  // leaves of a binary node's left child
  const float4* lbox;
  const float4* tris;    // Morton order
  int64_t n;
  uint8_t* wnodes;       // 256-byte records
  float4* wtris;         // 48-byte records, each node's leaf runs together
  int4* wroot;           // the binary node a wide node is opened from, its first leaf and leaf count
  int* n_tris;           // triangles placed
  int* level;            // [kWideLevels] wide nodes that a level's opening made
  int cap;
};

// Levels the launch can need: a wide node's children lie at least one binary
// level below it, and a path holds at most 30 code bits and 30 position bits.
constexpr int kWideLevels = 64;

// Eight lanes a wide node: a lane a child.  Starting from the binary node's two
// children, the two children of the largest boxes with more than three
// triangles are replaced by their own two a round, until eight are held (three
// rounds of loads, mostly); at most three triangles make a leaf run.  The nodes
// of a level are opened together, the levels separated by a grid barrier (a
// cooperative launch); a block numbers its new nodes and triangles with one
// atomic each.  Bound by the latency of those rounds and barriers.  On 500 k
// triangles, launch plus a cast of 2.9 M rays: one child a round 1.12 ms (the
// best tree, 0.23 ms here), two 1.11, all there is room for 1.15 (a worse tree).
__global__ void __launch_bounds__(256) k_lbvh_wide(const WideArgs a) {
  namespace cg = cooperative_groups;
  cg::grid_group grid = cg::this_grid();
  __shared__ int s_new[2], s_base[2];
  __shared__ int s_ref[32][8], s_first[32][8], s_count[32][8];
  __shared__ Box s_box[32][8];
  const unsigned FULL = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31, q = lane & 7, group = lane & 24, gi = threadIdx.x >> 3;
  const unsigned gmask = 0xFFu << group;
  int begin = 0, end = 1;
  for (int lv = 0; lv < kWideLevels && begin < end; ++lv) {
    for (int w0 = begin + blockIdx.x * 32; w0 < end; w0 += gridDim.x * 32) {  // block-uniform
      const int w = w0 + gi;
      const bool live = w < end;
      if (threadIdx.x < 2) s_new[threadIdx.x] = 0;
      __syncthreads();
      // this lane's child: reference, first leaf, leaves, box
      constexpr int kNone = 0x7FFFFFFF;
      int ref = kNone, first = 0, count = 0, held = 0;
      Box box = {{0.f, 0.f, 0.f, 0.f, 0.f, 0.f}};
      // node r of the leaves [f, f + c): its left child here, its right one in
      // the group's slot `to`
      auto open = [&](int r, int f, int c, int to) {
        const float4 A = __ldcg(&a.nodes[r].a), B = __ldcg(&a.nodes[r].b), C = __ldcg(&a.nodes[r].c);
        const int4 D = __ldcg(&a.nodes[r].d);
        const int left = __ldcg(a.split + r);
        s_ref[gi][to] = D.y;
        s_first[gi][to] = f + left;
        s_count[gi][to] = c - left;
        s_box[gi][to] = Box{{B.z, B.w, C.x, C.y, C.z, C.w}};
        ref = D.x;
        first = f;
        count = left;
        box = Box{{A.x, A.y, A.z, A.w, B.x, B.y}};
      };
      auto collect = [&](int from, int to) {  // lanes [from, to) take what was put in their slots
        __syncwarp();
        if (q >= from && q < to) {
          ref = s_ref[gi][q];
          first = s_first[gi][q];
          count = s_count[gi][q];
          box = s_box[gi][q];
        }
        __syncwarp();
      };
      if (live && a.n == 1) {
        const float4 lo = a.lbox[0], hi = a.lbox[1];
        if (q == 0) {
          ref = ~0;
          count = 1;
          box = Box{{lo.x, lo.y, lo.z, hi.x, hi.y, hi.z}};
        }
        held = 1;
      } else if (live) {
        const int4 root = __ldcg(a.wroot + w);
        if (q == 0) open(root.x, root.y, root.z, 1);
        held = 2;
      }
      collect(held == 2 ? 1 : 8, held);
      for (int round = 0; round < 6; ++round) {
        const float dx = box.v[3] - box.v[0], dy = box.v[4] - box.v[1], dz = box.v[5] - box.v[2];
        const float area = ref >= 0 && ref != kNone && count > 3 ? dx * dy + dy * dz + dz * dx : -1.f;
        int rank = 0, n_open = 0;  // among the group's children that can be opened, largest first
#pragma unroll
        for (int o = 0; o < 8; ++o) {
          const float other = __shfl_sync(FULL, area, group + o);
          rank += other > area || (other == area && o < q) ? 1 : 0;
          n_open += other >= 0.f ? 1 : 0;
        }
        const int now = min(min(n_open, 8 - held), 2);
        if (__all_sync(FULL, now == 0)) break;
        if (area >= 0.f && rank < now) open(ref, first, count, held + rank);
        collect(held, held + now);
        held += now;
      }
      const bool some = ref != kNone, inner = some && count > 3;
      const int tri = some && !inner ? count : 0;
      const unsigned im = (__ballot_sync(FULL, inner) & gmask) >> group;
      int before = tri;  // leaf triangles of the lower lanes of the group
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        const int u = __shfl_up_sync(FULL, before, o, 8);
        if (q >= o) before += u;
      }
      const int n_tri = __shfl_sync(FULL, before, group + 7);
      before -= tri;
      // the node's corner
      float lo[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        lo[c] = some ? box.v[c] : INFINITY;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) lo[c] = fminf(lo[c], __shfl_xor_sync(FULL, lo[c], o));
      }
      int my_node = 0, my_tri = 0;
      if (live && q == 0) {
        my_node = atomicAdd(&s_new[0], __popc(im));
        my_tri = atomicAdd(&s_new[1], n_tri);
      }
      __syncthreads();
      if (threadIdx.x < 2)
        s_base[threadIdx.x] = atomicAdd(threadIdx.x == 0 ? a.level + lv : a.n_tris, s_new[threadIdx.x]);
      __syncthreads();
      const int child_base = __shfl_sync(FULL, my_node, group) + end + s_base[0];
      const int tri_base = __shfl_sync(FULL, my_tri, group) + s_base[1];
      if (live && w < a.cap) {
        float* rec = reinterpret_cast<float*>(a.wnodes + (size_t)w * node_stride(8));
        uint32_t* recu = reinterpret_cast<uint32_t*>(rec);
        if (q < 3) rec[q] = q == 0 ? lo[0] : (q == 1 ? lo[1] : lo[2]);
        if (q >= 3) recu[q] = q == 3 ? im : (q == 4 ? (uint32_t)child_base : (q == 5 ? (uint32_t)tri_base : 0u));
#pragma unroll
        for (int c = 0; c < 3; ++c) {  // offsets rounded outward: the corner plus an offset bounds the box
          rec[8 + 8 * c + q] = some ? __fsub_rd(box.v[c], lo[c]) : 0.f;
          rec[32 + 8 * c + q] = some ? __fsub_ru(box.v[3 + c], lo[c]) : 0.f;
        }
        recu[56 + q] = inner ? 1u << (24 + q) : ((1u << tri) - 1u) << before;
        if (inner) {
          const int child = child_base + __popc(im & ((1u << q) - 1u));
          if (child < a.cap) a.wroot[child] = make_int4(ref, first, count, 0);
        }
        for (int k = 0; k < tri; ++k)
#pragma unroll
          for (int v = 0; v < 3; ++v)
            a.wtris[3 * ((int64_t)tri_base + before + k) + v] = a.tris[3 * ((int64_t)first + k) + v];
      }
    }
    grid.sync();
    begin = end;  // a level's count is final here: the next level adds to its own
    end = min(end + __ldcg(a.level + lv), a.cap);
  }
}

// ---------------------------------------------------------------------------
// cast over the binary tree: one thread per ray, a local stack of nodes with
// their entry distances, nearer child first, children and stacked nodes beyond
// the best hit culled
// ---------------------------------------------------------------------------
constexpr int kLbvhStack = 96;

struct LbvhCast {
  const LbvhNode* nodes;
  const float4* tris;
  int64_t nt;
  const float4* dirs;
  const float* poses;
  int32_t n_env, n_rays;
  float min_range, max_range;
  float* out_range;
  int32_t* out_tri;
};

// Slab test of one child box against (best) with the ray's precomputed
// -o * inv_d offsets: t = fma(plane, inv_d, -o inv_d).
__device__ __forceinline__ bool slab(float lx, float ly, float lz, float hx, float hy, float hz,
                                     const dev::Ray& r, float nox, float noy, float noz,
                                     float tmin, float tmax, float& tn) {
  const float x0 = fmaf(lx, r.ix, nox), x1 = fmaf(hx, r.ix, nox);
  const float y0 = fmaf(ly, r.iy, noy), y1 = fmaf(hy, r.iy, noy);
  const float z0 = fmaf(lz, r.iz, noz), z1 = fmaf(hz, r.iz, noz);
  tn = dev::max3f(fminf(x0, x1), fminf(y0, y1), fmaxf(fminf(z0, z1), tmin));
  const float tf = dev::min3f(fmaxf(x0, x1), fmaxf(y0, y1), fminf(fmaxf(z0, z1), tmax));
  return tn <= tf;
}

template <bool TMIN>
__global__ void k_lbvh_cast(const LbvhCast a, unsigned* status) {
  const int64_t total = (int64_t)a.n_env * a.n_rays;
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= total) return;
  const int env = (int)(gid / a.n_rays);
  const int j = (int)(gid - (int64_t)env * a.n_rays);
  const float4 ds = __ldg(a.dirs + j);
  float ox, oy, oz, dx, dy, dz;
  dev::world_ray(a.poses + 12 * (int64_t)env, ds, ox, oy, oz, dx, dy, dz);
  dev::Tracer<8, false, TMIN> tr;  // ray, best hit and the (t, id) rule; no wide traversal
  dev::setup_ray(tr.r, ox, oy, oz, dx, dy, dz);
  tr.tmin_ = TMIN ? a.min_range : 0.f;
  tr.best_t = a.max_range;
  tr.best_id = dev::kNoHit;
  const float tmin = TMIN ? a.min_range : 0.f;
  const float nox = -ox * tr.r.ix, noy = -oy * tr.r.iy, noz = -oz * tr.r.iz;
  auto test_tri = [&](int64_t k) {
#ifdef FGL_CHECKED
    if (k < 0 || k >= (int64_t)a.nt) {  // checked library: no read past the triangles
      atomicOr(status, 4u);
      return;
    }
#endif
    const float4* tp = a.tris + 3 * k;
    const float4 v0 = __ldg(tp), v1 = __ldg(tp + 1), v2 = __ldg(tp + 2);
    tr.consider(dev::tri_hit(tr.r, v0, v1, v2, tr.best_t), __float_as_int(v0.w));
  };
  if (a.nt == 1) {
    test_tri(0);
  } else {
    int stack[kLbvhStack];
    float stq[kLbvhStack];
    int sp = 0;
    int node = 0;
    for (;;) {
#ifdef FGL_CHECKED
      if (node < 0 || (int64_t)node >= (int64_t)a.nt - 1) {  // checked library: no read past the nodes
        atomicOr(status, 4u);
        break;
      }
#endif
      const LbvhNode* nd = a.nodes + node;
      const float4 A = __ldg(&nd->a), B = __ldg(&nd->b), C = __ldg(&nd->c);
      const int4 D = __ldg(&nd->d);
      float tl, trr;
      bool hl = slab(A.x, A.y, A.z, A.w, B.x, B.y, tr.r, nox, noy, noz, tmin, tr.best_t, tl);
      bool hr = slab(B.z, B.w, C.x, C.y, C.z, C.w, tr.r, nox, noy, noz, tmin, tr.best_t, trr);
      if (hl && D.x < 0) {
        test_tri(~D.x);
        hl = false;
      }
      if (hr && D.y < 0) {
        test_tri(~D.y);
        hr = false;
      }
      hl = hl && tl <= tr.best_t;
      hr = hr && trr <= tr.best_t;
      if (hl && hr) {
        const bool lfirst = tl <= trr;
        if (sp >= kLbvhStack) {
          atomicOr(status, 1u);
          break;
        }
        stack[sp] = lfirst ? D.y : D.x;
        stq[sp] = lfirst ? trr : tl;
        ++sp;
        node = lfirst ? D.x : D.y;
        continue;
      }
      if (hl) {
        node = D.x;
        continue;
      }
      if (hr) {
        node = D.y;
        continue;
      }
      bool found = false;
      while (sp > 0) {
        --sp;
        if (stq[sp] <= tr.best_t) {
          node = stack[sp];
          found = true;
          break;
        }
      }
      if (!found) break;
    }
  }
  float rg;
  int32_t id;
  tr.result(rg, id);
  const int64_t o = (int64_t)env * a.n_rays + __float_as_int(ds.w);
  __stcs(a.out_range + o, rg);  // evict-first: keep L2 for the tree
  __stcs(a.out_tri + o, id);
}

fgl_status err(int status, const std::string& msg) {
  record_error(status, msg.c_str());
  return (fgl_status)status;
}

#define LCUDA(call)                                                                     \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess) return err(FGL_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

namespace fgl {
cudaError_t launch_lbvh_cast(const fgl_lbvh_s* L, const void* dirs, const float* poses, int n_env,
                             int n_rays, float min_range, float max_range, float* out_range,
                             int32_t* out_tri, cudaStream_t s) {
  unsigned* status = L->status;
  const int64_t total = (int64_t)n_env * n_rays;
  if (total == 0) return cudaSuccess;
  LbvhCast a;
  a.nodes = (const LbvhNode*)L->nodes;
  a.tris = (const float4*)L->tris;
  a.nt = L->nt;
  a.dirs = (const float4*)dirs;
  a.poses = poses;
  a.n_env = n_env;
  a.n_rays = n_rays;
  a.min_range = min_range;
  a.max_range = max_range;
  a.out_range = out_range;
  a.out_tri = out_tri;
  const unsigned grid = (unsigned)((total + 127) / 128);
  if (min_range > 0.f) k_lbvh_cast<true><<<grid, 128, 0, s>>>(a, status);
  else k_lbvh_cast<false><<<grid, 128, 0, s>>>(a, status);
  return cudaGetLastError();
}

// The wide form as a cast item.
ItemDesc lbvh_item(const fgl_lbvh_s* L) {
  ItemDesc d{};
  d.nodes = L->wnodes;
  d.tris = L->wtris;
  d.width = 8;
  d.n_nodes = (uint32_t)L->n_wide;
  d.n_tris = (uint32_t)L->nt;
  return d;
}

unsigned* lbvh_status(const fgl_lbvh_s* L) { return L->status; }
bool lbvh_built(const fgl_lbvh_s* L) { return L->built; }
}  // namespace fgl

extern "C" fgl_status fgl_lbvh_build(const float* d_verts, int64_t nv, const int32_t* d_tris,
                                     int64_t nt, fgl_stream stream, fgl_lbvh* out) {
  fgl::NvtxRange range("fgl_lbvh_build");
  if (!out) return err(FGL_ERR_INVALID, "out is null");
  if (!d_verts || !d_tris) return err(FGL_ERR_INVALID, "null vertex or triangle pointer");
  if (nv < 1 || nt < 1) return err(FGL_ERR_INVALID, "mesh needs at least one vertex and triangle");
  if (nt >= ((int64_t)1 << 30)) return err(FGL_ERR_INVALID, "too many triangles (max 2^30 - 1)");
  fgl_lbvh L = *out ? *out : new fgl_lbvh_s();
  const bool fresh = *out == nullptr;
  cudaStream_t s = (cudaStream_t)stream;
  auto t0 = std::chrono::steady_clock::now();
  if (!L->status) {
    if (cudaMalloc(&L->status, sizeof(unsigned)) != cudaSuccess ||
        cudaMemset(L->status, 0, sizeof(unsigned)) != cudaSuccess) {
      if (fresh) delete L;
      return err(FGL_ERR_OOM, "cannot allocate the LBVH status word");
    }
  }
  L->built = false;  // from here on the arrays change: no casts until the build is through
  if (L->nt != nt) {
    for (void** b : {&L->nodes, &L->tris, &L->wnodes, &L->wtris}) {
      if (*b) cudaFree(*b);
      *b = nullptr;
    }
    L->nt = 0;
    cudaError_t e = cudaMalloc(&L->nodes, (size_t)std::max<int64_t>(1, nt - 1) * sizeof(LbvhNode));
    if (e == cudaSuccess) e = cudaMalloc(&L->tris, (size_t)nt * 48);
    if (e != cudaSuccess) {
      cudaGetLastError();
      for (void** b : {&L->nodes, &L->tris}) {
        if (*b) cudaFree(*b);
        *b = nullptr;
      }
      if (fresh) {
        cudaFree(L->status);
        delete L;
      }
      return err(FGL_ERR_OOM, "cannot allocate LBVH arrays");
    }
    L->nt = nt;
  }
  // scratch
  const size_t n_in = (size_t)std::max<int64_t>(1, nt - 1);
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off = al256(off + bytes); return o; };
  const size_t o_tbox = take((size_t)nt * 32), o_k0 = take((size_t)nt * 4), o_v0 = take((size_t)nt * 4),
               o_k1 = take((size_t)nt * 4), o_v1 = take((size_t)nt * 4), o_par = take((size_t)nt * 4),
               o_flags = take(n_in * 4), o_lbox = take((size_t)nt * 32),
               o_sort = take(radix_sort_tmp_elems(nt) * 4), o_split = take(n_in * 4),
               o_roots = take((size_t)nt * 8), o_wroot = take((size_t)wide_capacity(nt) * 16),
               o_bounds = take(sizeof(int) * (16 + kWideLevels));
  if (off > L->work_cap) {
    cudaStreamSynchronize(s);
    if (L->work) cudaFree(L->work);
    L->work = nullptr;
    L->work_cap = 0;
    if (cudaMalloc(&L->work, off) != cudaSuccess) {
      cudaGetLastError();
      if (fresh) fgl_lbvh_destroy(L);
      return err(FGL_ERR_OOM, "cannot allocate LBVH build scratch");
    }
    L->work_cap = off;
  }
  // The wide form is a third of the LBVH: a mesh that fits without it is built
  // without it, and its casts take the binary tree.
  if (!L->wnodes && (cudaMalloc(&L->wnodes, (size_t)wide_capacity(nt) * node_stride(8)) != cudaSuccess ||
                     cudaMalloc(&L->wtris, (size_t)nt * 48) != cudaSuccess)) {
    cudaGetLastError();
    if (L->wnodes) cudaFree(L->wnodes);
    L->wnodes = L->wtris = nullptr;
  }
  char* w = (char*)L->work;
  float4* tbox = (float4*)(w + o_tbox);
  uint32_t *k0 = (uint32_t*)(w + o_k0), *v0 = (uint32_t*)(w + o_v0), *k1 = (uint32_t*)(w + o_k1),
           *v1 = (uint32_t*)(w + o_v1);
  int32_t* par = (int32_t*)(w + o_par);
  uint32_t* flags = (uint32_t*)(w + o_flags);
  float4* nbox = tbox;  // the triangles' boxes are done with once gathered
  float4* lbox = (float4*)(w + o_lbox);
  int* bounds = (int*)(w + o_bounds);
  // words 0..6 the bounds, 7 the depth, 8 the status, 9 the block roots, 10 the
  // wide form's triangles, from 16 on its levels' nodes
  int init[16 + kWideLevels];
  for (int a = 0; a < 3; ++a) {
    init[a] = 0x7FFFFFFF;          // ford(+inf) and beyond
    init[3 + a] = (int)0x80000000; // below ford(-inf)
  }
  for (int a = 6; a < 16 + kWideLevels; ++a) init[a] = 0;
  int32_t* status = bounds + 8;
  LCUDA(cudaMemcpyAsync(bounds, init, sizeof(init), cudaMemcpyHostToDevice, s));
  LCUDA(cudaMemsetAsync(flags, 0, n_in * 4, s));
  int32_t* split = (int32_t*)(w + o_split);
  int2* roots = (int2*)(w + o_roots);
  int4* wroot = (int4*)(w + o_wroot);
  const int4 root = make_int4(0, 0, (int)nt, 0);  // wide node 0 is opened from the binary root
  LCUDA(cudaMemcpyAsync(wroot, &root, sizeof(root), cudaMemcpyHostToDevice, s));
  const unsigned gb = (unsigned)((nt + 255) / 256);
  k_lbvh_boxes<<<gb, 256, 0, s>>>(d_verts, nv, d_tris, nt, tbox, bounds, status);
  LCUDA(cudaGetLastError());
  k_lbvh_morton<<<gb, 256, 0, s>>>(tbox, nt, bounds, k0, v0);
  LCUDA(cudaGetLastError());
  int launches = 0;
  bool second = false;
  LCUDA(radix_sort_pairs(k0, v0, k1, v1, nt, 30, (uint32_t*)(w + o_sort), s, &launches, &second));
  if (second) {
    std::swap(k0, k1);
    std::swap(v0, v1);
  }
  k_lbvh_gather<<<gb, 256, 0, s>>>(d_verts, d_tris, nv, v0, tbox, nt, bounds, (float4*)L->tris, lbox);
  LCUDA(cudaGetLastError());
  if (nt > 1) {
    k_lbvh_karras<<<(unsigned)((nt + kLbvhBlock - 1) / kLbvhBlock), kLbvhBlock, 0, s>>>(
        k0, nt, (LbvhNode*)L->nodes, par, split, lbox, nbox, roots, bounds + 9);
    LCUDA(cudaGetLastError());
    const int64_t top = (nt + kLbvhBlock - 1) / kLbvhBlock * 16;  // a block's roots: about ten
    k_lbvh_top<<<(unsigned)std::min<int64_t>((top + 127) / 128, 152 * 16), 128, 0, s>>>(
        (LbvhNode*)L->nodes, par, flags, nbox, lbox, roots, bounds + 9, bounds + 7);
    LCUDA(cudaGetLastError());
  }
  if (L->wnodes) {
    WideArgs a{(const LbvhNode*)L->nodes, split, lbox, (const float4*)L->tris, nt, (uint8_t*)L->wnodes,
               (float4*)L->wtris, wroot, bounds + 10, bounds + 16, (int)wide_capacity(nt)};
    int dev = 0, sms = 0, per_sm = 0;
    LCUDA(cudaGetDevice(&dev));
    LCUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    LCUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lbvh_wide, 256, 0));
    // a small tree needs fewer blocks than fit
    const int64_t want = (wide_capacity(nt) + 63) / 64;
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sms * std::min(per_sm, 4)));
    void* args[] = {&a};
    LCUDA(cudaLaunchCooperativeKernel((const void*)k_lbvh_wide, dim3(blocks), dim3(256), args, 0, s));
  }
  int host[16 + kWideLevels];
  LCUDA(cudaMemcpyAsync(host, bounds, sizeof(host), cudaMemcpyDeviceToHost, s));
  LCUDA(cudaStreamSynchronize(s));
  const int32_t st = host[8];
  if (st) {
    if (fresh) fgl_lbvh_destroy(L);
    return err(FGL_ERR_INVALID, "a triangle has a vertex id out of range or a non-finite vertex");
  }
  for (int a = 0; a < 3; ++a) {
    L->lo[a] = iord(host[a]);
    L->hi[a] = iord(host[3 + a]);
  }
  L->margin = std::ldexp(std::max(1.f, iord(host[6])), -17);
  L->depth = nt > 1 ? host[7] : 1;
  L->n_wide = L->wnodes ? 1 : 0;
  for (int lv = 0; lv < kWideLevels; ++lv) L->n_wide += host[16 + lv];
  L->built = true;
  cudaGetDevice(&L->device);
  L->build_ms =
      (float)std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  *out = L;
  return FGL_OK;
}

extern "C" fgl_status fgl_lbvh_destroy(fgl_lbvh L) {
  if (!L) return FGL_OK;
  cudaDeviceSynchronize();
  for (void* b : {L->nodes, L->tris, L->wnodes, L->wtris})
    if (b) cudaFree(b);
  if (L->work) cudaFree(L->work);
  if (L->status) cudaFree(L->status);
  delete L;
  return FGL_OK;
}

extern "C" fgl_status fgl_lbvh_get_stats(fgl_lbvh L, fgl_lbvh_stats* o) {
  if (!L || !o) return err(FGL_ERR_INVALID, "null argument");
  o->n_tris = L->nt;
  o->n_nodes = L->nt > 1 ? L->nt - 1 : 0;
  o->depth = L->depth;
  o->build_ms = L->build_ms;
  unsigned st = 0;
  if (L->status) LCUDA(cudaMemcpy(&st, L->status, sizeof(st), cudaMemcpyDeviceToHost));
  o->overflow = (int32_t)((st & 1u) | ((st & 4u) ? 2u : 0u));
  o->margin = L->margin;
  for (int a = 0; a < 3; ++a) {
    o->centroid_lo[a] = L->lo[a];
    o->centroid_hi[a] = L->hi[a];
  }
  return FGL_OK;
}

extern "C" fgl_status fgl_lbvh_export(fgl_lbvh L, void* nodes, int64_t node_bytes, void* tris,
                                      int64_t tri_bytes) {
  if (!L) return err(FGL_ERR_INVALID, "null LBVH");
  if (!L->built) return err(FGL_ERR_INVALID, "the LBVH holds no tree: its last build failed");
  const int64_t nb = (L->nt > 1 ? L->nt - 1 : 0) * (int64_t)sizeof(LbvhNode), tb = L->nt * 48;
  if (nodes) {
    if (node_bytes != nb) return err(FGL_ERR_INVALID, "node_bytes mismatch");
    LCUDA(cudaMemcpy(nodes, L->nodes, nb, cudaMemcpyDeviceToHost));
  }
  if (tris) {
    if (tri_bytes != tb) return err(FGL_ERR_INVALID, "tri_bytes mismatch");
    LCUDA(cudaMemcpy(tris, L->tris, tb, cudaMemcpyDeviceToHost));
  }
  return FGL_OK;
}
