// Gaussian-to-occupancy conversion (paper Sec. IV-A): eq. D(v) on a voxel
// grid, restricted per tile to the tile's candidate Gaussians (eq. C_tile),
// then eqs. V_occ, Int and Surf.
//
// Pipeline (all on the caller's stream; one host synchronisation to size the
// pair buffers):
//   k_gauss_prep   per Gaussian: validity, the float32 candidate tile range
//                  (the exact operation sequence of fgl.h), the count of
//                  covered tiles, and the density parameters (mean, alpha^2,
//                  the inverse covariance pre-scaled for exp2);
//   scan           exclusive prefix sum of the counts -> pair offsets (sort.cu);
//   k_emit         (tile, Gaussian) pairs, in Gaussian order;
//   radix sort     stable LSD sort of the pairs by tile (8-bit digits, sort.cu), so
//                  every tile's candidates end up in increasing Gaussian
//                  index and the float32 sums are deterministic;
//   k_tile_bounds  begin/end of every tile's candidate run;
//   k_density<B>   one block per tile: each warp stages candidates in shared
//                  memory and sums them over the tile's x-rows, a row's voxels
//                  from three exponentials;
//   k_occ_surf     D > theta and the 6-neighbour surface test.
//
// The paper finds the candidates of a tile with an LBVH query over Gaussian
// AABBs (Karras); binning each Gaussian to the tiles its AABB covers gives
// the same candidate sets without building or traversing a tree.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <memory>
#include <mutex>
#include <string>
#include <unordered_map>
#include <vector>

#include "fgl.h"
#include "fgl_internal.h"
#include "nvtx_range.h"
#include "ptx_ops.cuh"
#include "sort.h"


using namespace fgl;

namespace {

constexpr float kHalfLog2e = 0.72134752044448170368f;  // log2(e) / 2

// Density parameters of one Gaussian, 48 bytes:
//   a = (mu_x, mu_y, mu_z, alpha^2)
//   b = (M00, M11, M22, M01), c = (M02, M12, valid, 0), M = -(log2 e / 2) * 2^[a!=b] Sigma^-1
// so that alpha^2 * exp(-q/2) = alpha^2 * exp2(M00 dx^2 + M11 dy^2 + M22 dz^2
//                                               + M01 dx dy + M02 dx dz + M12 dy dz).
struct GaussParams {
  float4 a, b, c;
};

struct TileRange {
  int lo[3], hi[3];
};

// Candidate tile range in float32, the operation sequence of fgl.h (no FMA).
__device__ __forceinline__ bool tile_range(const float* mu, const float* s, const float* q,
                                           const float o[3], float cell, int ntiles[3],
                                           TileRange& t, float R[3][3]) {
  for (int a = 0; a < 3; ++a)
    if (!isfinite(mu[a]) || !isfinite(s[a]) || !(s[a] > 0.0f)) return false;
  float w = q[0], x = q[1], y = q[2], z = q[3];
  float n2 = __fadd_rn(__fmul_rn(w, w), __fmul_rn(x, x));
  n2 = __fadd_rn(n2, __fmul_rn(y, y));
  n2 = __fadd_rn(n2, __fmul_rn(z, z));
  if (!(n2 > 0.0f) || !isfinite(n2)) return false;
  const float n = __fsqrt_rn(n2);
  w = __fdiv_rn(w, n);
  x = __fdiv_rn(x, n);
  y = __fdiv_rn(y, n);
  z = __fdiv_rn(z, n);
  const float xx = __fmul_rn(x, x), yy = __fmul_rn(y, y), zz = __fmul_rn(z, z);
  const float xy = __fmul_rn(x, y), xz = __fmul_rn(x, z), yz = __fmul_rn(y, z);
  const float wx = __fmul_rn(w, x), wy = __fmul_rn(w, y), wz = __fmul_rn(w, z);
  R[0][0] = __fsub_rn(1.0f, __fmul_rn(2.0f, __fadd_rn(yy, zz)));
  R[0][1] = __fmul_rn(2.0f, __fsub_rn(xy, wz));
  R[0][2] = __fmul_rn(2.0f, __fadd_rn(xz, wy));
  R[1][0] = __fmul_rn(2.0f, __fadd_rn(xy, wz));
  R[1][1] = __fsub_rn(1.0f, __fmul_rn(2.0f, __fadd_rn(xx, zz)));
  R[1][2] = __fmul_rn(2.0f, __fsub_rn(yz, wx));
  R[2][0] = __fmul_rn(2.0f, __fsub_rn(xz, wy));
  R[2][1] = __fmul_rn(2.0f, __fadd_rn(yz, wx));
  R[2][2] = __fsub_rn(1.0f, __fmul_rn(2.0f, __fadd_rn(xx, yy)));
  for (int a = 0; a < 3; ++a) {
    const float p0 = __fmul_rn(R[a][0], s[0]), p1 = __fmul_rn(R[a][1], s[1]),
                p2 = __fmul_rn(R[a][2], s[2]);
    float v = __fadd_rn(__fmul_rn(p0, p0), __fmul_rn(p1, p1));
    v = __fadd_rn(v, __fmul_rn(p2, p2));
    const float e = __fmul_rn(3.0f, __fsqrt_rn(v));
    const float lo = __fsub_rn(__fsub_rn(mu[a], e), o[a]);
    const float hi = __fsub_rn(__fadd_rn(mu[a], e), o[a]);
    const float flo = fminf(fmaxf(floorf(__fdiv_rn(lo, cell)), -1073741824.0f), 1073741824.0f);
    const float fhi = fminf(fmaxf(floorf(__fdiv_rn(hi, cell)), -1073741824.0f), 1073741824.0f);
    t.lo[a] = max((int)flo, 0);
    t.hi[a] = min((int)fhi, ntiles[a] - 1);
    if (t.lo[a] > t.hi[a]) return false;
  }
  return true;
}

struct GridArgs {
  float o[3];
  float h;
  float cell;
  int dims[3];
  int ntiles[3];
};

__global__ void k_gauss_prep(const float* __restrict__ mu, const float* __restrict__ scale,
                             const float* __restrict__ quat, const float* __restrict__ alpha,
                             int64_t n, GridArgs g, GaussParams* __restrict__ params,
                             int4* __restrict__ ranges, unsigned long long* __restrict__ counts) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float m[3], s[3], q[4];
  for (int a = 0; a < 3; ++a) {
    m[a] = mu[3 * i + a];
    s[a] = scale[3 * i + a];
  }
  for (int a = 0; a < 4; ++a) q[a] = quat[4 * i + a];
  TileRange t;
  float R[3][3];
  const bool ok = tile_range(m, s, q, g.o, g.cell, g.ntiles, t, R);
  GaussParams P;
  P.a = make_float4(m[0], m[1], m[2], 0.f);
  P.b = make_float4(0.f, 0.f, 0.f, 0.f);
  P.c = make_float4(0.f, 0.f, 0.f, 0.f);
  unsigned long long cnt = 0;
  int4 r0 = make_int4(0, 0, 0, 0), r1 = make_int4(-1, -1, -1, 0);
  if (ok) {
    const float al = alpha[i];
    P.a.w = al * al;
    // Sigma^-1 = R diag(1/s^2) R^T, times -(log2 e)/2, off-diagonals doubled
    const float i0 = 1.0f / (s[0] * s[0]), i1 = 1.0f / (s[1] * s[1]), i2 = 1.0f / (s[2] * s[2]);
    float M[3][3];
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b)
        M[a][b] = R[a][0] * R[b][0] * i0 + R[a][1] * R[b][1] * i1 + R[a][2] * R[b][2] * i2;
    const float k = -kHalfLog2e;
    P.b = make_float4(k * M[0][0], k * M[1][1], k * M[2][2], 2.f * k * M[0][1]);
    P.c = make_float4(2.f * k * M[0][2], 2.f * k * M[1][2], 1.f, 0.f);
    cnt = (unsigned long long)(t.hi[0] - t.lo[0] + 1) * (t.hi[1] - t.lo[1] + 1) *
          (t.hi[2] - t.lo[2] + 1);
    r0 = make_int4(t.lo[0], t.lo[1], t.lo[2], 0);
    r1 = make_int4(t.hi[0], t.hi[1], t.hi[2], 0);
  }
  params[i] = P;
  ranges[2 * i] = r0;
  ranges[2 * i + 1] = r1;
  counts[i] = cnt;
}

// ---------------------------------------------------------------------------
// pairs, stable radix sort by tile, tile bounds
// ---------------------------------------------------------------------------
// One warp per 32 consecutive Gaussians: the warp writes each Gaussian's
// pairs in turn with its 32 lanes, so the stores are contiguous and a
// Gaussian covering many tiles does not hold up its neighbours.  Each lane
// prepares its own Gaussian's range, reciprocals and place in shared memory, so
// the turns read two words instead of shuffling seven and dividing again.  Bound
// by issue: 720 k Gaussians, 19.4 M pairs 79 -> 50 us.
constexpr int kEmitWarps = 8;

struct __align__(16) EmitRange {
  int ex, ey, cnt, tile0;  // tiles along x and y, tiles, the first one
  float ix, iy;            // 1 / ex, 1 / ey
  unsigned long long off;
};

__global__ void __launch_bounds__(32 * kEmitWarps)
    k_emit(const int4* __restrict__ ranges, const unsigned long long* __restrict__ offs, int64_t n, GridArgs g,
           uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  __shared__ EmitRange s_range[kEmitWarps][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t g0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane);
  if (g0 >= n) return;
  const int64_t mine = g0 + lane;
  EmitRange e = {0, 0, 0, 0, 0.f, 0.f, 0ull};
  if (mine < n) {
    const int4 lo = ranges[2 * mine], hi = ranges[2 * mine + 1];
    const int ez = hi.z - lo.z + 1;
    e.ex = hi.x - lo.x + 1;
    e.ey = hi.y - lo.y + 1;
    e.cnt = e.ex <= 0 || e.ey <= 0 || ez <= 0 ? 0 : e.ex * e.ey * ez;
    e.tile0 = (lo.z * g.ntiles[1] + lo.y) * g.ntiles[0] + lo.x;
    e.ix = 1.0f / (float)e.ex;
    e.iy = 1.0f / (float)e.ey;
    e.off = offs[mine];
  }
  s_range[wid][lane] = e;
  __syncwarp();
  const int row = g.ntiles[0], plane = g.ntiles[0] * g.ntiles[1];
  for (int j = 0; j < 32; ++j) {
    const EmitRange r = s_range[wid][j];
    const uint32_t gid = (uint32_t)(g0 + j);
    uint32_t* k = keys + r.off;
    uint32_t* v = vals + r.off;
    for (int p = lane; p < r.cnt; p += 32) {
      // p / ex from the reciprocal: below 2^20 the quotient of p + 1/2 stays
      // off the integers by more than its rounding
      const int q = r.cnt <= (1 << 20) ? (int)(((float)p + 0.5f) * r.ix) : p / r.ex;
      const int c = r.cnt <= (1 << 20) ? (int)(((float)q + 0.5f) * r.iy) : q / r.ey;
      k[p] = (uint32_t)(r.tile0 + c * plane + (q - c * r.ey) * row + (p - q * r.ex));
      v[p] = gid;
    }
  }
}

// begin/end of every tile's run in the sorted keys.  A warp finds its tile's
// first key by 32-way search: each step is one round of loads, so 87 M keys
// take six instead of a pass over all of them (a tenth of its time on the
// 19 M keys of 10,304 tiles).
__global__ void k_tile_bounds(const uint32_t* __restrict__ keys, int64_t n, int64_t n_tiles,
                              uint32_t* __restrict__ begin, uint32_t* __restrict__ end) {
  const int lane = threadIdx.x & 31;
  const int64_t tile = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (tile > n_tiles) return;  // warp n_tiles finds the end of the last tile
  int64_t lo = 0, len = n;     // the first key >= tile lies in [lo, lo + len]
  while (len > 0) {
    const int64_t step = (len + 31) / 32, at = lo + (lane + 1) * step - 1;
    const unsigned less = __ballot_sync(0xFFFFFFFFu, at < lo + len && keys[at] < (uint32_t)tile);
    const int64_t skip = (int64_t)__popc(less) * step;
    const int64_t left = len - skip;
    lo += skip;
    len = left < step ? left : step - 1;
  }
  if (lane == 0) {
    if (tile < n_tiles) begin[tile] = (uint32_t)lo;
    if (tile > 0) end[tile - 1] = (uint32_t)lo;
  }
}

// ---------------------------------------------------------------------------
// density: one block per tile of B^3 voxels.  Each warp of the block sums
// every S-th batch of 32 candidates over the whole tile (two x-rows a lane, so
// that a staged candidate is read once for 64 rows); the warps' sums are added
// in warp order.  In a grid of few tiles, one of more than 2 x 32 S candidates is
// shared by the K blocks of a cluster, whose sums the first adds in block order
// (the others of a smaller tile leave at once).  Bound by instruction issue and the FMA pipe about equally
// (32 warp instructions for a candidate and 32 rows, counted over a launch, of which
// 3 exponentials; one exponential a voxel took 40, and 8 of them held the MUFU pipe
// longest).
// 720 k Gaussians, 10,304 tiles of 2.5 cm voxels: 2.16 ms with one exponential a
// voxel, 1.41 so; 85 k Gaussians, 630 tiles of 5 cm, up to 11,400 candidates a
// tile: 0.67 and 0.11 ms (the least of eight 0.670 and 0.109).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// A row's exponent is a parabola in x: about the row's middle xm,
//   q(xm + d) = q(xm) + g d + M00 d^2,
// so its B values are E P^j c_j with E = 2^q(xm), P = 2^(g h / 2) and
// c_j = alpha^2 2^(M00 (j h / 2)^2), j = +-1, +-3, .. the voxel's distance
// from the middle in half voxels: three exponentials a row (E, P, 1 / P) and
// two packed operations a voxel pair instead of one exponential a voxel.
// Taken when the parabola falls by at most 2^kRowFall from the middle to the
// end of the row: E P^j then stays below 2^kRowFall, and where E underflows
// (below 2^-126) the row's largest value is below 2^-45.  P^2 has to stay
// finite too (|g h / 2| <= kRowSlope), so that a row far from the Gaussian adds
// 0 and not 0 times infinity; a Gaussian that would widen the band below too far
// (kMaxSpread) or whose alpha^2 is above kMaxWeight is left out as well.  A Gaussian
// outside these limits (steep) is evaluated voxel by voxel.
constexpr float kRowFall = 20.f, kRowSlope = 60.f;

// Voxels whose density may lie on either side of theta, depending on the rounding
// of the factored form and of the warps' partial sums, are summed again voxel by
// voxel in candidate order, so that the masks are those of that sum to the last
// bit.  Steep Gaussians' terms are that sum's, bit for bit.  A factored term's
// exponent differs from that sum's by at most u = 2^-24 times
//   14.4 X G + 6 Q + 150,   X = |dx|, G = |M01| |dy| + |M02| |dz| + 2 |M00| |dx|,
//                           Q = |M11| dy^2 + |M12 dy dz| + |M22| dz^2,
// each at its largest over the tile: roundings of xm and dx (1 and 4 u X, each times
// the slope G), of the x coefficient (2 and 3 u G, times X), of the slope's up to B - 1
// half voxels and the middle's value (35 u G h / 2, 15 for B = 4, where X >= B h / 2), of
// the y/z part (3 u Q in each form) and of the sums (exponents to -64 and the middle's
// 84 beyond the slope; smaller terms are below the slack).  The exponentials and
// products add 5e-6.  Sums of n
// positive terms in candidate order and in N parts err by at most n u and n u / N
// (and kBand covers the parts' own sum).  So the band is
//   kBand + (1 + 1 / N) n u + max over the tile's factored Gaussians of u (10.5 X G + 4.5 Q)
// relative, and 2^-44 kMaxWeight a candidate absolute for rows whose middle flushes.
// On 60 k to 90 k Gaussians of 1 to 20 cm at 2.5 to 5 cm voxels the band is about
// 7e-4 (one tile in 14 to 50 has a voxel in it) and kMaxSpread makes 1-4% of the
// factored Gaussians steep; twice that, up to 0.4%.  A tile of many candidates with
// such a voxel can hold up a grid of few tiles (29 k Gaussians, 120 tiles: the call 120
// us, 141 at twice that), and so do steep Gaussians (243 k: 301 us, 308 at a third).
constexpr float kUnit = 5.9604645e-8f;  // u
constexpr float kBand = 2e-5f, kMaxSpread = 6e-4f, kMaxWeight = 4.f;
constexpr int kCloseAtOnce = 8;

// One staged candidate.  bx = M01 dy + M02 dz is the x coefficient and
// syz = M11 dy^2 + M12 dy dz + M22 dz^2 the y/z part of the exponent.
struct __align__(16) StagedGauss {
  float4 at;     // dY, dZ (tile corner minus mean), xm, M00 xm; steep: dX in z, 0 in w
  float4 m;      // M11, M22, M12, M01
  float4 n;      // M02, M00 xm h / 2, alpha^2, M00
  float4 c[2];   // c_1, c_1, c_3, c_3 | c_5, c_5, c_7, c_7
};

template <int B>
struct DensityCfg {
  static constexpr int ROWS = B * B;
  static constexpr int LANES = ROWS / 2;    // lanes that cover the tile, two rows each
  static constexpr int SUB = 32 / LANES;    // candidates a warp takes at once
};

template <int B, int S, int K>
__global__ void __launch_bounds__(32 * S)
    k_density(const GaussParams* __restrict__ params, const uint32_t* __restrict__ cand,
              const uint32_t* __restrict__ begin, const uint32_t* __restrict__ end, GridArgs g, float theta,
              float max_spread, float* __restrict__ out) {
  using C = DensityCfg<B>;
  constexpr int NT = 32 * S;
  namespace cg = cooperative_groups;
  constexpr int kRow = NT + 4;  // a voxel's terms of a batch of NT candidates, on banks of their own
  __shared__ union {
    StagedGauss batch[S][32];
    float terms[2][1 + kCloseAtOnce][kRow];  // alpha^2, then 2^q of each voxel
  } sh;
  __shared__ float s_sum[S > 1 ? S - 1 : 1][C::ROWS * B];
  const unsigned FULL = 0xFFFFFFFFu;
  const int tile = blockIdx.x / K, rank = blockIdx.x % K;
  const int tx = tile % g.ntiles[0], ty = (tile / g.ntiles[0]) % g.ntiles[1],
            tz = tile / (g.ntiles[0] * g.ntiles[1]);
  const uint32_t b0 = begin[tile], b1 = end[tile];
  // the tile's batches go round the warps of one block or of the whole cluster
  const bool split = K > 1 && b1 - b0 > 2 * NT;
  if (K > 1 && !split && rank > 0) return;  // all of the cluster's blocks agree
  if (K == 1 && b0 == b1) {  // nobody's tile: most of a sparse grid's
    for (int v = threadIdx.x; v < C::ROWS * B; v += NT) {
      const int x = tx * B + v % B, vy = ty * B + v / B % B, vz = tz * B + v / (B * B);
      if (x < g.dims[0] && vy < g.dims[1] && vz < g.dims[2])
        out[((int64_t)vz * g.dims[1] + vy) * g.dims[0] + x] = 0.f;
    }
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t first = b0 + 32 * (split ? rank * S + warp : warp), stride = split ? 32 * S * K : 32 * S;
  const int slot = lane % C::LANES, sub = lane / C::LANES, y = slot % B, z = slot / B;  // rows (y, z), (y, z + B / 2)
  StagedGauss* st = sh.batch[warp];
  // tile corner in FP64 (the offsets to the means are formed there, then
  // rounded once: |tile corner - mu| is small, so the float offset is accurate)
  const double cx = (double)g.o[0] + (double)(tx * B) * (double)g.h;
  const double cy = (double)g.o[1] + (double)(ty * B) * (double)g.h;
  const double cz = (double)g.o[2] + (double)(tz * B) * (double)g.h;
  const double mid = (double)(B / 2) * (double)g.h;
  const float hh = 0.5f * g.h, end_d = (float)(B - 1) * hh;
  const float jy = (float)y + 0.5f, jz[2] = {(float)z + 0.5f, (float)(z + B / 2) + 0.5f};
  uint64_t acc[2][B / 2];  // voxel pairs mirrored about the row's middle, innermost first
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int p = 0; p < B / 2; ++p) acc[r][p] = 0ull;
  // a batch's parameters travel while the one before it is summed, its
  // candidate numbers one batch earlier
  GaussParams P = {};
  uint32_t next = 0;
  float spread = 0.f;  // the largest u (10.5 X G + 4.5 Q) of the lane's factored candidates
  if (first + lane < b1) P = params[cand[first + lane]];
  if (first + stride + lane < b1) next = cand[first + stride + lane];
  for (uint32_t c0 = first; c0 < b1; c0 += stride) {
    __syncwarp();  // the batch before this one is summed
    const bool valid = c0 + lane < b1;
    const float dX = (float)(cx - (double)P.a.x), dY = (float)(cy - (double)P.a.y), dZ = (float)(cz - (double)P.a.z);
    // the offsets' magnitudes over the tile's voxels, from above
    const float edge = (float)B * g.h;
    const float X = fmaxf(fabsf(dX), fabsf(dX + edge)), Y = fmaxf(fabsf(dY), fabsf(dY + edge)),
                Z = fmaxf(fabsf(dZ), fabsf(dZ + edge));
    const float G = fabsf(P.b.w) * Y + fabsf(P.c.x) * Z + 2.f * fabsf(P.b.x) * X, slope = hh * G;  // |g h / 2| at most: P^2 stays finite
    const float Q = fabsf(P.b.y) * (Y * Y) + fabsf(P.c.y) * (Y * Z) + fabsf(P.b.z) * (Z * Z);
    const float d_spread = kUnit * (10.5f * (X * G) + 4.5f * Q);
    const bool fast = valid && fabsf(P.b.x) * (end_d * end_d) <= kRowFall && slope <= kRowSlope &&
                      d_spread <= max_spread && P.a.w <= kMaxWeight;
    if (fast) spread = fmaxf(spread, d_spread);
    // the factored ones first, steep ones from the end
    const unsigned fm = __ballot_sync(FULL, fast), sm = __ballot_sync(FULL, valid && !fast);
    const unsigned below = (1u << lane) - 1u;
    const int nf = __popc(fm), ns = __popc(sm);
    if (valid) {
      StagedGauss& q = st[fast ? __popc(fm & below) : 31 - __popc(sm & below)];
      const float xm = (float)((cx + (fast ? mid : 0.0)) - (double)P.a.x), u = fast ? P.b.x * xm : 0.f;
      q.at = make_float4(dY, dZ, xm, u);
      q.m = make_float4(P.b.y, P.b.z, P.c.y, P.b.w);
      q.n = make_float4(P.c.x, u * hh, P.a.w, P.b.x);
      if (fast) {
        const float k1 = P.b.x * hh * hh;
        const float c1 = P.a.w * exp2f(k1), c3 = P.a.w * exp2f(9.f * k1), c5 = P.a.w * exp2f(25.f * k1),
                    c7 = P.a.w * exp2f(49.f * k1);
        q.c[0] = make_float4(c1, c1, c3, c3);
        q.c[1] = make_float4(c5, c5, c7, c7);
      }
    }
    __syncwarp();
    if (c0 + stride + lane < b1) P = params[next];
    if (c0 + 2 * stride + lane < b1) next = cand[c0 + 2 * stride + lane];
#pragma unroll 1
    for (int i = sub; i < nf; i += C::SUB) {
      const float4 at = st[i].at, m = st[i].m, n = st[i].n;
      const float4 w0 = st[i].c[0], w1 = st[i].c[1];
      const float dy = __fmaf_rn(jy, g.h, at.x);
      const float ay = (m.x * dy) * dy, by = fmaf(m.w, dy, at.w);
      uint64_t t2[2], PP[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float dz = __fmaf_rn(jz[r], g.h, at.y);
        const float a = fmaf(n.x, dz, by);
        const float qm = fmaf(a, at.z, fmaf(fmaf(m.z, dy, m.y * dz), dz, ay));
        const float gh = fmaf(a, hh, n.y);
        const float E = dev::ex2_approx(qm), Pl = dev::ex2_approx(-gh), Pr = dev::ex2_approx(gh);
        t2[r] = dev::pack2f(E * Pl, E * Pr);
        PP[r] = dev::pack2f(Pl * Pl, Pr * Pr);
      }
#pragma unroll
      for (int p = 0; p < B / 2; ++p) {
        const float4 w = p < 2 ? w0 : w1;
        const uint64_t w2 = (p & 1) ? dev::pack2f(w.z, w.w) : dev::pack2f(w.x, w.y);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          if (p) t2[r] = mul2(t2[r], PP[r]);
          acc[r][p] = dev::ffma2(t2[r], w2, acc[r][p]);
        }
      }
    }
#pragma unroll 1
    for (int i = 31 - sub; i > 31 - ns; i -= C::SUB) {
      const float4 at = st[i].at, m = st[i].m, n = st[i].n;
      const float dy = __fmaf_rn(jy, g.h, at.x);
      const uint64_t M002 = dev::pack2f(n.w, n.w), dX2 = dev::pack2f(at.z, at.z), a22 = dev::pack2f(n.z, n.z);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        // the operations of the voxel-by-voxel sum below, one by one
        const float dz = __fmaf_rn(jz[r], g.h, at.y);
        const float syz = __fmaf_rn(__fmaf_rn(m.x, dy, __fmul_rn(m.z, dz)), dy, __fmul_rn(__fmul_rn(m.y, dz), dz));
        const float bx = __fmaf_rn(m.w, dy, __fmul_rn(n.x, dz));
        const uint64_t bx2 = dev::pack2f(bx, bx), syz2 = dev::pack2f(syz, syz);
#pragma unroll
        for (int p = 0; p < B / 2; ++p) {
          const uint64_t dx2 =
              add2(dX2, dev::pack2f(__fmul_rn((float)(B / 2 - 1 - p) + 0.5f, g.h), __fmul_rn((float)(B / 2 + p) + 0.5f, g.h)));
          float q0, q1;
          dev::unpack2f(dev::ffma2(dev::ffma2(M002, dx2, bx2), dx2, syz2), q0, q1);  // <= 0
          acc[r][p] = dev::ffma2(a22, dev::pack2f(dev::ex2_approx(q0), dev::ex2_approx(q1)), acc[r][p]);
        }
      }
    }
  }
  __shared__ float s_band[K * S];  // the warps' largest spread (non-negative floats order as integers)
  spread = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(spread)));
  if (lane == 0) s_band[warp] = spread;
  float d[2][B];  // the rows' densities, complete in warp 0's lanes of sub 0
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int p = 0; p < B / 2; ++p) dev::unpack2f(acc[r][p], d[r][B / 2 - 1 - p], d[r][B / 2 + p]);
#pragma unroll
  for (int o = C::LANES; o < 32; o <<= 1)
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int i = 0; i < B; ++i) d[r][i] += __shfl_xor_sync(FULL, d[r][i], o);
  if (S > 1) {
    if (warp > 0 && sub == 0) {
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int i = 0; i < B; ++i) s_sum[warp - 1][(r * B + i) * C::LANES + slot] = d[r][i];
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll 1
      for (int v = 0; v + 1 < S; ++v)
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int i = 0; i < B; ++i) d[r][i] += s_sum[v][(r * B + i) * C::LANES + slot];
    }
  }
  if (K > 1 && split) {  // rank 0 adds the blocks' sums in rank order
    __shared__ float s_part[C::ROWS * B];
    cg::cluster_group cl = cg::this_cluster();
    if (warp == 0 && sub == 0) {
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int i = 0; i < B; ++i) s_part[(r * B + i) * C::LANES + slot] = d[r][i];
    }
    cl.sync();
    if (rank == 0) {
      for (int v = threadIdx.x; v < C::ROWS * B; v += NT) {
        float part[K];
#pragma unroll
        for (int k = 1; k < K; ++k) part[k] = *cl.map_shared_rank(s_part + v, k);
        float sum = s_part[v];
#pragma unroll
        for (int k = 1; k < K; ++k) sum += part[k];
        s_part[v] = sum;  // read by nobody else
      }
      for (int t = S + threadIdx.x; t < K * S; t += NT) s_band[t] = *cl.map_shared_rank(s_band + t % S, t / S);
    }
    cl.sync();  // and the others' memory stays until it is read
    if (rank > 0) return;
    if (warp == 0 && sub == 0) {
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int i = 0; i < B; ++i) d[r][i] = s_part[(r * B + i) * C::LANES + slot];
    }
  }
  const int gx = tx * B, gy = ty * B + y;
  const bool owner = warp == 0 && sub == 0 && gy < g.dims[1];
  // the tile's densities; the voxels in theta's band are then listed and summed
  // again, kCloseAtOnce at a time: their terms a candidate a thread, each
  // voxel's sum a lane's, in candidate order
  __shared__ uint16_t s_close[C::ROWS * B];
  __shared__ int s_n_close;
  if (threadIdx.x == 0) s_n_close = 0;
  __syncthreads();
  if (owner) {
    float band = 0.f;
    for (int t = 0; t < (split ? K * S : S); ++t) band = fmaxf(band, s_band[t]);
    const float n = (float)(b1 - b0), slack = n * (max_spread < 0.f ? 0x1p-148f : kMaxWeight * 0x1p-44f);
    band += kBand + (1.f + 1.f / (float)(C::SUB * S * (split ? K : 1))) * kUnit * n;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int gz = tz * B + z + r * (B / 2);
      if (gz >= g.dims[2]) break;
      float* dst = out + ((int64_t)gz * g.dims[1] + gy) * g.dims[0];
#pragma unroll
      for (int i = 0; i < B; ++i) {
        if (gx + i >= g.dims[0]) break;
        dst[gx + i] = d[r][i];
        // theta <= 0: a density above it is one in any order
        if (theta > 0.f && fabsf(d[r][i] - theta) <= band * fmaxf(d[r][i], theta) + slack)
          s_close[atomicAdd(&s_n_close, 1)] = (uint16_t)(((z + r * (B / 2)) * B + y) * B + i);
      }
    }
  }
  __syncthreads();
  const int n_close = s_n_close;
  for (int v0 = 0; v0 < n_close; v0 += kCloseAtOnce) {
    const int n = min(kCloseAtOnce, n_close - v0);
    float sum = 0.f;
    // a batch's parameters travel while the one before it is summed, its
    // candidate numbers one batch earlier
    GaussParams Q = {};
    uint32_t ahead = 0;
    if (b0 + threadIdx.x < b1) Q = params[cand[b0 + threadIdx.x]];
    if (b0 + NT + threadIdx.x < b1) ahead = cand[b0 + NT + threadIdx.x];
    int buf = 0;
    for (uint32_t c0 = b0; c0 < b1; c0 += NT, buf ^= 1) {
      const bool some = c0 + threadIdx.x < b1;
      const float ex = (float)(cx - (double)Q.a.x), ey = (float)(cy - (double)Q.a.y), ez = (float)(cz - (double)Q.a.z);
      sh.terms[buf][0][threadIdx.x] = some ? Q.a.w : 0.f;
#pragma unroll 1
      for (int v = 0; v < n; ++v) {
        const int at = s_close[v0 + v];
        // x rounded in two steps and y, z in one, as voxel by voxel sums always
        // were: the masks at theta stay what they are to the last bit
        const float dx = __fadd_rn(ex, __fmul_rn((float)(at % B) + 0.5f, g.h)),
                    dy = __fmaf_rn((float)(at / B % B) + 0.5f, g.h, ey),
                    dz = __fmaf_rn((float)(at / (B * B)) + 0.5f, g.h, ez);
        const float syz = fmaf(fmaf(Q.b.y, dy, __fmul_rn(Q.c.y, dz)), dy, __fmul_rn(__fmul_rn(Q.b.z, dz), dz));
        const float bx = fmaf(Q.b.w, dy, __fmul_rn(Q.c.x, dz));
        sh.terms[buf][1 + v][threadIdx.x] = some ? dev::ex2_approx(fmaf(fmaf(Q.b.x, dx, bx), dx, syz)) : 0.f;
      }
      if (c0 + NT + threadIdx.x < b1) Q = params[ahead];
      if (c0 + 2 * NT + threadIdx.x < b1) ahead = cand[c0 + 2 * NT + threadIdx.x];
      __syncthreads();  // and the batch before this one is summed
      if (threadIdx.x < (unsigned)n) {
#pragma unroll 4
        for (int k = 0; k < NT; k += 4) {
          const float4 w = *reinterpret_cast<const float4*>(&sh.terms[buf][0][k]);
          const float4 e = *reinterpret_cast<const float4*>(&sh.terms[buf][1 + threadIdx.x][k]);
          sum = fmaf(w.w, e.w, fmaf(w.z, e.z, fmaf(w.y, e.y, fmaf(w.x, e.x, sum))));
        }
      }
    }
    if (threadIdx.x < (unsigned)n) {  // over the owner's store, a barrier ago
      const int at = s_close[v0 + threadIdx.x];
      out[((int64_t)(tz * B + at / (B * B)) * g.dims[1] + ty * B + at / B % B) * g.dims[0] + gx + at % B] = sum;
    }
    __syncthreads();
  }
}

template <int B, int S, int K>
cudaError_t launch_density(int64_t n_tiles, const GaussParams* params, const uint32_t* cand, const uint32_t* begin,
                           const uint32_t* end, const GridArgs& g, float theta, float max_spread, float* out,
                           cudaStream_t s) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = K;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(n_tiles * K));
  cfg.blockDim = dim3(32 * S);
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = K > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_density<B, S, K>, params, cand, begin, end, g, theta, max_spread, out);
}

// eqs. V_occ, Int, Surf: a warp 32 voxels of a row, a block eight rows of a
// plane (planes and row groups past the grid limits in a stride loop); an
// occupied voxel loads its six neighbours at once.  One voxel a thread, so
// that all loads of the grid are in flight (a loop over rows took 31 us on
// 5.1 M voxels).
constexpr int kOccRows = 8;

__global__ void __launch_bounds__(32 * kOccRows) k_occ_surf(const float* __restrict__ D, GridArgs g, float theta,
                                                            uint8_t* __restrict__ occ, uint8_t* __restrict__ surf) {
  const int nx = g.dims[0], ny = g.dims[1], nz = g.dims[2];
  const int x = blockIdx.x * 32 + threadIdx.x;
  if (x >= nx) return;
  const int64_t plane = (int64_t)nx * ny;
  for (int z = blockIdx.z; z < nz; z += gridDim.z) {
    for (int y = blockIdx.y * kOccRows + threadIdx.y; y < ny; y += gridDim.y * kOccRows) {
      const int64_t i = z * plane + (int64_t)y * nx + x;
      const bool o = D[i] > theta;
      bool interior = false;
      if (o) {
        const bool xm = x > 0 && D[i - 1] > theta;
        const bool xp = x + 1 < nx && D[i + 1] > theta;
        const bool ym = y > 0 && D[i - nx] > theta;
        const bool yp = y + 1 < ny && D[i + nx] > theta;
        const bool zm = z > 0 && D[i - plane] > theta;
        const bool zp = z + 1 < nz && D[i + plane] > theta;
        interior = xm && xp && ym && yp && zm && zp;
      }
      if (occ) occ[i] = o ? 1 : 0;
      if (surf) surf[i] = (o && !interior) ? 1 : 0;
    }
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct Scratch {
  int device = -1;
  void* params = nullptr;
  size_t params_cap = 0;
  void* ranges = nullptr;
  size_t ranges_cap = 0;
  void* counts = nullptr;
  size_t counts_cap = 0;
  void* sums = nullptr;
  size_t sums_cap = 0;
  void* pairs = nullptr;  // keys, vals, keys', vals'
  size_t pairs_cap = 0;
  void* hist = nullptr;
  size_t hist_cap = 0;
  void* bounds = nullptr;
  size_t bounds_cap = 0;
  cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
  std::mutex mu;
};
std::mutex g_scr_mu;
std::unordered_map<uint64_t, std::unique_ptr<Scratch>> g_scr;

Scratch* get_scratch(cudaStream_t s) {
  int dev = 0;
  cudaGetDevice(&dev);
  const uint64_t key = (uint64_t)(uintptr_t)s ^ ((uint64_t)dev << 56);
  std::lock_guard<std::mutex> lk(g_scr_mu);
  auto& p = g_scr[key];
  if (!p) {
    p.reset(new Scratch());
    p->device = dev;
  }
  return p.get();
}

// grow a device buffer (contents not preserved); synchronises the stream first
cudaError_t ensure(void** buf, size_t* cap, size_t bytes, cudaStream_t s) {
  if (bytes <= *cap) return cudaSuccess;
  cudaError_t e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e;
  if (*buf) cudaFree(*buf);
  *buf = nullptr;
  *cap = 0;
  const size_t nb = std::max<size_t>(bytes + bytes / 4, 1 << 16);
  e = cudaMalloc(buf, nb);
  if (e != cudaSuccess) {
    *buf = nullptr;
    return e;
  }
  *cap = nb;
  return cudaSuccess;
}

fgl_status err(int status, const std::string& msg) {
  record_error(status, msg.c_str());
  return (fgl_status)status;
}

fgl_status cuda_err(cudaError_t e, const char* what) {
  return err(FGL_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

#define DCUDA(call)                                   \
  do {                                                \
    cudaError_t e_ = (call);                          \
    if (e_ != cudaSuccess) return cuda_err(e_, #call); \
  } while (0)

}  // namespace

extern "C" fgl_status fgl_gaussian_density(const fgl_gaussians* gs, const fgl_grid* grid,
                                           float theta, float* out_density, uint8_t* out_occ,
                                           uint8_t* out_surf, fgl_density_stats* stats,
                                           fgl_stream stream) {
  fgl::NvtxRange range("fgl_gaussian_density");
  if (!gs || !grid) return err(FGL_ERR_INVALID, "null gaussians or grid");
  if (gs->n < 0) return err(FGL_ERR_INVALID, "n < 0");
  if (gs->n > 0 && (!gs->mu || !gs->scale || !gs->quat || !gs->opacity))
    return err(FGL_ERR_INVALID, "null Gaussian parameter pointer");
  if (gs->n >= ((int64_t)1 << 32)) return err(FGL_ERR_INVALID, "too many Gaussians (max 2^32 - 1)");
  if (!out_density) return err(FGL_ERR_INVALID, "out_density is null");
  const int B = grid->tile ? grid->tile : 8;
  if (B != 4 && B != 8) return err(FGL_ERR_INVALID, "tile must be 4 or 8");
  if (!(std::isfinite(grid->h) && grid->h > 0.f)) return err(FGL_ERR_INVALID, "h must be finite and > 0");
  for (int a = 0; a < 3; ++a) {
    if (grid->dims[a] < 1) return err(FGL_ERR_INVALID, "grid dims must be >= 1");
    if (!std::isfinite(grid->origin[a])) return err(FGL_ERR_INVALID, "grid origin must be finite");
  }
  if (!std::isfinite(theta)) return err(FGL_ERR_INVALID, "theta must be finite");
  GridArgs g;
  for (int a = 0; a < 3; ++a) {
    g.o[a] = grid->origin[a];
    g.dims[a] = grid->dims[a];
    g.ntiles[a] = (grid->dims[a] + B - 1) / B;
  }
  g.h = grid->h;
  g.cell = (float)B * grid->h;
  const int64_t n_vox = (int64_t)g.dims[0] * g.dims[1] * g.dims[2];
  const int64_t n_tiles = (int64_t)g.ntiles[0] * g.ntiles[1] * g.ntiles[2];
  if (n_tiles >= ((int64_t)1 << 31)) return err(FGL_ERR_INVALID, "grid has too many tiles");
  cudaStream_t s = (cudaStream_t)stream;
  Scratch& S = *get_scratch(s);
  std::lock_guard<std::mutex> lk(S.mu);
  const int64_t n = gs->n;
  const bool timing = stats && stats->timing == 1;
  int launches = 0;
  if (timing && !S.ev[0]) {
    for (int k = 0; k < 4; ++k) DCUDA(cudaEventCreate(&S.ev[k]));
  }
  if (timing) DCUDA(cudaEventRecord(S.ev[0], s));

  DCUDA(ensure(&S.bounds, &S.bounds_cap, (size_t)n_tiles * 2 * sizeof(uint32_t), s));
  uint32_t* begin = (uint32_t*)S.bounds;
  uint32_t* end = begin + n_tiles;

  uint64_t n_pairs = 0;
  if (n > 0) {
    DCUDA(ensure(&S.params, &S.params_cap, (size_t)n * sizeof(GaussParams), s));
    DCUDA(ensure(&S.ranges, &S.ranges_cap, (size_t)n * 2 * sizeof(int4), s));
    DCUDA(ensure(&S.counts, &S.counts_cap, (size_t)(n + 1) * sizeof(unsigned long long), s));
    const size_t tmp_g = scan_tmp_elems(n + 1);
    DCUDA(ensure(&S.sums, &S.sums_cap, tmp_g * sizeof(unsigned long long), s));
    GaussParams* params = (GaussParams*)S.params;
    int4* ranges = (int4*)S.ranges;
    unsigned long long* counts = (unsigned long long*)S.counts;
    const unsigned gb = (unsigned)((n + 255) / 256);
    k_gauss_prep<<<gb, 256, 0, s>>>(gs->mu, gs->scale, gs->quat, gs->opacity, n, g, params, ranges,
                                    counts);
    ++launches;
    DCUDA(cudaGetLastError());
    DCUDA(cudaMemsetAsync(counts + n, 0, sizeof(unsigned long long), s));
    DCUDA(scan_exclusive_u64(counts, n + 1, (unsigned long long*)S.sums, tmp_g, s, &launches));
    DCUDA(cudaMemcpyAsync(&n_pairs, counts + n, sizeof(n_pairs), cudaMemcpyDeviceToHost, s));
    DCUDA(cudaStreamSynchronize(s));
    if (n_pairs >= ((uint64_t)1 << 31))
      return err(FGL_ERR_INVALID, "too many (Gaussian, tile) pairs (max 2^31 - 1): use a larger tile or voxel");
  }
  if (n_pairs > 0) {
    DCUDA(ensure(&S.pairs, &S.pairs_cap, (size_t)n_pairs * 4 * sizeof(uint32_t), s));
    uint32_t* k0 = (uint32_t*)S.pairs;
    uint32_t* v0 = k0 + n_pairs;
    uint32_t* k1 = v0 + n_pairs;
    uint32_t* v1 = k1 + n_pairs;
    const unsigned gb = (unsigned)((n + 255) / 256);
    k_emit<<<gb, 32 * kEmitWarps, 0, s>>>((const int4*)S.ranges, (const unsigned long long*)S.counts, n, g, k0,
                              v0);
    ++launches;
    DCUDA(cudaGetLastError());
    // stable LSD radix sort by tile id
    int bits = 1;
    while (((int64_t)1 << bits) < n_tiles) ++bits;
    DCUDA(ensure(&S.hist, &S.hist_cap, radix_sort_tmp_elems((int64_t)n_pairs) * sizeof(uint32_t), s));
    bool second = false;
    DCUDA(radix_sort_pairs(k0, v0, k1, v1, (int64_t)n_pairs, bits, (uint32_t*)S.hist, s, &launches,
                           &second));
    if (second) {
      k0 = k1;
      v0 = v1;
    }
    k_tile_bounds<<<(unsigned)((n_tiles + 1 + 7) / 8), 256, 0, s>>>(k0, (int64_t)n_pairs, n_tiles, begin, end);
    ++launches;
    DCUDA(cudaGetLastError());
    if (timing) DCUDA(cudaEventRecord(S.ev[1], s));
    // Warps a tile, by the mean of its candidates (wall time of the call, us):
    //   candidates a tile          0.1    5   16   53  211  729 1885    5, half of them within 10 cm
    //   two warps                  816  393  457  643 1547  541         776
    //   four                       917  553  581  727 1473  522 1828    648
    //   eight                                   1152 1603  529 1815
    //   four in each of two
    //   blocks, a cluster         1275  895  919 1182 2494  566 1877    852
    //   (two warps that share every candidate, one exponential a voxel:
    //                             1155  411  464  827 2216  782 2940    838)
    // over 262,144 tiles with 2,000 Gaussians, 62,500 with 20 k to 800 k, 6,500 and
    // 10,304 dense ones: two warps for a sparse grid, eight for a dense one, whose
    // heaviest tiles they even out best (5,000 tiles of 400 k Gaussians 790 us, four
    // 828).  A grid of fewer than 16 tiles an SM takes eight warps in four blocks, or
    // its heaviest tiles would run on alone (630 tiles: the call 0.54 ms in one block,
    // 0.49 in two, 0.475 in four or eight).  Tiles of 4^3 voxels have fewer candidates
    // each: one block of one warp where there are many (25,000 tiles: 1.60 ms; two
    // blocks 2.33).
    const GaussParams* params = (const GaussParams*)S.params;
    const bool few = n_tiles < 152 * 16;
    // where theta is as small as what flushed rows leave out (or 0: any density
    // counts), every Gaussian is summed voxel by voxel
    const float max_spread = theta >= 0.f && theta < 0x1p-30f ? -1.f : kMaxSpread;
    const int64_t mean = (int64_t)n_pairs / n_tiles;
    if (B == 8 && few) DCUDA((launch_density<8, 8, 4>(n_tiles, params, v0, begin, end, g, theta, max_spread, out_density, s)));
    else if (B == 8 && mean < 32) DCUDA((launch_density<8, 2, 1>(n_tiles, params, v0, begin, end, g, theta, max_spread, out_density, s)));
    else if (B == 8 && mean < 256) DCUDA((launch_density<8, 4, 1>(n_tiles, params, v0, begin, end, g, theta, max_spread, out_density, s)));
    else if (B == 8) DCUDA((launch_density<8, 8, 1>(n_tiles, params, v0, begin, end, g, theta, max_spread, out_density, s)));
    else if (few) DCUDA((launch_density<4, 4, 4>(n_tiles, params, v0, begin, end, g, theta, max_spread, out_density, s)));
    else DCUDA((launch_density<4, 1, 1>(n_tiles, params, v0, begin, end, g, theta, max_spread, out_density, s)));
    ++launches;
    DCUDA(cudaGetLastError());
    if (timing) DCUDA(cudaEventRecord(S.ev[2], s));
  } else {
    DCUDA(cudaMemsetAsync(out_density, 0, (size_t)n_vox * sizeof(float), s));
  }
  if (out_occ || out_surf) {
    const dim3 og((unsigned)((grid->dims[0] + 31) / 32),
                  (unsigned)std::min((grid->dims[1] + kOccRows - 1) / kOccRows, 65535),
                  (unsigned)std::min(grid->dims[2], 65535));
    k_occ_surf<<<og, dim3(32, kOccRows), 0, s>>>(out_density, g, theta, out_occ, out_surf);
    ++launches;
    DCUDA(cudaGetLastError());
  }
  if (stats) {
    stats->n_pairs = (int64_t)n_pairs;
    stats->n_tiles = n_tiles;
    stats->n_voxels = n_vox;
    stats->ms_total = stats->ms_density = 0.f;
    stats->n_launches = launches;
  }
  if (timing) {
    DCUDA(cudaEventRecord(S.ev[3], s));
    DCUDA(cudaEventSynchronize(S.ev[3]));
    DCUDA(cudaEventElapsedTime(&stats->ms_total, S.ev[0], S.ev[3]));
    if (n_pairs > 0) DCUDA(cudaEventElapsedTime(&stats->ms_density, S.ev[1], S.ev[2]));
  }
  return FGL_OK;
}
