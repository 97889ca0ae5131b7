// Device-wide exclusive scans and a stable LSD radix sort of (key, value)
// pairs, shared by the Gaussian-to-occupancy pipeline (pairs sorted by tile)
// and the GPU triangle LBVH builder (triangles sorted by Morton code).
#include <cuda_runtime.h>

#include <algorithm>

#include "sort.h"

namespace fgl {
namespace {

// ---------------------------------------------------------------------------
// exclusive scan (in place), 2048 items per block, recursive over block sums
// ---------------------------------------------------------------------------
template <class T>
__global__ void k_scan_blocks(T* __restrict__ x, int64_t n, T* __restrict__ sums) {
  __shared__ T warp_tot[32];
  const int64_t base = (int64_t)blockIdx.x * 2048;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int64_t i0 = base + 2 * t;
  T a = i0 < n ? x[i0] : T(0);
  T b = i0 + 1 < n ? x[i0 + 1] : T(0);
  T v = a + b;  // inclusive warp scan of pair sums
  T incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    T w = warp_tot[lane];
    T wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      T u = __shfl_up_sync(0xFFFFFFFFu, wi, o);
      if (lane >= o) wi += u;
    }
    warp_tot[lane] = wi - w;  // exclusive warp offsets
    if (lane == 31 && sums) sums[blockIdx.x] = wi;
  }
  __syncthreads();
  const T excl = warp_tot[wid] + incl - v;
  if (i0 < n) x[i0] = excl;
  if (i0 + 1 < n) x[i0 + 1] = excl + a;
}

template <class T>
__global__ void k_scan_add(T* __restrict__ x, int64_t n, const T* __restrict__ sums) {
  const int64_t i = (int64_t)blockIdx.x * 2048 + threadIdx.x;
  const T add = sums[blockIdx.x];
  if (i < n) x[i] += add;
  if (i + 1024 < n) x[i + 1024] += add;
}

// ---------------------------------------------------------------------------
// radix sort pass: digit counts of every block's slice, their exclusive
// prefixes within each digit, then a stable scatter
// ---------------------------------------------------------------------------

// Digit counts of a slice of THREADS * ROUNDS keys: hist[digit][block].
template <int THREADS, int ROUNDS>
__global__ void __launch_bounds__(THREADS) k_radix_hist(const uint32_t* __restrict__ keys, int64_t n, int shift,
                                                        uint32_t* __restrict__ hist, int nblocks) {
  __shared__ uint32_t h[256];
  if (threadIdx.x < 256) h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * (THREADS * ROUNDS);
  uint32_t d[ROUNDS];  // every key loaded before the first count: one memory latency
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const int64_t i = base + r * THREADS + threadIdx.x;
    d[r] = i < n ? (keys[i] >> shift) & 255u : 256u;
  }
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r)
    if (d[r] < 256u) atomicAdd(&h[d[r]], 1u);
  __syncthreads();
  if (threadIdx.x < 256) hist[(int64_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// Block d turns digit d's counts into exclusive prefixes in place and writes
// their sum (the digits' own prefixes are taken by the scatter).
__global__ void __launch_bounds__(256) k_radix_rows(uint32_t* __restrict__ hist, int nblocks,
                                                    uint32_t* __restrict__ totals) {
  __shared__ uint32_t warp_tot[8];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  uint32_t* row = hist + (int64_t)blockIdx.x * nblocks;
  uint32_t carry = 0;
  for (int b0 = 0; b0 < nblocks; b0 += 256) {
    const uint32_t v = b0 + t < nblocks ? row[b0 + t] : 0u;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += u;
    }
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    uint32_t before = carry, all = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (k < w) before += warp_tot[k];
      all += warp_tot[k];
    }
    if (b0 + t < nblocks) row[b0 + t] = before + incl - v;
    carry += all;
    __syncthreads();
  }
  if (t == 0) totals[blockIdx.x] = carry;
}

// Stable scatter.  Each warp owns a contiguous run of ROUNDS * 32 items, so
// index order is (warp, round, lane).  An item's rank among its warp's items
// of the same digit is the warp's running count of the digit plus the lower
// lanes of the round that hold it; the lanes of a digit are collected in a
// shared-memory word by atomic OR.  A block barrier turns the counts into block-local offsets
// (digit-major, then warp); the items are placed in shared memory sorted by
// digit, and the write-out copies the block's digit runs to their global
// offsets, consecutive threads writing consecutive addresses.  Keys and values
// are read once, all of a thread's loads in flight together.
template <int THREADS, int ROUNDS>
struct ScatterSmem {
  static constexpr int NW = THREADS / 32, ITEMS = THREADS * ROUNDS;
  uint32_t wcount[NW][256];  // digit counts, then the warps' local offsets
  uint32_t gofs[256];        // a digit's global start in this block less its local start
  uint32_t wsum[2][8];
  uint32_t k[ITEMS], v[ITEMS];
};

template <int THREADS, int ROUNDS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) k_radix_scatter(const uint32_t* __restrict__ kin,
                                                           const uint32_t* __restrict__ vin, int64_t n, int shift,
                                                           const uint32_t* __restrict__ rows,
                                                           const uint32_t* __restrict__ totals, int nblocks,
                                                           uint32_t* __restrict__ kout, uint32_t* __restrict__ vout) {
  using Sm = ScatterSmem<THREADS, ROUNDS>;
  extern __shared__ __align__(16) unsigned char scatter_smem[];
  Sm& sm = *reinterpret_cast<Sm*>(scatter_smem);
  const unsigned FULL = 0xFFFFFFFFu;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int64_t block0 = (int64_t)blockIdx.x * Sm::ITEMS;
  const int64_t base = block0 + (int64_t)w * (32 * ROUNDS) + lane;
  uint32_t key[ROUNDS];
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) key[r] = base + r * 32 < n ? kin[base + r * 32] : 0u;
  uint32_t* held = sm.k + 256 * w;  // by digit, the round's lanes that hold it (the items are placed later)
  for (int d = lane; d < 256; d += 32) sm.wcount[w][d] = held[d] = 0;
  __syncwarp();
  const unsigned lt = (1u << lane) - 1u;
  uint16_t rank[ROUNDS];
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const bool in = base + r * 32 < n;
    const uint32_t d = (key[r] >> shift) & 255u;
    if (in) atomicOr(&held[d], 1u << lane);
    __syncwarp();
    const unsigned peers = held[d];
    const uint32_t below = __popc(peers & lt), c = sm.wcount[w][d];
    rank[r] = (uint16_t)(c + below);
    __syncwarp();
    if (in && below == 0) {
      held[d] = 0;
      sm.wcount[w][d] = c + __popc(peers);
    }
    __syncwarp();
  }
  uint32_t val[ROUNDS];  // on their way while the offsets are made
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) val[r] = base + r * 32 < n ? vin[base + r * 32] : 0u;
  __syncthreads();
  {
    // thread t < 256 is digit t: its count in the block and its total, their
    // exclusive prefixes over the digits, and the warps' offsets
    uint32_t tot = 0, incl = 0, gtot = 0, gincl = 0;
    if (t < 256) {
#pragma unroll
      for (int k = 0; k < Sm::NW; ++k) tot += sm.wcount[k][t];
      gtot = totals[t];
      incl = tot;
      gincl = gtot;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(FULL, incl, o), g = __shfl_up_sync(FULL, gincl, o);
        if (lane >= o) {
          incl += u;
          gincl += g;
        }
      }
      if (lane == 31) {
        sm.wsum[0][w] = incl;
        sm.wsum[1][w] = gincl;
      }
    }
    __syncthreads();
    if (t < 256) {
      uint32_t run = incl - tot, gstart = gincl - gtot;
      for (int k = 0; k < w; ++k) {
        run += sm.wsum[0][k];
        gstart += sm.wsum[1][k];
      }
      sm.gofs[t] = gstart + rows[(int64_t)t * nblocks + blockIdx.x] - run;
#pragma unroll
      for (int k = 0; k < Sm::NW; ++k) {
        const uint32_t c = sm.wcount[k][t];
        sm.wcount[k][t] = run;
        run += c;
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    if (base + r * 32 < n) {
      const uint32_t pos = sm.wcount[w][(key[r] >> shift) & 255u] + rank[r];
      sm.k[pos] = key[r];
      sm.v[pos] = val[r];
    }
  }
  __syncthreads();
  const int cnt = n - block0 < (int64_t)Sm::ITEMS ? (int)(n - block0) : Sm::ITEMS;
#pragma unroll 4
  for (int i = t; i < cnt; i += THREADS) {
    const uint32_t k = sm.k[i];
    const uint32_t pos = sm.gofs[(k >> shift) & 255u] + (uint32_t)i;
    kout[pos] = k;
    vout[pos] = sm.v[i];
  }
}

// Slices: a longer one leaves longer digit runs to write (16 items on average
// at 4096), a shorter one more blocks at once.  The two passes over 19 M pairs made
// an occupancy call 1.5% shorter at 4096 items than at 8192 (which spills
// registers); arrays whose 4096-item slices would not fill the chip
// twice take 2048.
constexpr int kBigThreads = 512, kBigRounds = 8, kSmallThreads = 256, kSmallRounds = 8;
constexpr int64_t kBigFrom = (int64_t)152 * 2 * kBigThreads * kBigRounds;

int slice_items(int64_t n) { return n >= kBigFrom ? kBigThreads * kBigRounds : kSmallThreads * kSmallRounds; }

template <int THREADS, int ROUNDS>
cudaError_t radix_pass(const uint32_t* k0, const uint32_t* v0, uint32_t* k1, uint32_t* v1, int64_t n, int shift,
                       uint32_t* hist, cudaStream_t s) {
  const int nblocks = (int)((n + THREADS * ROUNDS - 1) / (THREADS * ROUNDS));
  uint32_t* totals = hist + (int64_t)256 * nblocks;
  k_radix_hist<THREADS, ROUNDS><<<nblocks, THREADS, 0, s>>>(k0, n, shift, hist, nblocks);
  k_radix_rows<<<256, 256, 0, s>>>(hist, nblocks, totals);
  const size_t smem = sizeof(ScatterSmem<THREADS, ROUNDS>);
  auto* fn = k_radix_scatter<THREADS, ROUNDS>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  fn<<<nblocks, THREADS, smem, s>>>(k0, v0, n, shift, hist, totals, nblocks, k1, v1);
  return cudaGetLastError();
}

}  // namespace

// exclusive scan of n values in place; `tmp` holds the per-level block sums
template <class T>
cudaError_t scan_exclusive_t(T* x, int64_t n, T* tmp, size_t tmp_elems, cudaStream_t s,
                           int* launches) {
  if (n <= 0) return cudaSuccess;
  const int64_t nb = (n + 2047) / 2048;
  if (nb == 1) {
    k_scan_blocks<T><<<1, 1024, 0, s>>>(x, n, (T*)nullptr);
    ++*launches;
    return cudaGetLastError();
  }
  if ((size_t)nb > tmp_elems) return cudaErrorInvalidValue;
  k_scan_blocks<T><<<(unsigned)nb, 1024, 0, s>>>(x, n, tmp);
  ++*launches;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = scan_exclusive_t<T>(tmp, nb, tmp + nb, tmp_elems - nb, s, launches);
  if (e != cudaSuccess) return e;
  k_scan_add<T><<<(unsigned)nb, 1024, 0, s>>>(x, n, tmp);
  ++*launches;
  return cudaGetLastError();
}

// block sums needed by scan_exclusive over n values, all levels
size_t scan_tmp_elems(int64_t n) {
  size_t t = 0;
  while (n > 2048) {
    n = (n + 2047) / 2048;
    t += (size_t)n;
  }
  return t + 1;
}


cudaError_t scan_exclusive_u64(unsigned long long* x, int64_t n, unsigned long long* tmp,
                               size_t tmp_elems, cudaStream_t s, int* launches) {
  return scan_exclusive_t<unsigned long long>(x, n, tmp, tmp_elems, s, launches);
}

size_t radix_sort_tmp_elems(int64_t n) {
  const int items = slice_items(n);
  return (size_t)(256 * ((n + items - 1) / items) + 256);
}

cudaError_t radix_sort_pairs(uint32_t* k0, uint32_t* v0, uint32_t* k1, uint32_t* v1, int64_t n,
                             int bits, uint32_t* tmp, cudaStream_t s, int* launches,
                             bool* in_second) {
  *in_second = false;
  if (n <= 0) return cudaSuccess;
  for (int shift = 0; shift < bits; shift += 8) {
    const cudaError_t e = n >= kBigFrom
                              ? radix_pass<kBigThreads, kBigRounds>(k0, v0, k1, v1, n, shift, tmp, s)
                              : radix_pass<kSmallThreads, kSmallRounds>(k0, v0, k1, v1, n, shift, tmp, s);
    if (e != cudaSuccess) return e;
    *launches += 3;
    std::swap(k0, k1);
    std::swap(v0, v1);
    *in_second = !*in_second;
  }
  return cudaSuccess;
}

}  // namespace fgl
