// Optional sensor effects on cast returns: seeded return dropout and range
// noise, applied in place after a cast.
//
// The paper's return is the nearest hit only (Sec. IV-C, eq. t_j*) and it
// leaves richer sensor physics to future work; this pass is an extension on
// top of eq. t_j*, reproducible bit for bit in its random decisions:
//   - random words: Philox-4x32-10 (Salmon et al., SC 2011) with key
//     (seed low, seed high) and counter (ray j, env_offset + e, step, 0);
//   - dropout: a hit is dropped -- reported as the miss (max_range, -1) --
//     when (x0 >> 8) 2^-24 < drop_prob (both exact in float32);
//   - noise: a kept hit at range t becomes t + (sigma0 + sigma1 t) n,
//     n = sqrt(-2 ln u1) cos(2 pi u2) (Box-Muller), u1 = ((x1 >> 8) + 1) 2^-24,
//     u2 = (x2 >> 8) 2^-24, clamped to [0, max_range]; float32 arithmetic.
// Misses are left as they are.
#include <cuda_runtime.h>

#include <cmath>
#include <string>

#include "fgl.h"
#include "nvtx_range.h"

namespace fgl {
void record_error(int status, const char* msg);  // api.cu
}

namespace {

// The ten round keys, the key schedule of (seed low, seed high): made once on
// the host, they reach the rounds as constants.
struct RoundKeys {
  uint32_t k0[10], k1[10];
};

__device__ __forceinline__ void philox4x32_10(uint32_t& c0, uint32_t& c1, uint32_t& c2, uint32_t& c3,
                                              const RoundKeys& k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint64_t p0 = (uint64_t)0xD2511F53u * c0, p1 = (uint64_t)0xCD9E8D57u * c2;
    const uint32_t lo0 = (uint32_t)p0, hi0 = (uint32_t)(p0 >> 32), lo1 = (uint32_t)p1, hi1 = (uint32_t)(p1 >> 32);
    const uint32_t n0 = hi1 ^ c1 ^ k.k0[r], n2 = hi0 ^ c3 ^ k.k1[r];
    c0 = n0;
    c1 = lo1;
    c2 = n2;
    c3 = lo0;
  }
}

// One return: true when it changed its range; *drop when it became a miss.
struct Effects {
  RoundKeys key;
  uint32_t step;
  int32_t env_offset;
  float drop_prob, sigma0, sigma1, max_range;
};

__device__ __forceinline__ bool apply(const Effects& fx, uint32_t ray, uint32_t env, float& t, int32_t& tri) {
  if (tri < 0) return false;
  uint32_t x0 = ray, x1 = env, x2 = fx.step, x3 = 0u;
  philox4x32_10(x0, x1, x2, x3, fx.key);
  const float inv24 = 5.9604644775390625e-8f;  // 2^-24
  if ((float)(x0 >> 8) * inv24 < fx.drop_prob) {
    t = fx.max_range;
    tri = -1;
    return true;
  }
  if (fx.sigma0 == 0.f && fx.sigma1 == 0.f) return false;
  const float u1 = (float)((x1 >> 8) + 1u) * inv24, u2 = (float)(x2 >> 8) * inv24;
  const float nrm = sqrtf(-2.f * logf(u1)) * cospif(2.f * u2);
  t = fminf(fmaxf(t + (fx.sigma0 + fx.sigma1 * t) * nrm, 0.f), fx.max_range);
  return true;
}

constexpr int kFxThreads = 256, kFxItems = 4, kFxBlock = kFxThreads * kFxItems;

// A block takes kFxBlock consecutive returns.  One thread finds the block's
// first (environment, ray) with the 64-bit division; from there a return's
// environment is a 32-bit division of its offset.  VEC: four consecutive
// returns a thread in 16-byte accesses (both arrays 16-byte aligned).
template <bool VEC>
__global__ void __launch_bounds__(kFxThreads) k_effects(float* __restrict__ range, int32_t* __restrict__ tri,
                                                        int64_t n, uint32_t n_rays, const Effects fx) {
  __shared__ uint32_t s_env, s_ray;
  const int64_t base = (int64_t)blockIdx.x * kFxBlock;
  if (threadIdx.x == 0) {
    const int64_t e = base / n_rays;
    s_env = (uint32_t)fx.env_offset + (uint32_t)e;
    s_ray = (uint32_t)(base - e * n_rays);
  }
  __syncthreads();
  const uint32_t env0 = s_env, ray0 = s_ray;  // ray0 + kFxBlock < 2^32
  const uint32_t left = n - base < kFxBlock ? (uint32_t)(n - base) : (uint32_t)kFxBlock;
  uint32_t ray, env;  // of the return at hand
  auto at = [&](uint32_t off) {
    const uint32_t r = ray0 + off, de = r / n_rays;
    ray = r - de * n_rays;
    env = env0 + de;
  };
  auto next = [&](float& t, int32_t& id) {
    const bool changed = apply(fx, ray, env, t, id);
    if (++ray == n_rays) {
      ray = 0;
      ++env;
    }
    return changed;
  };
  if (VEC) {
    const uint32_t off = threadIdx.x * kFxItems;
    if (off + kFxItems <= left) {
      float4 t = *reinterpret_cast<const float4*>(range + base + off);
      int4 id = *reinterpret_cast<const int4*>(tri + base + off);
      const int4 id0 = id;
      at(off);
      const bool c0 = next(t.x, id.x), c1 = next(t.y, id.y), c2 = next(t.z, id.z), c3 = next(t.w, id.w);
      if (c0 | c1 | c2 | c3) *reinterpret_cast<float4*>(range + base + off) = t;
      if ((id.x ^ id0.x) | (id.y ^ id0.y) | (id.z ^ id0.z) | (id.w ^ id0.w))
        *reinterpret_cast<int4*>(tri + base + off) = id;
      return;
    }
    for (uint32_t o = off; o < left; ++o) {  // the last, partial four
      float t = range[base + o];
      int32_t id = tri[base + o];
      const int32_t id0 = id;
      at(o);
      if (next(t, id)) range[base + o] = t;
      if (id != id0) tri[base + o] = id;
    }
  } else {
#pragma unroll
    for (int k = 0; k < kFxItems; ++k) {
      const uint32_t o = threadIdx.x + k * kFxThreads;
      if (o >= left) break;
      float t = range[base + o];
      int32_t id = tri[base + o];
      const int32_t id0 = id;
      at(o);
      if (next(t, id)) range[base + o] = t;
      if (id != id0) tri[base + o] = id;
    }
  }
}

fgl_status err(int status, const char* msg) {
  fgl::record_error(status, msg);
  return (fgl_status)status;
}

}  // namespace

extern "C" fgl_status fgl_apply_sensor_effects(const fgl_sensor_effects* fx, float* range, int32_t* tri,
                                               int32_t n_env, int32_t n_rays, fgl_stream stream) {
  fgl::NvtxRange nvtx("fgl_apply_sensor_effects");
  if (!fx) return err(FGL_ERR_INVALID, "null effects");
  if (n_env < 0 || n_rays < 1) return err(FGL_ERR_INVALID, "n_env must be >= 0 and n_rays >= 1");
  if ((int64_t)fx->env_offset + n_env > ((int64_t)1 << 32))
    return err(FGL_ERR_INVALID, "env_offset + n_env must fit in 32 bits");
  if (fx->env_offset < 0) return err(FGL_ERR_INVALID, "env_offset must be >= 0");
  if (!(fx->drop_prob >= 0.f && fx->drop_prob <= 1.f))
    return err(FGL_ERR_INVALID, "drop_prob must be in [0, 1]");
  if (!(fx->noise_sigma0 >= 0.f && fx->noise_sigma1 >= 0.f) || !std::isfinite(fx->noise_sigma0) ||
      !std::isfinite(fx->noise_sigma1))
    return err(FGL_ERR_INVALID, "noise sigmas must be finite and >= 0");
  if (!(std::isfinite(fx->max_range) && fx->max_range > 0.f))
    return err(FGL_ERR_INVALID, "max_range must be finite and > 0");
  const int64_t n = (int64_t)n_env * n_rays;
  if (n == 0) return FGL_OK;
  if (!range || !tri) return err(FGL_ERR_INVALID, "null range or tri");
  const int64_t blocks = (n + kFxBlock - 1) / kFxBlock;
  if (blocks > 0x7FFFFFFF) return err(FGL_ERR_INVALID, "too many returns (more than 2^41)");
  Effects p{{}, fx->step, fx->env_offset, fx->drop_prob, fx->noise_sigma0, fx->noise_sigma1, fx->max_range};
  for (uint32_t r = 0; r < 10; ++r) {
    p.key.k0[r] = (uint32_t)fx->seed + r * 0x9E3779B9u;
    p.key.k1[r] = (uint32_t)(fx->seed >> 32) + r * 0xBB67AE85u;
  }
  const bool vec = (((uintptr_t)range | (uintptr_t)tri) & 15u) == 0;
  if (vec) k_effects<true><<<(unsigned)blocks, kFxThreads, 0, (cudaStream_t)stream>>>(range, tri, n, (uint32_t)n_rays, p);
  else k_effects<false><<<(unsigned)blocks, kFxThreads, 0, (cudaStream_t)stream>>>(range, tri, n, (uint32_t)n_rays, p);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return err(FGL_ERR_CUDA, cudaGetErrorString(e));
  return FGL_OK;
}
