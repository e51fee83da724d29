// returns.cu — REINFORCE returns and GAE advantages over the [T][E] rollout
// buffer (Sec. 4.3; GAE after Schulman et al. 2016), and the mean-return baseline.
//
// Both recurrences are first-order affine maps run backwards in time,
//   x_t = delta_t + c_t x_{t+1},
// REINFORCE: x = G, delta_t = r_t, c_t = gamma (1 - d_t), x_T = last_value;
// GAE:       x = A, delta_t = r_t + gamma (1 - d_t) V_{t+1} - V_t,
//            c_t = gamma lambda (1 - d_t), x_T = 0.
// Env counts from 65,536 with 16-byte aligned rows take k_returns_wide: one thread owns four
// adjacent envs for the whole horizon (one pass: every input read once, every output
// written once, 17 bytes per sample for GAE), loading 8 time steps ahead with 16-byte
// loads, so a block reads 1 KB of each row per step.
// Otherwise a block owns 32 envs (threadIdx.x) and S chunks of the horizon (threadIdx.y).  Each
// thread composes its chunk's map x_{t0} = a x_{t1} + b, one thread per env chains the S maps in
// shared memory, then every thread replays its chunk from the right carry.  Loads are coalesced
// across envs; no global scratch is needed.
//   k_returns_long: chunks of ceil(T / S) steps, read twice, no barrier between a chunk's steps.
//   k_returns_gae (many envs, see kOnceMinEnvs): windows of S chunks of 8 steps held in registers,
//   every input read once; each window is a round trip to memory and three barriers.  Past L2
//   HBM bounds it (60,000 envs x 1024 238 us, 4.4 TB/s, k_returns_long 299); below, the latency of
//   that round trip (16,384 envs x 256: 18.4 us, 3.9 TB/s, with the buffers not in L2, against 20.4).
#include <cstdint>

#include "kernels.h"

namespace simx {

constexpr int kRetMaxChunks = 32;
constexpr int kRetL = 8;   // steps per chunk, held in registers

// One thread's chunk of one window: kRetL steps of one env from step t0 on.  Steps past the
// horizon stand for the state after it: value `last`, no reward.
template <bool GAE>
struct RetChunk {
  float r[kRetL], v[GAE ? kRetL : 1];
  uint32_t d;   // bit i: step i ends its segment
  __device__ __forceinline__ void load(const float* __restrict__ rew, const float* __restrict__ val,
                                       const uint8_t* __restrict__ done, int64_t t0, int64_t T, int64_t ld,
                                       int64_t e, bool live, float last) {
    uint8_t dd[kRetL];
#pragma unroll
    for (int i = 0; i < kRetL; ++i) {
      const bool in = live && t0 + i < T;
      const int64_t o = (t0 + i) * ld + e;
      r[i] = in ? rew[o] : 0.0f;
      dd[i] = in ? done[o] : (uint8_t)0;
      if (GAE) v[i] = in ? val[o] : last;
    }
    d = 0u;
#pragma unroll
    for (int i = 0; i < kRetL; ++i) d |= dd[i] ? 1u << i : 0u;
  }
};

// A block owns 32 envs and walks the horizon backwards in windows of S chunks of kRetL steps,
// the next window's loads in flight while this one is chained.  Every input is read once.
template <bool GAE>
__global__ void __launch_bounds__(1024)
k_returns_gae(const float* __restrict__ rew, const float* __restrict__ val,
              const uint8_t* __restrict__ done, const float* __restrict__ last_val, int64_t T,
              int64_t E, int64_t ld, float gamma, float lam, float* __restrict__ ret,
              float* __restrict__ adv) {
  __shared__ float sa[kRetMaxChunks][32], sb[kRetMaxChunks][32], scarry[kRetMaxChunks][32];
  __shared__ float sv[kRetMaxChunks + 1][32];   // row j: chunk j's first value; row S: the window after
  const int x = threadIdx.x, j = threadIdx.y, S = blockDim.y;
  const int64_t e = (int64_t)blockIdx.x * 32 + x;
  const bool live = e < E;
  const float cmul = GAE ? gamma * lam : gamma;
  const float last = live && last_val ? last_val[e] : 0.0f;
  const int64_t W = (int64_t)S * kRetL;
  int64_t t0 = (T + W - 1) / W * W - W + (int64_t)j * kRetL;
  float carry = GAE ? 0.0f : last;   // (threads of chunk 0) the recurrence entering from the right
  if (GAE && j == 0) sv[S][x] = last;
  RetChunk<GAE> c;
  c.load(rew, val, done, t0, T, ld, e, live, last);
  for (;;) {
    RetChunk<GAE> nx;
    if (t0 >= W) nx.load(rew, val, done, t0 - W, T, ld, e, live, last);
    if (GAE) {
      sv[j][x] = c.v[0];
      __syncthreads();
    }
    // this chunk's map x_{t0} = a x_{t1} + b; r becomes delta
    float vnext = GAE ? sv[j + 1][x] : 0.0f;
    float a = 1.0f, b = 0.0f;
#pragma unroll
    for (int i = kRetL - 1; i >= 0; --i) {
      const float mask = (c.d >> i) & 1u ? 0.0f : 1.0f;
      if (GAE) {
        c.r[i] = c.r[i] + gamma * mask * vnext - c.v[i];
        vnext = c.v[i];
      }
      if (t0 + i < T) {
        const float cc = cmul * mask;
        b = c.r[i] + cc * b;
        a = cc * a;
      }
    }
    sa[j][x] = a;
    sb[j][x] = b;
    __syncthreads();
    if (j == 0) {
      if (GAE) sv[S][x] = c.v[0];
#pragma unroll 4
      for (int q = S - 1; q >= 0; --q) {
        scarry[q][x] = carry;
        carry = sb[q][x] + sa[q][x] * carry;
      }
    }
    __syncthreads();
    // replay with the carry that enters the chunk from the right
    float y = scarry[j][x];
#pragma unroll
    for (int i = kRetL - 1; i >= 0; --i) {
      if (live && t0 + i < T) {
        const float mask = (c.d >> i) & 1u ? 0.0f : 1.0f;
        const int64_t o = (t0 + i) * ld + e;
        y = c.r[i] + cmul * mask * y;
        if (GAE) {
          adv[o] = y;
          ret[o] = y + c.v[i];
        } else {
          ret[o] = y;
          if (adv) adv[o] = y;
        }
      }
    }
    if (t0 < W) break;   // the same for every thread of the block: W divides each window's start
    t0 -= W;
    c = nx;
  }
}

// A block owns 32 envs and up to 32 chunks of ceil(T / S) steps, each read twice.  Everything below
// kOnceMinEnvs keeps this composition: training runs carry a last bit of it on.
__global__ void __launch_bounds__(1024)
k_returns_long(const float* __restrict__ rew, const float* __restrict__ val,
              const uint8_t* __restrict__ done, const float* __restrict__ last_val, int64_t T,
              int64_t E, int64_t ld, float gamma, float lam, float* __restrict__ ret,
              float* __restrict__ adv) {
  __shared__ float sa[kRetMaxChunks][32], sb[kRetMaxChunks][32], scarry[kRetMaxChunks][32];
  const int64_t e = (int64_t)blockIdx.x * 32 + threadIdx.x;
  const int S = blockDim.y, j = threadIdx.y;
  const bool gae_mode = lam >= 0.0f;
  const float cmul = gae_mode ? gamma * lam : gamma;
  const int64_t L = (T + S - 1) / S;
  const int64_t t0 = (int64_t)j * L;
  const int64_t t1 = t0 + L < T ? t0 + L : T;
  const bool live = e < E;
  float last = 0.0f;
  if (live && last_val) last = last_val[e];
  // pass 1: this chunk's map with a zero carry
  float a = 1.0f, b = 0.0f;
  if (live) {
    float vnext = 0.0f;
    if (gae_mode) vnext = (t1 < T) ? val[t1 * ld + e] : last;
    for (int64_t t = t1 - 1; t >= t0; --t) {
      const int64_t o = t * ld + e;
      const float mask = done[o] ? 0.0f : 1.0f;
      float delta = rew[o];
      if (gae_mode) {
        const float v = val[o];
        delta = delta + gamma * mask * vnext - v;
        vnext = v;
      }
      const float c = cmul * mask;
      b = delta + c * b;
      a = c * a;
    }
  }
  sa[j][threadIdx.x] = a;
  sb[j][threadIdx.x] = b;
  __syncthreads();
  if (j == 0) {
    float carry = gae_mode ? 0.0f : last;
    for (int q = S - 1; q >= 0; --q) {
      scarry[q][threadIdx.x] = carry;
      carry = sb[q][threadIdx.x] + sa[q][threadIdx.x] * carry;
    }
  }
  __syncthreads();
  if (!live) return;
  // pass 2: replay with the carry that enters the chunk from the right
  float x = scarry[j][threadIdx.x];
  float vnext = 0.0f;
  if (gae_mode) vnext = (t1 < T) ? val[t1 * ld + e] : last;
  for (int64_t t = t1 - 1; t >= t0; --t) {
    const int64_t o = t * ld + e;
    const float mask = done[o] ? 0.0f : 1.0f;
    float delta = rew[o];
    float v = 0.0f;
    if (gae_mode) {
      v = val[o];
      delta = delta + gamma * mask * vnext - v;
      vnext = v;
    }
    x = delta + cmul * mask * x;
    if (gae_mode) {
      adv[o] = x;
      ret[o] = x + v;
    } else {
      ret[o] = x;
      if (adv) adv[o] = x;
    }
  }
}

constexpr int kWideU = 8;                 // time steps loaded ahead
constexpr int kWideThreads = 64;          // 256 envs per block: every SM gets blocks from 65,536 envs
constexpr int64_t kWideMinEnvs = 65536;
// The lines of k_returns_gae.  GAE, us with the buffers in L2 and not, k_returns_long against it:
// 10,000 envs x 256 10.9 and 16.7 against 11.3 and 15.9; 16,383 15.1 and 22.4 against 14.5 and 18.8;
// 20,000 17.5 and 26.6 against 19.8 and 25.6; 16,384 x 1024 82 against 63.  REINFORCE, a third
// less to read: 16,384 x 512 16.1 and 23.5 against 23.4 and 26.5, x 1024 44.5 against 50.5; 30,000 x
// 1024 91.3 against 86.3.
constexpr int64_t kOnceMinEnvs = 16384;
constexpr int64_t kOnceMinSamples = 24 << 20;   // REINFORCE

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

template <bool GAE>
__global__ void __launch_bounds__(kWideThreads, 8)
k_returns_wide(const float* __restrict__ rew, const float* __restrict__ val,
               const uint8_t* __restrict__ done, const float* __restrict__ last_val, int64_t T,
               int64_t E, int64_t ld, float gamma, float lam, float* __restrict__ ret,
               float* __restrict__ adv) {
  const int64_t e = ((int64_t)blockIdx.x * kWideThreads + threadIdx.x) * 4;
  if (e >= E) return;
  const float cmul = GAE ? gamma * lam : gamma;
  float4 last = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (last_val) last = ld4(last_val + e);
  float x[4] = {GAE ? 0.0f : last.x, GAE ? 0.0f : last.y, GAE ? 0.0f : last.z, GAE ? 0.0f : last.w};
  float vn[4] = {last.x, last.y, last.z, last.w};
  for (int64_t tb = T; tb > 0; tb -= kWideU) {
    const int n = tb < kWideU ? (int)tb : kWideU;
    float4 r[kWideU], v[kWideU];
    uint32_t d[kWideU];
#pragma unroll
    for (int i = 0; i < kWideU; ++i) {
      if (i < n) {
        const int64_t o = (tb - 1 - i) * ld + e;
        r[i] = ld4(rew + o);
        d[i] = *reinterpret_cast<const uint32_t*>(done + o);
        if (GAE) v[i] = ld4(val + o);
      }
    }
#pragma unroll
    for (int i = 0; i < kWideU; ++i) {
      if (i < n) {
        const int64_t o = (tb - 1 - i) * ld + e;
        const float rv[4] = {r[i].x, r[i].y, r[i].z, r[i].w};
        float vv[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (GAE) {
          vv[0] = v[i].x;
          vv[1] = v[i].y;
          vv[2] = v[i].z;
          vv[3] = v[i].w;
        }
        float o4[4], g4[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float mask = ((d[i] >> (8 * k)) & 0xFFu) ? 0.0f : 1.0f;
          float delta = rv[k];
          if (GAE) {
            delta = delta + gamma * mask * vn[k] - vv[k];
            vn[k] = vv[k];
          }
          x[k] = delta + cmul * mask * x[k];
          o4[k] = x[k];
          g4[k] = x[k] + vv[k];
        }
        if (GAE) {
          st4(adv + o, make_float4(o4[0], o4[1], o4[2], o4[3]));
          st4(ret + o, make_float4(g4[0], g4[1], g4[2], g4[3]));
        } else {
          st4(ret + o, make_float4(o4[0], o4[1], o4[2], o4[3]));
          if (adv) st4(adv + o, make_float4(o4[0], o4[1], o4[2], o4[3]));
        }
      }
    }
  }
}

static bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

cudaError_t launch_returns_gae(const float* rew, const float* val, const uint8_t* done,
                               const float* last_val, int64_t T, int64_t E, int64_t ld,
                               float gamma, float lam, float* ret, float* adv, cudaStream_t s) {
  if (T <= 0 || E <= 0) return cudaSuccess;
  const bool gae = lam >= 0.0f;
  if (E >= kWideMinEnvs && E % 4 == 0 && ld % 4 == 0 && aligned16(rew) && aligned16(ret) &&
      ((uintptr_t)done & 3u) == 0 && (!gae || aligned16(val)) && (!adv || aligned16(adv)) &&
      (!last_val || aligned16(last_val))) {
    const unsigned grid = (unsigned)((E / 4 + kWideThreads - 1) / kWideThreads);
    if (gae)
      k_returns_wide<true><<<grid, kWideThreads, 0, s>>>(rew, val, done, last_val, T, E, ld, gamma, lam, ret, adv);
    else
      k_returns_wide<false><<<grid, kWideThreads, 0, s>>>(rew, val, done, last_val, T, E, ld, gamma, lam, ret, adv);
    count_launches(1);
    return cudaGetLastError();
  }
  const bool once = E >= kOnceMinEnvs && (gae || T * E >= kOnceMinSamples);
  int S = 1;
  if (once) {
    // Chunks per window: about 130k threads, whose loads in flight cover the memory latency, in
    // one wave of blocks; no more chunks than the horizon has.
    while (S < kRetMaxChunks && E * S * 2 <= 160000 && (int64_t)S * kRetL < T) S *= 2;
  } else {
    // Enough (env, chunk) threads to fill the GPU: ~300k threads, chunks of >= 16 steps.
    while (S < kRetMaxChunks && E * S * 2 <= 311296 && T / (S * 2) >= 16) S *= 2;
  }
  const auto kernel = !once ? k_returns_long : gae ? k_returns_gae<true> : k_returns_gae<false>;
  kernel<<<(unsigned)((E + 31) / 32), dim3(32, S), 0, s>>>(rew, val, done, last_val, T, E, ld, gamma,
                                                           lam, ret, adv);
  count_launches(1);
  return cudaGetLastError();
}

// Mean-return baseline: per-block fp64 partial sums, then every block of the second
// kernel reduces the partials in block order (same mean everywhere) and centres.  fp64
// arithmetic per element, at this GPU's rate, is the bound; sums as pairs of fp32, whose low
// words lose bits where the elements cancel, would take about half the time and are not used.
constexpr int kBaseThreads = 256;

int baseline_blocks(int64_t n) {
  int64_t b = (n + kBaseThreads * 8 - 1) / (kBaseThreads * 8);
  if (b > 1024) b = 1024;
  if (b < 1) b = 1;
  return (int)b;
}

__global__ void __launch_bounds__(kBaseThreads)
k_base_partial(const float* __restrict__ x, int64_t n, double* __restrict__ part) {
  __shared__ double sh[kBaseThreads];
  double acc = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * kBaseThreads + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * kBaseThreads)
    acc += (double)x[i];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int d = kBaseThreads / 2; d > 0; d >>= 1) {
    if ((int)threadIdx.x < d) sh[threadIdx.x] += sh[threadIdx.x + d];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

__global__ void __launch_bounds__(kBaseThreads)
k_base_center(const float* __restrict__ x, int64_t n, const double* __restrict__ part, int nparts,
              float* __restrict__ adv, float* __restrict__ mean_out) {
  __shared__ double sh[kBaseThreads];
  double acc = 0.0;
  for (int i = threadIdx.x; i < nparts; i += kBaseThreads) acc += part[i];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int d = kBaseThreads / 2; d > 0; d >>= 1) {
    if ((int)threadIdx.x < d) sh[threadIdx.x] += sh[threadIdx.x + d];
    __syncthreads();
  }
  const double mean = sh[0] / (double)n;
  if (blockIdx.x == 0 && threadIdx.x == 0 && mean_out) mean_out[0] = (float)mean;
  if (!adv) return;
  for (int64_t i = (int64_t)blockIdx.x * kBaseThreads + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * kBaseThreads)
    adv[i] = (float)((double)x[i] - mean);
}

cudaError_t launch_baseline(const float* x, int64_t n, float* adv, float* mean_out, double* ws,
                            int nblocks, cudaStream_t s) {
  k_base_partial<<<nblocks, kBaseThreads, 0, s>>>(x, n, ws);
  k_base_center<<<nblocks, kBaseThreads, 0, s>>>(x, n, ws, nblocks, adv, mean_out);
  count_launches(2);
  return cudaGetLastError();
}

}  // namespace simx
