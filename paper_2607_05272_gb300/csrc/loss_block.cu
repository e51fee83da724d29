// loss_block.cu — REINFORCE / PPO loss gradient (Sec. 4.3) in FP32, for tanh / identity policies
// whose weights, in both orders, fit one SM's shared memory beside a tile of rows, over minibatches
// that one tile per SM covers.
//
// A block of 512 threads takes one tile of R minibatch rows with every weight matrix resident
// (bulk copies that land during the gather).  Gather, forward (activations stay in shared memory,
// feature-major), loss head, then per layer dW, db and dZ of the layer below, written in place
// over its activations.  R is the smallest multiple of 8 that gives every SM at most one tile.
//   forward, dZ: 4 x 8 (rows x outputs) register tiles, paired fmas on adjacent outputs, the
//                k-ordered fma chains of the rollout's forward;
//   dW:          4 x 8 (outputs x inputs) tiles over the tile's rows, paired fmas on adjacent
//                rows: every operand pair comes out of a 16-byte load as it is.
// The block partials are summed in block order.
//
// What bounds it: latency between barriers (16 warps per SM issue in 36 % of the cycles; the top
// stalls are the barriers, 3.0 cycles an instruction, and shared-memory loads, 2.5).  The fused kernel
// (loss_fused.cu) stages one layer's weights at a time and holds dZ apart, which leaves 8 warps per
// SM on 32-row tiles: above 32 rows per SM they are two rounds of its blocks, against one round here
// (13-128-128-17 on 152 SMs: 4865 rows 73 us against 60, 8192 75 against 66).  A second tile per
// block would add to a partial in L2 and measured slower than the fused kernel (65,536 rows: 645 us
// against 420), as did equal rows per block (4096 rows: 49 against 43), so those stay there.  The
// price of the range is that it is narrow: three layers of 98 to 128 at 33 to 56 rows per SM (see
// loss_block_taken in loss.cu).
#include <cstdint>

#include "fwd_block.cuh"
#include "kernels.h"

namespace simx {

namespace {

constexpr int NT = 512;          // threads
constexpr int kMaxRows = 64;     // rows per tile at most
constexpr int kLanes = NT / kMaxRows;   // lanes per row in the gather and the loss head
constexpr int kMostSmem = kMaxSmem - 2048;   // the static statistics and a margin

struct BlockLoss {
  LossArgs a;
  const float* Wt[SIMX_MAX_LAYERS];  // [K][npad] transposed, in the workspace
  const float* Wn[SIMX_MAX_LAYERS];  // [N][kpad] (layers >= 1)
  int npad[SIMX_MAX_LAYERS], kpad[SIMX_MAX_LAYERS];
  int act_off[SIMX_MAX_LAYERS + 1];  // first row of each layer's input (and the logits)
  int wt_off[SIMX_MAX_LAYERS], wn_off[SIMX_MAX_LAYERS];  // floats, in shared memory
  int b_off[SIMX_MAX_LAYERS];        // biases, floats
  int poff[SIMX_MAX_LAYERS];
  int n_params, R, ld;
  int bar_off;                       // bytes
  int withheld;                      // the last copy is never issued (tests)
  float* part;
  double* spart;
};

// Y[j][r] = epi(j, rows, sum_k W[k][j] X[k][r]): tiles of TE rows x TO outputs.
template <int TE, int TO, class Epi>
__device__ __forceinline__ void product(const float* W, int ldw, int K, int N, const float* X, int ld, int R,
                                        Epi epi) {
  const int neb = R / TE, nt = neb * ((N + TO - 1) / TO);
  const uint32_t wb = tcx::su32(W), xb = tcx::su32(X);
  for (int tile = (int)threadIdx.x; tile < nt; tile += NT) {
    const int eb = tile % neb, ob = tile / neb;
    uint64_t acc[TE][TO / 2];
#pragma unroll
    for (int e = 0; e < TE; ++e)
#pragma unroll
      for (int o = 0; o < TO / 2; ++o) acc[e][o] = 0ull;
    uint32_t w = wb + 4u * (uint32_t)(TO * ob), x = xb + 4u * (uint32_t)(TE * eb);
#pragma unroll 8
    for (int k = 0; k < K; ++k) {
      fwd::Frag<TE, TO> f;
      f.load(w, x, x);
      w += 4u * (uint32_t)ldw;
      x += 4u * (uint32_t)ld;
      f.mul(acc);
    }
#pragma unroll
    for (int o = 0; o < TO; ++o) {
      const int j = TO * ob + o;
      if (j >= N) continue;
      float v[TE];
#pragma unroll
      for (int e = 0; e < TE; ++e) {
        float lo, hi;
        f2_unpack(acc[e][o / 2], lo, hi);
        v[e] = (o & 1) ? hi : lo;
      }
      epi(j, TE * eb, v);
    }
  }
}

// The tiles of a product: 4 x 8 where they give three eighths of the threads one (their copies of
// each activation into pairs weigh least), 4 x 4 likewise, else 1 x 4.
template <class Epi>
__device__ __forceinline__ void product_of(const float* W, int ldw, int K, int N, const float* X, int ld, int R,
                                           Epi epi) {
  if (ldw % 8 == 0 && (R / 4) * (ldw / 8) * 8 >= 3 * NT) product<4, 8>(W, ldw, K, N, X, ld, R, epi);
  else if ((R / 4) * (ldw / 4) * 8 >= 3 * NT) product<4, 4>(W, ldw, K, N, X, ld, R, epi);
  else product<1, 4>(W, ldw, K, N, X, ld, R, epi);
}

// Lane mask of the S adjacent lanes that share an output.
__device__ __forceinline__ unsigned lane_group(int S) {
  const unsigned lane = threadIdx.x & 31u;
  return S == 32 ? 0xFFFFFFFFu : (((1u << S) - 1u) << (lane & ~(unsigned)(S - 1)));
}

// dW[j][k] = sum_r dz[j][r] H[k][r].  Block (jb, kb): j = jb + p nj, k = kb + q nk, so that
// neighbouring lanes read neighbouring features, whose 16-byte loads are free of bank conflicts
// (ld = 4 mod 8).  S adjacent lanes share a block's groups of four rows; a fixed butterfly
// combines them.
__device__ __forceinline__ void weight_grad(const float* dz, const float* H, int N, int K, int ld, int R,
                                            float* out) {
  const int nj = (N + 3) / 4, nk = (K + 7) / 8, nblk = nj * nk;
  int S = 1;
  while (S < 32 && 8 * S <= R && nblk * S * 2 <= NT) S *= 2;
  for (int i = (int)threadIdx.x; i < nblk * S; i += NT) {
    const int blk = i / S, sp = i % S, jb = blk / nk, kb = blk % nk;
    uint64_t acc[4][8];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 8; ++q) acc[p][q] = 0ull;
    for (int g = sp; g < R / 4; g += S) {
      ulonglong2 d[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const int j = jb + p * nj < N ? jb + p * nj : N - 1;   // past the end: computed, not written
        d[p] = *reinterpret_cast<const ulonglong2*>(dz + j * ld + 4 * g);
      }
#pragma unroll
      for (int q0 = 0; q0 < 8; q0 += 4) {
        ulonglong2 h[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int k = kb + (q0 + q) * nk < K ? kb + (q0 + q) * nk : K - 1;
          h[q] = *reinterpret_cast<const ulonglong2*>(H + k * ld + 4 * g);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            acc[p][q0 + q] = f2_fma(d[p].x, h[q].x, acc[p][q0 + q]);
            acc[p][q0 + q] = f2_fma(d[p].y, h[q].y, acc[p][q0 + q]);
          }
      }
    }
    const unsigned gm = lane_group(S);
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        float lo, hi;
        f2_unpack(acc[p][q], lo, hi);
        float v = __fadd_rn(lo, hi);
        for (int s = S / 2; s > 0; s >>= 1) v = __fadd_rn(v, __shfl_xor_sync(gm, v, s, 32));
        const int j = jb + p * nj, k = kb + q * nk;
        if (sp == 0 && j < N && k < K) out[(size_t)j * K + k] = v;
      }
  }
}

// db[j] = sum_r dz[j][r].
__device__ __forceinline__ void bias_grad(const float* dz, int N, int ld, int R, float* out) {
  int S = 1;
  while (S < 32 && 8 * S <= R && N * S * 2 <= NT) S *= 2;
  for (int i = (int)threadIdx.x; i < N * S; i += NT) {
    const int j = i / S, sp = i % S;
    float v = 0.0f;
    for (int g = sp; g < R / 4; g += S) {
      const float4 x = *reinterpret_cast<const float4*>(dz + j * ld + 4 * g);
      v = __fadd_rn(v, __fadd_rn(__fadd_rn(x.x, x.y), __fadd_rn(x.z, x.w)));
    }
    const unsigned gm = lane_group(S);
    for (int s = S / 2; s > 0; s >>= 1) v = __fadd_rn(v, __shfl_xor_sync(gm, v, s, 32));
    if (sp == 0) out[j] = v;
  }
}

constexpr long long kWait = 2000000000LL;   // bound on the wait for the weights (about 1 s)

}  // namespace

__global__ void __launch_bounds__(NT, 1) k_loss_block(const __grid_constant__ BlockLoss F) {
  extern __shared__ __align__(128) float sm[];
  __shared__ double sstat[NT / 32][4];
  const LossArgs& a = F.a;
  const int L = a.n_layers, R = F.R, ld = F.ld, tid = (int)threadIdx.x;
  const int D = a.dims[0], A = a.n_actions, NL = a.dims[L];
  uint64_t* bar = reinterpret_cast<uint64_t*>(reinterpret_cast<unsigned char*>(sm) + F.bar_off);
  if (tid == 0) {
    tcx::mbar_init(bar, 1);
    tcx::mbar_fence_init();
    // launched while k_pack_loss_w runs: the packed weights are read only after this
    asm volatile("griddepcontrol.wait;" ::: "memory");
    uint32_t total = 0u;
    for (int l = 0; l < L; ++l)
      total += (uint32_t)(a.dims[l] * F.npad[l] + (l ? a.dims[l + 1] * F.kpad[l] : 0)) * 4u;
    tcx::mbar_arrive_expect_tx(bar, total);
    for (int l = 0; l < L; ++l) {
      if (l + 1 < L || !F.withheld)
        tcx::bulk_g2s(sm + F.wt_off[l], F.Wt[l], (uint32_t)(a.dims[l] * F.npad[l]) * 4u, bar);
      if (l) tcx::bulk_g2s(sm + F.wn_off[l], F.Wn[l], (uint32_t)(a.dims[l + 1] * F.kpad[l]) * 4u, bar);
    }
  }
  for (int l = 0; l < L; ++l)
    for (int i = tid; i < a.dims[l + 1]; i += NT) sm[F.b_off[l] + i] = __ldg(a.b[l] + i);
  float* part = F.part + (size_t)blockIdx.x * F.n_params;
  double st_pg = 0.0, st_v = 0.0, st_h = 0.0, st_cf = 0.0;
  const float inv_n = 1.0f / (float)a.n;
  const int64_t r0 = (int64_t)blockIdx.x * R;
  // gather X [D][R]; rows past n are zero and get zero dZ
  {
    const int r = tid & 63;
    if (r < R) {
      const int64_t rr = r0 + r;
      const bool in = rr < a.n;
      const int64_t row = in ? (a.idx ? a.idx[rr] : rr) : 0;
      const float* src = a.obs + row / a.E * D * a.E + row % a.E;
      float* X = sm + (size_t)F.act_off[0] * ld;
      for (int d = tid >> 6; d < D; d += kLanes) X[d * ld + r] = in ? src[(int64_t)d * a.E] : 0.0f;
    }
  }
  __syncthreads();
  const bool fine = tcx::mbar_wait(bar, 0u, kWait);
  for (int l = 0; l < L; ++l) {
    const int K = a.dims[l], N = a.dims[l + 1];
    const float* X = sm + (size_t)F.act_off[l] * ld;
    float* Y = sm + (size_t)F.act_off[l + 1] * ld;
    const float* bias = sm + F.b_off[l];
    const bool th = a.act[l] == 0;
    auto epi = [&](int j, int r, auto& v) {
      const float bj = bias[j];
      constexpr int TE = sizeof(v) / sizeof(float);
#pragma unroll
      for (int e = 0; e < TE; ++e) {
        const float z = __fadd_rn(v[e], bj);
        v[e] = z;
      }
      if constexpr (TE == 4) *reinterpret_cast<float4*>(Y + j * ld + r) = make_float4(v[0], v[1], v[2], v[3]);
      else Y[j * ld + r] = v[0];
    };
    product_of(sm + F.wt_off[l], F.npad[l], K, N, X, ld, R, epi);
    __syncthreads();
    if (th) {
      const int per = R / 4;
      for (int i = tid; i < N * per; i += NT) {
        float4* y = reinterpret_cast<float4*>(Y + i / per * ld + 4 * (i % per));
        float4 v = *y;
        v.x = fwd::tanh_flat(v.x);
        v.y = fwd::tanh_flat(v.y);
        v.z = fwd::tanh_flat(v.z);
        v.w = fwd::tanh_flat(v.w);
        *y = v;
      }
      __syncthreads();
    }
  }
  // loss head, kLanes lanes per row: dL/dZ over the logits (the numbers of the fused kernel)
  {
    float* Z = sm + (size_t)F.act_off[L] * ld;
    const int r = tid / kLanes, q = tid % kLanes;
    const unsigned gm = lane_group(kLanes);
    const int64_t rr = r0 + r;
    if (r < R && rr < a.n) {
      const int64_t row = a.idx ? a.idx[rr] : rr;
      const int ac = a.action[row];
      const float ad = a.adv[row];
      const float lpo = a.algo == SIMX_ALGO_PPO ? a.logp_old[row] : 0.0f;
      const float rt = a.has_value ? a.ret[row] : 0.0f;
      float m = -__uint_as_float(0x7F800000u);
      for (int i = q; i < A; i += kLanes) m = fmaxf(m, Z[i * ld + r]);
#pragma unroll
      for (int d = kLanes / 2; d > 0; d >>= 1) m = fmaxf(m, __shfl_xor_sync(gm, m, d, kLanes));
      float S = 0.0f;
      for (int i = q; i < A; i += kLanes) S += det_exp(Z[i * ld + r] - m);
#pragma unroll
      for (int d = kLanes / 2; d > 0; d >>= 1) S += __shfl_xor_sync(gm, S, d, kLanes);
      const float lse = m + det_log(S);
      const float invS = 1.0f / S;
      float H = 0.0f;
      for (int i = q; i < A; i += kLanes) {
        const float z = Z[i * ld + r];
        H -= det_exp(z - m) * invS * (z - lse);
      }
#pragma unroll
      for (int d = kLanes / 2; d > 0; d >>= 1) H += __shfl_xor_sync(gm, H, d, kLanes);
      const float lpa = Z[ac * ld + r] - lse;
      const float zv = a.has_value ? Z[A * ld + r] : 0.0f;
      __syncwarp(gm);   // every lane of the row has read its logits
      float coef, pg;
      if (a.algo == SIMX_ALGO_REINFORCE) {
        coef = ad;
        pg = -ad * lpa;
      } else {
        const float rho = det_exp(lpa - lpo);
        const float s1 = rho * ad;
        const float s2 = fminf(fmaxf(rho, 1.0f - a.clip_eps), 1.0f + a.clip_eps) * ad;
        pg = -fminf(s1, s2);
        coef = (s1 <= s2 ? ad : 0.0f) * rho;
        if (q == 0) st_cf += fabsf(rho - 1.0f) > a.clip_eps ? 1.0 : 0.0;
      }
      for (int i = q; i < A; i += kLanes) {
        const float z = Z[i * ld + r], lp = z - lse;
        const float p = det_exp(z - m) * invS;
        const float onehot = (i == ac) ? 1.0f : 0.0f;
        Z[i * ld + r] = (-coef * (onehot - p) + a.c_entropy * p * (lp + H)) * inv_n;
      }
      if (q == 0) {
        if (a.has_value) {
          const float dv = zv - rt;
          st_v += (double)dv * (double)dv;
          Z[A * ld + r] = 2.0f * a.c_value * dv * inv_n;
        }
        st_pg += pg;
        st_h += H;
      }
    } else if (r < R) {
      for (int i = q; i < NL; i += kLanes) Z[i * ld + r] = 0.0f;
    }
  }
  __syncthreads();
  for (int l = L - 1; l >= 0; --l) {
    const int K = a.dims[l], N = a.dims[l + 1];
    const float* dz = sm + (size_t)F.act_off[l + 1] * ld;
    float* H = sm + (size_t)F.act_off[l] * ld;
    float* gW = part + F.poff[l];
    weight_grad(dz, H, N, K, ld, R, gW);
    bias_grad(dz, N, ld, R, gW + (size_t)N * K);
    __syncthreads();
    if (l > 0) {
      // dZ of the layer below over its activations: times 1 - H^2 (tanh) or 1
      const bool th = a.act[l - 1] == 0;
      auto epi = [&](int k, int r, auto& v) {
        constexpr int TE = sizeof(v) / sizeof(float);
        float* h = H + k * ld + r;
        if constexpr (TE == 4) {
          const float4 x = *reinterpret_cast<const float4*>(h);
          if (th) {
            v[0] = v[0] * (1.0f - x.x * x.x);
            v[1] = v[1] * (1.0f - x.y * x.y);
            v[2] = v[2] * (1.0f - x.z * x.z);
            v[3] = v[3] * (1.0f - x.w * x.w);
          }
          *reinterpret_cast<float4*>(h) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
          h[0] = th ? v[0] * (1.0f - h[0] * h[0]) : v[0];
        }
      };
      product_of(sm + F.wn_off[l], F.kpad[l], N, K, dz, ld, R, epi);
      __syncthreads();
    }
  }
  if (!fine && tid == 0) tcx::mbar_wait(bar, 0u, kWait);   // no copy outlives the block
  for (int d = 16; d > 0; d >>= 1) {
    st_pg += __shfl_xor_sync(0xFFFFFFFFu, st_pg, d);
    st_v += __shfl_xor_sync(0xFFFFFFFFu, st_v, d);
    st_h += __shfl_xor_sync(0xFFFFFFFFu, st_h, d);
    st_cf += __shfl_xor_sync(0xFFFFFFFFu, st_cf, d);
  }
  if ((tid & 31) == 0) {
    sstat[tid / 32][0] = st_pg;
    sstat[tid / 32][1] = st_v;
    sstat[tid / 32][2] = st_h;
    sstat[tid / 32][3] = st_cf;
  }
  const bool bad = __syncthreads_or(!fine);
  if (bad)   // the weights never landed: the gradient and the statistics say so
    for (int i = tid; i < F.n_params; i += NT) part[i] = __uint_as_float(0x7FC00000u);
  if (tid < 4) {
    double v = 0.0;
    for (int w = 0; w < NT / 32; ++w) v += sstat[w][tid];
    F.spart[(size_t)blockIdx.x * 4 + tid] = bad ? __longlong_as_double(0x7FF8000000000000LL) : v;
  }
}

namespace {

struct BlockPlan {
  bool ok;
  int R, grid;
  int npad[SIMX_MAX_LAYERS], kpad[SIMX_MAX_LAYERS], act_off[SIMX_MAX_LAYERS + 1];
  int wt_off[SIMX_MAX_LAYERS], wn_off[SIMX_MAX_LAYERS], b_off[SIMX_MAX_LAYERS], poff[SIMX_MAX_LAYERS];
  int n_params, bar_off;
  size_t smem, w_off[SIMX_MAX_LAYERS][2], part_off, spart_off, total;
};

int up4(int x) { return (x + 3) / 4 * 4; }

BlockPlan plan(const LossArgs& a) {
  BlockPlan p{};
  const int L = a.n_layers;
  if (a.grid || a.n < 1) return p;
  for (int l = 0; l + 1 < L; ++l)
    if (a.act[l] == 2) return p;
  int rows = 0, nb = 0, P = 0, wfl = 0;
  for (int l = 0; l <= L; ++l) {
    p.act_off[l] = rows;
    rows += up4(a.dims[l]);
  }
  for (int l = 0; l < L; ++l) {
    const int K = a.dims[l], N = a.dims[l + 1];
    p.npad[l] = up4(N);
    p.kpad[l] = up4(K);
    wfl += K * p.npad[l] + (l ? N * p.kpad[l] : 0);
    p.poff[l] = P;
    P += N * K + N;
    nb += up4(N);
  }
  p.n_params = P;
  const int64_t sms = sm_count();
  for (p.R = 8; p.R <= kMaxRows && (a.n + p.R - 1) / p.R > sms;) p.R += 8;
  if (p.R > kMaxRows) return p;
  p.smem = ((size_t)rows * (p.R + 4) + wfl + nb) * sizeof(float) + 16;
  if (p.smem > (size_t)kMostSmem) return p;
  p.grid = (int)((a.n + p.R - 1) / p.R);
  int off = rows * (p.R + 4);
  for (int l = 0; l < L; ++l) {
    p.wt_off[l] = off;
    off += a.dims[l] * p.npad[l];
    p.wn_off[l] = off;
    if (l) off += a.dims[l + 1] * p.kpad[l];
  }
  for (int l = 0; l < L; ++l) {
    p.b_off[l] = off;
    off += up4(a.dims[l + 1]);
  }
  p.bar_off = off * 4;
  size_t w = 0;
  auto take = [&](size_t b) {
    const size_t o = w;
    w += (b + 255) & ~(size_t)255;
    return o;
  };
  for (int l = 0; l < L; ++l) {
    p.w_off[l][0] = take((size_t)a.dims[l] * p.npad[l] * sizeof(float));
    p.w_off[l][1] = take((size_t)a.dims[l + 1] * p.kpad[l] * sizeof(float));
  }
  p.part_off = take((size_t)p.grid * P * sizeof(float));
  p.spart_off = take((size_t)p.grid * 4 * sizeof(double));
  p.total = w;
  p.ok = true;
  return p;
}

}  // namespace

int loss_block_rows(const LossArgs& a) {
  const BlockPlan p = plan(a);
  return p.ok ? p.R : 0;
}
size_t loss_block_workspace(const LossArgs& a) { return plan(a).total; }

cudaError_t launch_loss_block(const LossArgs& a, void* ws, size_t ws_bytes, cudaStream_t s) {
  const BlockPlan p = plan(a);
  if (!p.ok || ws_bytes < p.total) return cudaErrorInvalidValue;
  char* base = static_cast<char*>(ws);
  BlockLoss F{};
  F.a = a;
  LossPack pk{};
  pk.n_layers = a.n_layers;
  for (int l = 0; l < a.n_layers; ++l) {
    float* Wt = reinterpret_cast<float*>(base + p.w_off[l][0]);
    float* Wn = reinterpret_cast<float*>(base + p.w_off[l][1]);
    F.Wt[l] = Wt;
    F.Wn[l] = Wn;
    pk.W[l] = a.W[l];
    pk.Wt[l] = Wt;
    pk.Wn[l] = Wn;
    pk.N[l] = a.dims[l + 1];
    pk.K[l] = a.dims[l];
    pk.npad[l] = F.npad[l] = p.npad[l];
    pk.kpad[l] = F.kpad[l] = p.kpad[l];
    F.wt_off[l] = p.wt_off[l];
    F.wn_off[l] = p.wn_off[l];
    F.b_off[l] = p.b_off[l];
    F.poff[l] = p.poff[l];
  }
  for (int l = 0; l <= a.n_layers; ++l) F.act_off[l] = p.act_off[l];
  F.n_params = p.n_params;
  F.R = p.R;
  F.ld = p.R + 4;
  F.bar_off = p.bar_off;
  F.withheld = copies_withheld() != 0u;
  F.part = reinterpret_cast<float*>(base + p.part_off);
  F.spart = reinterpret_cast<double*>(base + p.spart_off);
  launch_pack_loss_w(pk, s);
  if (const cudaError_t e = allow_smem(k_loss_block, kMostSmem)) return e;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)p.grid);
  lc.blockDim = dim3((unsigned)NT);
  lc.dynamicSmemBytes = p.smem;
  lc.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&lc, k_loss_block, F);
  if (e != cudaSuccess) return e;
  count_launches(1);
  launch_loss_reduce(F.part, p.grid, p.n_params, F.spart, a, s);
  return cudaGetLastError();
}

}  // namespace simx
