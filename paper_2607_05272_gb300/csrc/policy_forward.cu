// policy_forward.cu — the batched policy forward (Sec. 4.2), and the plans of the
// block forward (fwd_block.cuh) that it shares with the router's rollout.
//
// A persistent block takes tiles of NE observation columns: 64 columns on 256 threads with 8x8
// register tiles where there are columns enough, fewer for small batches.  The weights stream
// through two shared-memory stages without a break from tile to tile, so they cross L2 once per
// 64 columns.  65,536 columns of c4's policy: 296 us, 38 TFLOP/s (the lane-group kernel, which
// read the weights through L1 once per 32 columns and waited on it: 896 us).  Bound by the
// products' issue and shared-memory reads (fwd_block.cuh): 14.6 warps per SM issue in 53 % of the
// cycles, stalled on the math pipes and on fixed latencies; tanh is an eighth (with identity layers
// the same call takes 250 us, in a loop of its own in which it takes 287).
#include <cstdint>
#include <cstring>

#include "fwd_block.cuh"
#include "kernels.h"

namespace simx {

template <int MINB, bool BIG, bool GRID>
__global__ void __launch_bounds__(256, MINB) k_forward_block(const __grid_constant__ PolicyArgs A) {
  extern __shared__ __align__(128) float smem[];
  const FwdPlan& P = A.fwd;
  const DevMlp& m = A.mlp;
  const int vt = (int)threadIdx.x, NE = 1 << P.ne_shift, G = 256 >> P.ne_shift, ld = P.ld;
  const int slot = vt & (NE - 1), part = vt >> P.ne_shift, producer = 256 - 32;
  unsigned char* sb = reinterpret_cast<unsigned char*>(smem);
  const fwd::Pipe p = fwd::pipe_at(sb, P);
  fwd::Place at{0u, 0u};
  const int64_t tiles = (A.n + NE - 1) >> P.ne_shift;
  const int64_t mine = (tiles - blockIdx.x + gridDim.x - 1) / gridDim.x;
  if (vt == producer) fwd::start<false>(m, P, p, (uint32_t)mine * (uint32_t)P.n);
  fwd::load_biases(m, P, p);
  const int D = m.dims[0], NA = m.n_actions;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t col = (tile << P.ne_shift) + slot;
    const bool live = col < A.n;
    for (int d = part; d < D; d += G) smem[d * ld + slot] = live ? __ldg(A.obs + (int64_t)d * A.ld + col) : 0.0f;
    fwd::forward<BIG, GRID, false>(m, P, p, at, smem, NE, ld, vt, []() {});
    if (*p.flag) {   // a wait for weights ran out: every output from here on says so
      for (int j = part; j < m.dims[m.n_layers]; j += G) smem[j * ld + slot] = __uint_as_float(0x7FC00000u);
      __syncthreads();
    }
    const float* z = smem + slot;
    if (live && A.logits)
      for (int j = part; j < NA; j += G) A.logits[(int64_t)j * A.ld + col] = z[j * ld];
    if (live && A.value && part == 0) A.value[col] = m.has_value ? z[NA * ld] : 0.0f;
    if (A.action || A.logp) {
      float* ex = smem + (size_t)P.ex_row * ld + slot;
      const float mx = fwd::softmax_parts(z, ex, reinterpret_cast<float*>(sb + P.red_off), NA, ld, vt, part,
                                          slot, G, NE);
      if (live && part == 0) {
        const uint32_t env = A.env_base + (uint32_t)col;
        const uint32_t word = philox(A.step, env, kStreamPolicy, 0u, A.key0, A.key1).x;
        float sum;
        const int a = fwd::draw(z, ex, NA, ld, mx, A.mode == SIMX_POLICY_ARGMAX, word, sum);
        if (A.action) A.action[col] = (uint8_t)a;
        if (A.logp) A.logp[col] = __fsub_rn(__fsub_rn(z[a * ld], mx), det_log(sum));
      }
    }
    __syncthreads();   // the next tile's observations replace the logits
  }
  if (vt == producer && *p.flag) fwd::drain(P, p);
}

bool fwd_pick_tiles(const DevMlp& m, int NE, int threads, bool big, int pct, FwdPlan& P) {
  static const int shapes[6][2] = {{8, 8}, {4, 8}, {2, 8}, {4, 4}, {2, 4}, {1, 4}};
  P.ne_shift = 0;
  while ((1 << P.ne_shift) < NE) ++P.ne_shift;
  if ((1 << P.ne_shift) != NE) return false;
  for (int l = 0; l < m.n_layers; ++l) {
    const int N = m.dims[l + 1], Np = m.npad[l + 1];
    int best = -1, best_nt = 0;
    for (int q = big ? 0 : 1; q < 6; ++q) {
      const int te = shapes[q][0], to = shapes[q][1];
      if (NE % te != 0 || Np % to != 0) continue;
      const int nt = (NE / te) * ((N + to - 1) / to);
      if (nt > threads) continue;
      if (100 * nt >= pct * threads) {
        best = q;
        break;
      }
      if (nt > best_nt) {
        best_nt = nt;
        best = q;
      }
    }
    if (best < 0) return false;
    P.te[l] = shapes[best][0];
    P.to[l] = shapes[best][1];
  }
  return true;
}

size_t fwd_plan_biases(const DevMlp& m, FwdPlan& P) {
  int nb = 0;
  for (int l = 0; l < m.n_layers; ++l) {
    P.boff[l] = nb;
    nb += m.dims[l + 1];
  }
  return (size_t)nb * sizeof(float);
}

bool fwd_plan_stages(const DevMlp& m, size_t off, size_t budget, FwdPlan& P) {
  int maxnp = 0;
  for (int l = 1; l <= m.n_layers; ++l) maxnp = m.npad[l] > maxnp ? m.npad[l] : maxnp;
  off = (off + 127) / 128 * 128;
  P.off = (uint32_t)off;
  P.S = 2;
  uint32_t cb = 32768;
  while (cb > 2048 && off + (size_t)P.S * cb + 128 > budget) cb -= 1024;
  if (cb < (uint32_t)maxnp * 4u) cb = (uint32_t)(maxnp * 4 + 127) / 128u * 128u;   // at least one row
  if (off + (size_t)P.S * cb + 128 > 227 * 1024) return false;
  P.cb = cb;
  P.n = 0;
  for (int l = 0; l < m.n_layers; ++l) {
    const int K = m.dims[l];
    int rpc = (int)(cb / (uint32_t)(m.npad[l + 1] * 4));
    if (rpc >= 16) rpc &= ~7;   // whole passes of the unrolled loop
    rpc = rpc < K ? rpc : K;
    P.rpc[l] = rpc;
    P.cnt[l] = (K + rpc - 1) / rpc;
    P.n += P.cnt[l];
  }
  P.bar_off = (uint32_t)(off + (size_t)P.S * cb);
  return true;
}

bool fwd_plan_resident(const DevMlp& m, size_t off, size_t budget, FwdPlan& P) {
  off = (off + 127) / 128 * 128;
  P.off = (uint32_t)off;
  size_t w = 0;
  P.S = P.n = m.n_layers;
  for (int l = 0; l < m.n_layers; ++l) {
    P.woff[l] = (uint32_t)w;
    w += (size_t)m.dims[l] * m.npad[l + 1] * sizeof(float);   // a multiple of 16 bytes
    P.rpc[l] = m.dims[l];
    P.cnt[l] = 1;
  }
  if (off + w + 256 > budget) return false;
  P.bar_off = (uint32_t)(off + (w + 15) / 16 * 16);
  P.cb = 0;
  P.resident = 1;
  return true;
}

size_t fwd_smem(const FwdPlan& P) { return P.bar_off + fwd::pipe_bytes(P.S); }

// Policies (FP32 or grid) whose layers the register tiles cover.
bool plan_policy_block(PolicyArgs& p) {
  std::memset(&p.fwd, 0, sizeof(p.fwd));
  const DevMlp& m = p.mlp;
  int maxd = 0;
  for (int l = 0; l <= m.n_layers; ++l) maxd = m.dims[l] > maxd ? m.dims[l] : maxd;
  // columns per block: as many as still give every SM a block
  const int64_t sms = sm_count();
  FwdPlan P;
  std::memset(&P, 0, sizeof(P));
  const int NE = p.n > 48 * sms ? 64 : p.n > 32 * sms ? 32 : p.n > 14 * sms ? 16 : 8;
  const int last = (m.dims[m.n_layers] + 3) / 4 * 4, exr = (m.n_actions + 3) / 4 * 4;
  P.big = NE >= 32 && maxd > 128;
  if (!fwd_pick_tiles(m, NE, 256, P.big, P.big ? 40 : 75, P)) return false;
  P.ld = NE + 4;
  P.ex_row = last;
  const int rows = (maxd + 3) / 4 * 4 > last + exr ? (maxd + 3) / 4 * 4 : last + exr;
  size_t off = (size_t)rows * P.ld * sizeof(float);
  P.red_off = (uint32_t)off;
  off += 256 * sizeof(float);
  P.bias_off = (uint32_t)off;
  off += fwd_plan_biases(m, P);
  const int minb = P.big ? 2 : 3;
  const int64_t tiles = (p.n + NE - 1) / NE;
  int64_t per_sm = (tiles + sms - 1) / sms;
  if (per_sm > minb) per_sm = minb;
  if (!fwd_plan_stages(m, off, (size_t)(227 * 1024) / (size_t)per_sm - 1024, P)) return false;
  P.side_layer = -1;
  P.sms = (int)(per_sm * sms < tiles ? per_sm * sms : tiles);   // the grid
  P.withheld = copies_withheld();
  P.on = 1;
  p.fwd = P;
  return true;
}

cudaError_t launch_policy_block(const PolicyArgs& p, cudaStream_t s) {
  auto k = p.mlp.grid ? (p.fwd.big ? k_forward_block<2, true, true> : k_forward_block<3, false, true>)
                      : (p.fwd.big ? k_forward_block<2, true, false> : k_forward_block<3, false, false>);
  const size_t sh = fwd_smem(p.fwd);
  if (const cudaError_t e = allow_smem(k, kMaxSmem)) return e;
  k<<<(unsigned)p.fwd.sms, 256, sh, s>>>(p);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace simx
