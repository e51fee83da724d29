// rollout_route.cu — the router's rollout (ROUTE mode, Sec. 3.1, 4.1) with a policy network
// whose weights are streamed through shared memory: one thread per env runs the simulator,
// the whole block runs the policy forward.
//
// A routing step is short scalar work (one arrival, one or two batch starts), so a group of
// lanes per env that computes it redundantly (rollout.cu) spends most of its issue slots on
// copies of the same instructions: on the 4-server router about half of all instructions, and
// the 128 registers of its state and policy tiles left 16 warps per SM.  Here a block holds NE
// = threads / G envs, whose state stays in shared memory between steps.  Per step:
//   - the forward on all threads (fwd_block.cuh); beside its deepest product, warps without
//     tiles draw the arrival after the pending one (no action changes it) and the policy's
//     random word;
//   - the softmax, G threads per env; one thread per env (threads 0 .. NE-1 of an order rotated
//     from block to block, so that an SM's blocks load its schedulers evenly) draws the action
//     and puts the pending request into its queue;
//   - the servers' batch starts and features, one thread per server (G per env), whose totals
//     the env's thread adds up (integers: any order).
// What bounds it: the dependent chains of a block's step (products, then softmax, draw, starts),
// which the other blocks on the SM overlap.  c3 at 16,384 envs: 23.3 warps per SM issue in 55 % of
// the cycles, the barrier the largest stall (2.8 cycles an instruction), the FMA pipes 26 % busy; its
// kernel has 128 threads at 72 registers, without spills, so that 7 blocks fit.  Measured
// against the lane-group kernel, us per step: c4 at 65,536 envs 427 -> 317, at 4096 59 -> 32, at 1000
// 52 -> 20; c3 at 16,384 envs 49.5 -> 37.2, at 1000 12.2 -> 10.1; c3's env at 262,144 662 -> 444.
#include <cstdint>
#include <cstdlib>
#include <cstring>

#include "env_thread.cuh"
#include "fwd_block.cuh"
#include "kernels.h"

namespace simx {

using namespace envt;

namespace {

// Words of one env in shared memory: the header fields, the server of the step's action and
// the arrival time looked ahead, then six words per server.  The header fields of SINGLE mode,
// which routing neither reads nor writes, stay in global memory, and their places hold what
// lives only for the launch: the diurnal epoch whose factor is cached and the factor, the
// looked-ahead arrival's type, cost and status bits, and the policy draw's word.
enum : int { W_EPC = F_TLD, W_EPF = F_NLAST, W_NPTY = F_TLAST, W_NPC = F_LMW, W_NST = F_NA0, W_U = F_NA1 };
enum : int { W_NPT = F_COUNT, W_KK, W_SRV };
__device__ __forceinline__ bool word_saved(int w) {
  return !(w == F_TLD || w == F_NLAST || w == F_TLAST || w == F_LMW || w == F_NA0 || w == F_NA1 ||
           w == W_NPT || w == W_KK);
}
// Partial results of one thread's servers: requests started, batches, their waits by type,
// queued after the decision, status bits.
enum : int { Q_STN = 0, Q_NBAT, Q_W0L, Q_W0H, Q_W1L, Q_W1H, Q_QAF, Q_STAT, Q_WORDS };
enum : int { S_BUSY = 0, S_BSZ, S_QH0, S_QC0, S_QH1, S_QC1, S_WORDS };

// One env's words: word w at b[w * ne].
struct SmEnv {
  uint32_t* b;
  int ne;
  __device__ __forceinline__ uint32_t& operator[](int w) const { return b[w * ne]; }
  __device__ __forceinline__ uint32_t& srv(int k, int w) const { return b[(W_SRV + S_WORDS * k + w) * ne]; }
  __device__ __forceinline__ void add(int w, uint32_t v) const { b[w * ne] += v; }
};

__device__ __forceinline__ TSrv get_srv(const SmEnv& S, int k) {
  return TSrv{S.srv(k, S_BUSY), S.srv(k, S_BSZ), S.srv(k, S_QH0), S.srv(k, S_QC0), S.srv(k, S_QH1), S.srv(k, S_QC1)};
}
__device__ __forceinline__ void put_srv(const SmEnv& S, int k, const TSrv& r) {
  S.srv(k, S_BUSY) = r.busy;
  S.srv(k, S_QH0) = r.qh0;
  S.srv(k, S_QC0) = r.qc0;
  S.srv(k, S_QH1) = r.qh1;
  S.srv(k, S_QC1) = r.qc1;
}

// The observation (the ROUTE layout of rollout.cu) of one env into column x[d * ldx] and
// o[d * ld] (either may be null): server k's three features, and the others.
struct ObsOut {
  float* x;
  int ldx;
  float* o;
  int64_t ld;
  __device__ __forceinline__ void put(int d, float v) const {
    if (x) x[d * ldx] = v;
    if (o) o[(int64_t)d * ld] = v;
  }
};
__device__ __forceinline__ void observe_srv(const simx_config& c, int k, const TSrv& r, uint32_t now,
                                            const ObsOut& out) {
  const float inv_cap = __fdiv_rn(1.0f, __uint2float_rn(c.queue_cap));
  const uint32_t rem = r.busy > now ? r.busy - now : 0u;
  out.put(3 * k, over_cap(r.qc0, inv_cap));
  out.put(3 * k + 1, over_cap(c.n_types > 1 ? r.qc1 : 0u, inv_cap));
  out.put(3 * k + 2, __fdiv_rn(__uint2float_rn(rem), c.busy_norm_us));
}
__device__ __forceinline__ void observe_rest(const simx_config& c, const SmEnv& S, const ObsOut& out) {
  const int K = (int)c.n_servers;
  out.put(3 * K, __fdiv_rn(__uint_as_float(S[F_RATE]), c.rate_ref));
  if (c.obs_extra) {
    const uint32_t pty = S[F_PTY];
    out.put(3 * K + 1, pty == 0u ? 1.0f : 0.0f);
    out.put(3 * K + 2, pty == 1u ? 1.0f : 0.0f);
    const uint32_t ph = (S[F_NOW] + S[F_EPO] * c.epoch_us) % c.phase_period_us;
    out.put(3 * K + 3, __fdiv_rn(__uint2float_rn(ph), __uint2float_rn(c.phase_period_us)));
  }
}

// Ahead of the step: the policy draw's word, and the arrival after the pending one, which no
// action changes.  Only the arrival process's own state is updated here; a frozen env's stays.
template <bool TR>
__device__ __forceinline__ void look_ahead(const Ctx& x, const SmEnv& S) {
  S[W_U] = philox(S[F_TG], x.env, kStreamPolicy, 0u, x.A.key0, x.A.key1).x;
  if (S[F_STATUS] != 0u) return;
  TScal s;
  s.status = 0u;
  s.events = 0u;
  s.narr = 0u;
  s.cj = S[F_CJ];
  s.cT = S[F_CT];
  s.swi = S[F_SWI];
  s.swT = S[F_SWT];
  s.mst = S[F_MST];
  s.ep = S[F_EP];
  s.epo = S[F_EPO];
  s.ep_cached = S[W_EPC];
  s.ep_factor = __uint_as_float(S[W_EPF]);
  s.pt = S[F_PT];
  s.pty = S[F_PTY];
  s.pc = S[F_PC];
  t_next_arrival<TR>(x, s);
  S[F_CJ] = s.cj;
  S[F_CT] = s.cT;
  S[F_SWI] = s.swi;
  S[F_SWT] = s.swT;
  S[F_MST] = s.mst;
  S[F_EP] = s.ep;
  S[W_EPC] = s.ep_cached;
  S[W_EPF] = __float_as_uint(s.ep_factor);
  S[W_NPT] = s.pt;
  S[W_NPTY] = s.pty;
  S[W_NPC] = s.pc;
  S[W_NST] = s.status;
  S.add(F_NARR, s.narr);
}

// One routing decision, first part (the env's thread): the pending request joins the queue of
// the server that action `a` names.  Words for the servers' threads: the server (kNone for a
// frozen env), and the times between which they start batches.
__device__ __forceinline__ void route_apply(const Ctx& x, const SmEnv& S, int a, uint32_t extra_status) {
  const simx_config& c = x.A.cfg;
  const uint32_t kk = (uint32_t)a / c.n_bsizes, b = c.bsizes[(uint32_t)a % c.n_bsizes];
  const uint32_t status = S[F_STATUS] | extra_status;
  S[F_STATUS] = status;
  S[F_PREV] = S[F_PT];
  S[F_TG] += 1u;
  S[W_KK] = kNone;
  if (status != 0u) return;
  S[W_KK] = kk;
  const uint32_t cap = c.queue_cap, mt = S[F_PTY], now = S[F_PT];
  const uint32_t q = S.srv((int)kk, mt ? S_QC1 : S_QC0);
  if (q < cap) {
    const uint32_t slot = (S.srv((int)kk, mt ? S_QH1 : S_QH0) + q) & (cap - 1u);
    x.ring[((size_t)kk * c.n_types + mt) * cap + slot] = now;
    if ((int32_t)mt == c.cost_type) x.cost[(size_t)kk * cap + slot] = S[F_PC];
    S.srv((int)kk, mt ? S_QC1 : S_QC0) = q + 1u;
  } else {
    S.add(F_NDROP, 1u);
    S.add(mt ? F_ND1 : F_ND0, 1u);
  }
  S.srv((int)kk, S_BSZ) = b;
}

// Second part (the thread of server k): the batches that server k starts from now (if the
// request went to it) to the next arrival; `s` and the sums take their totals.
__device__ __forceinline__ void route_server(const Ctx& x, const SmEnv& S, int k, TSrv& r, TScal& s,
                                             uint32_t& stn, uint64_t& w0, uint64_t& w1, uint32_t& qafter) {
  const uint32_t kk = S[W_KK];
  r = get_srv(S, k);
  if (kk == (uint32_t)k && r.busy <= S[F_PREV]) t_start<4u>(x, s, r, k, S[F_PREV], stn, w0, w1);
  qafter += r.qc0 + r.qc1;
  if (kk != kNone)
    while (r.busy <= S[W_NPT] && r.qc0 + r.qc1 > 0u) t_start<4u>(x, s, r, k, r.busy, stn, w0, w1);
  put_srv(S, k, r);
}

// Third part (the env's thread), with the servers' totals.
__device__ __forceinline__ void route_finish(const simx_config& c, const SmEnv& S, uint32_t stn, uint32_t nbat,
                                             uint64_t w, uint32_t status) {
  if (S[W_KK] == kNone) return;
  const uint32_t now = S[F_PREV], pt = S[W_NPT];
  uint32_t gap = pt - now;
  if (gap < 1u) gap = 1u;
  const float inst = __fdiv_rn(1.0e6f, __uint2float_rn(gap));
  const float rate = __uint_as_float(S[F_RATE]);
  S[F_RATE] = __float_as_uint(__fadd_rn(rate, __fmul_rn(0.0625f, __fsub_rn(inst, rate))));
  S[F_NOW] = pt;
  S[F_PT] = pt;
  S[F_PTY] = S[W_NPTY];
  S[F_PC] = S[W_NPC];
  S[F_STATUS] = status | S[W_NST];
  S.add(F_NDISP, stn);
  S.add(F_NBAT, nbat);
  const uint64_t sw = ((uint64_t)S[F_SWLO] | ((uint64_t)S[F_SWHI] << 32)) + w;
  S[F_SWLO] = (uint32_t)sw;
  S[F_SWHI] = (uint32_t)(sw >> 32);
}

// State of the block's envs between global memory ([word][E]) and shared memory: one word of
// consecutive envs per pass, coalesced.  Word w's global array: the header fields, then per
// server busy, batch size, and per type head and length (type 1 absent with one type).
__device__ __forceinline__ uint32_t* word_ptr(const DevState& st, int w) {
  const size_t E = st.E;
  if (w < F_COUNT) return st.hdr + (size_t)w * E;
  const int i = w - W_SRV;
  const size_t k = (size_t)(i / S_WORDS);
  const int f = i % S_WORDS;
  if (f == S_BUSY) return st.srv + k * E;
  if (f == S_BSZ) return st.srv + (st.K + k) * E;
  const size_t t = f >= S_QH1 ? 1u : 0u;
  if (t >= st.T) return nullptr;
  return ((f == S_QH0 || f == S_QH1) ? st.qh : st.qc) + (k * st.T + t) * E;
}

}  // namespace

// What a phase derives from the thread's place.
struct Who {
  int vt, NE, slot, part;
  uint32_t env;
  bool live;
  float* X;        // activations, row stride ld
  float* ex;       // softmax exponentials [A][ld]
  float* red;      // [G][NE]
  SmEnv S;
  __device__ __forceinline__ explicit Who(const RolloutArgs& A, float* smem) {
    const FwdPlan& P = A.fwd;
    unsigned char* sb = reinterpret_cast<unsigned char*>(smem);
    vt = fwd::place_in_block(P.sms);
    NE = 1 << P.ne_shift;
    slot = vt & (NE - 1);
    part = vt >> P.ne_shift;
    env = blockIdx.x * (uint32_t)NE + (uint32_t)slot;
    live = env < A.st.E;
    X = smem;
    ex = smem + (size_t)P.ex_row * P.ld;
    red = reinterpret_cast<float*>(sb + P.red_off);
    S = SmEnv{reinterpret_cast<uint32_t*>(sb + P.st_off) + slot, NE};
  }
};

// The current observation of every env into X (`t` >= 0: and into step t's records), or into
// next_obs (t < 0).
__device__ __forceinline__ void phase_observe(const RolloutArgs& A, float* smem, int t) {
  const Who w(A, smem);
  if (!w.live) return;
  const ObsOut out = t >= 0 ? ObsOut{w.X + w.slot, A.fwd.ld, A.obs ? A.obs + (int64_t)t * A.obs_dim * A.ld + w.env : nullptr, A.ld}
                            : ObsOut{nullptr, 0, A.next_obs + w.env, A.next_ld};
  const int K = (int)A.cfg.n_servers;
  for (int k = w.part; k < K; k += A.G) observe_srv(A.cfg, k, get_srv(w.S, k), w.S[F_NOW], out);
  if (w.part == A.G - 1) observe_rest(A.cfg, w.S, out);
}

// Beside the products: the threads from side_vt on look ahead, one env each.
template <bool TR>
__device__ __forceinline__ void phase_ahead(const RolloutArgs& A, float* smem) {
  const FwdPlan& P = A.fwd;
  const int NE = 1 << P.ne_shift, i = fwd::place_in_block(P.sms) - P.side_vt;
  const uint32_t env = blockIdx.x * (uint32_t)NE + (uint32_t)i;
  if (i < 0 || i >= NE || env >= A.st.E) return;
  const Ctx x{A, env, nullptr, nullptr};   // the arrival process reads no ring
  look_ahead<TR>(x, SmEnv{reinterpret_cast<uint32_t*>(reinterpret_cast<unsigned char*>(smem) + P.st_off) + i, NE});
}

// The action from the logits in X, the step, the records of step t.
template <bool TR>
__device__ __forceinline__ void phase_step(const RolloutArgs& A, float* smem, int t) {
  const FwdPlan& P = A.fwd;
  const DevMlp& m = A.mlp;
  const simx_config& c = A.cfg;
  const int G = A.G, NA = m.n_actions, ld = P.ld;
  const Who w(A, smem);
  // the softmax, G threads per env: the largest logit, then the exponentials
  const float* z = w.X + w.slot;
  float* ex = w.ex + w.slot;
  const float mx = fwd::softmax_parts(z, ex, w.red, NA, ld, w.vt, w.part, w.slot, G, w.NE);
  const SmEnv& S = w.S;
  const bool owner = w.part == 0 && w.live;   // the env's thread
  const size_t env = w.live ? w.env : 0u;
  const Ctx x{A, (uint32_t)env, A.st.ring + env * c.n_servers * c.n_types * c.queue_cap,
              A.st.cost ? A.st.cost + env * c.n_servers * c.queue_cap : nullptr};
  const int64_t o = (int64_t)t * A.ld + w.env;
  if (owner) {
    if (P.side_layer < 0) look_ahead<TR>(x, S);
    float sum;
    const int a = fwd::draw(z, ex, NA, ld, mx, A.policy_mode == SIMX_POLICY_ARGMAX, S[W_U], sum);
    const fwd::Pipe p = fwd::pipe_at(reinterpret_cast<unsigned char*>(smem), P);
    route_apply(x, S, a, *p.flag ? SIMX_DEV_COPY_TIMEOUT : 0u);
    if (A.action) A.action[o] = (uint8_t)a;
    if (A.logp) A.logp[o] = __fsub_rn(__fsub_rn(z[a * ld], mx), det_log(sum));
    if (A.value) A.value[o] = m.has_value ? z[NA * ld] : 0.0f;
  }
  __syncthreads();
  // the servers, G threads per env, and their features of the next observation
  uint32_t* pq = reinterpret_cast<uint32_t*>(reinterpret_cast<unsigned char*>(smem) + P.part_off);
  const int nthr = (int)blockDim.x, K = (int)c.n_servers;
  const bool more = t + 1 < A.H;
  const ObsOut out = more ? ObsOut{w.X + w.slot, ld, A.obs ? A.obs + (int64_t)(t + 1) * A.obs_dim * A.ld + w.env : nullptr, A.ld}
                          : ObsOut{nullptr, 0, A.next_obs ? A.next_obs + w.env : nullptr, A.next_ld};
  if (w.live && w.part < K) {
    TScal s;
    s.status = s.ndisp = s.nbat = 0u;
    s.swait = 0u;
    uint32_t stn = 0u, qafter = 0u;
    uint64_t w0 = 0, w1 = 0;
    for (int k = w.part; k < K; k += G) {
      TSrv r;
      route_server(x, S, k, r, s, stn, w0, w1, qafter);
      observe_srv(c, k, r, S[W_KK] == kNone ? S[F_NOW] : S[W_NPT], out);
    }
    uint32_t* q = pq + w.vt;
    q[Q_STN * nthr] = stn;
    q[Q_NBAT * nthr] = s.nbat;
    q[Q_W0L * nthr] = (uint32_t)w0;
    q[Q_W0H * nthr] = (uint32_t)(w0 >> 32);
    q[Q_W1L * nthr] = (uint32_t)w1;
    q[Q_W1H * nthr] = (uint32_t)(w1 >> 32);
    q[Q_QAF * nthr] = qafter;
    q[Q_STAT * nthr] = s.status;
  }
  __syncthreads();
  if (!owner) return;
  uint32_t stn = 0u, nbat = 0u, qafter = 0u, status = 0u;
  uint64_t w0 = 0, w1 = 0;
  for (int i = 0; i < G && i < K; ++i) {
    const uint32_t* q = pq + (i << P.ne_shift) + w.slot;
    stn += q[Q_STN * nthr];
    nbat += q[Q_NBAT * nthr];
    w0 += (uint64_t)q[Q_W0L * nthr] | ((uint64_t)q[Q_W0H * nthr] << 32);
    w1 += (uint64_t)q[Q_W1L * nthr] | ((uint64_t)q[Q_W1H * nthr] << 32);
    qafter += q[Q_QAF * nthr];
    status |= q[Q_STAT * nthr];
  }
  route_finish(c, S, stn, nbat, w0 + w1, status);
  observe_rest(c, S, out);
  if (A.reward)
    A.reward[o] = __fsub_rn(__uint2float_rn(stn),
                            __fadd_rn(__fmul_rn(c.w_wait[0], __ull2float_rn(w0)),
                                      __fmul_rn(c.w_wait[1], __ull2float_rn(w1))));
  if (A.done) A.done[o] = (uint8_t)((S[F_TG] % c.episode_len) == 0u);
  if (A.trace) {
    int64_t* tr = A.trace + (int64_t)t * SIMX_TRACE_WIDTH * A.ld + w.env;
    tr[0] = S[F_PREV];
    tr[A.ld] = stn;
    tr[2 * A.ld] = (int64_t)(w0 + w1);
    tr[3 * A.ld] = qafter;
  }
}

template <bool TR, int NT, int MINB, bool BIG, bool GRID>
__global__ void __launch_bounds__(NT, MINB) k_route(const __grid_constant__ RolloutArgs A) {
  extern __shared__ __align__(128) float smem[];
  const FwdPlan& P = A.fwd;
  const DevMlp& m = A.mlp;
  const int NE = 1 << P.ne_shift, ld = P.ld;
  const int vt = fwd::place_in_block(P.sms), producer = (int)blockDim.x - 32;
  unsigned char* sb = reinterpret_cast<unsigned char*>(smem);
  const fwd::Pipe p = fwd::pipe_at(sb, P);
  fwd::Place at{0u, 0u};
  if (vt == producer) fwd::start<false>(m, P, p, (uint32_t)A.H * (uint32_t)P.n);
  fwd::load_biases(m, P, p);
  {
    const DevState& st = A.st;
    uint32_t* words = reinterpret_cast<uint32_t*>(sb + P.st_off);
    const uint32_t env0 = blockIdx.x * (uint32_t)NE;
    const int n = (W_SRV + S_WORDS * (int)A.cfg.n_servers) * NE;
    for (int i = (int)threadIdx.x; i < n; i += (int)blockDim.x) {
      const int w = i >> P.ne_shift, e = i & (NE - 1);
      uint32_t v = w == W_EPC ? kNone : 0u;
      if (env0 + (uint32_t)e < st.E && word_saved(w)) {
        const uint32_t* g = word_ptr(st, w);
        if (g) v = g[env0 + (uint32_t)e];
      }
      words[i] = v;
    }
    for (int i = (int)threadIdx.x; i < m.dims[0] * ld; i += (int)blockDim.x) smem[i] = 0.0f;  // envs past the last
  }
  __syncthreads();

  phase_observe(A, smem, 0);
  for (int t = 0; t < A.H; ++t) {
    fwd::forward<BIG, GRID, false>(m, P, p, at, smem, NE, ld, vt, [&]() { phase_ahead<TR>(A, smem); });
    phase_step<TR>(A, smem, t);
  }
  __syncthreads();
  if (vt == producer && *p.flag) fwd::drain(P, p);
  {
    const DevState& st = A.st;
    const uint32_t* words = reinterpret_cast<const uint32_t*>(sb + P.st_off);
    const uint32_t env0 = blockIdx.x * (uint32_t)NE;
    const int n = (W_SRV + S_WORDS * (int)A.cfg.n_servers) * NE;
    for (int i = (int)threadIdx.x; i < n; i += (int)blockDim.x) {
      const int w = i >> P.ne_shift, e = i & (NE - 1);
      if (!word_saved(w) || env0 + (uint32_t)e >= st.E) continue;
      uint32_t* g = word_ptr(st, w);
      if (g) g[env0 + (uint32_t)e] = words[i];
    }
  }
}

namespace {

template <bool TR, bool GRID>
const void* pick_kernel_t(const RolloutArgs& a) {
  if (a.fwd.big) return (const void*)k_route<TR, 256, 2, true, GRID>;
  if (a.threads > 128) return (const void*)k_route<TR, 256, 3, false, GRID>;
  return (const void*)k_route<TR, 128, 7, false, GRID>;
}
const void* pick_kernel(const RolloutArgs& a) {
  const bool tr = a.cfg.arrival_kind == SIMX_ARR_TRACE;
  if (a.mlp.grid) return tr ? pick_kernel_t<true, true>(a) : pick_kernel_t<false, true>(a);
  return tr ? pick_kernel_t<true, false>(a) : pick_kernel_t<false, false>(a);
}

int r4(int v) { return (v + 3) / 4 * 4; }

}  // namespace

// The plan of k_route for this launch: a.fwd.on when it applies (ROUTE mode, a policy network of
// at least kStageMinBytes of weights, or any with SIMX_STAGE=1; SIMX_STAGE=0 turns it off), with the
// shared-memory layout; returns the dynamic shared memory.
size_t plan_route(RolloutArgs& a) {
  std::memset(&a.fwd, 0, sizeof(a.fwd));
  const DevMlp& m = a.mlp;
  const bool net = a.policy_mode == SIMX_POLICY_SAMPLE || a.policy_mode == SIMX_POLICY_ARGMAX;
  if (a.cfg.mode != SIMX_MODE_ROUTE || !net) return 0;
  const bool forced = getenv("SIMX_LANES") || getenv("SIMX_THREADS");
  // A grid policy's forward on the tensor cores (rollout.cu) pays from about 65,536 envs on (c5:
  // 114 against 121 us per step there; c3 at 16,384 66 against 39, at 1000 46 against 11); it and
  // its FP32 form are also taken when asked for by their switches.
  if (m.grid && (forced || getenv("SIMX_TC_FORWARD") || a.st.E > 49152u)) return 0;
  int force = -1;
  if (const char* f = getenv("SIMX_STAGE"))
    if (f[0]) force = f[0] == '0' ? 0 : 1;
  if (force == 0) return 0;
  size_t wbytes = 0;
  for (int l = 0; l < m.n_layers; ++l) wbytes += (size_t)m.dims[l] * m.npad[l + 1] * sizeof(float);
  if (force < 0 && wbytes < kStageMinBytes) return 0;
  int maxd = 0;
  for (int l = 0; l <= m.n_layers; ++l) maxd = m.dims[l] > maxd ? m.dims[l] : maxd;
  const bool wide = maxd > 128;
  // Envs per block.  Every block streams the whole policy through its stages each step, so few
  // envs per block cost more copying than they win in parallel blocks: 256 threads take 8 envs
  // while that fills the SMs once, then 16, then 32 (the lane-group kernel's choice of 64-thread
  // blocks of 4 or 8 envs ran c4 at 4096 envs in 170 us per step, these in 34)
  int G = a.G, threads = a.threads;
  if (!forced) {
    const int64_t E = a.st.E, sms = sm_count();
    if (E <= 14 * sms) {
      threads = 256;
      G = 32;
    } else if (E <= 32 * sms) {
      threads = 256;
      G = 16;
    } else if (wide || E <= 96 * sms) {
      threads = 256;
      G = 8;
    }
  }
  const int NE = threads / G;
  if (NE < 4) return 0;
  FwdPlan P;
  std::memset(&P, 0, sizeof(P));
  const int last = r4(m.dims[m.n_layers]);
  P.big = threads == 256 && wide && NE >= 16;
  // 8x8 tiles on half of the threads beat 4x8 on all of them for 256-wide layers (c4, 65,536
  // envs: 320 against 340 us per step); narrower layers want every thread (c3, 16,384 envs:
  // 41 us per step with 2x8 tiles on all threads, 50 with 4x8 on half)
  if (!fwd_pick_tiles(m, NE, threads, P.big, P.big ? 40 : 75, P)) return 0;
  P.ld = NE + 4;
  P.ex_row = last;   // the exponentials follow the logits and the value row
  const int rows = r4(maxd) > last + r4(m.n_actions) ? r4(maxd) : last + r4(m.n_actions);
  size_t off = (size_t)rows * P.ld * sizeof(float);
  // the servers' partial results lie in the activation rows past the observation's, idle then
  P.part_off = (uint32_t)((size_t)r4(m.dims[0]) * P.ld * sizeof(float));
  if (P.part_off + (size_t)Q_WORDS * threads * sizeof(uint32_t) > off)
    off = P.part_off + (size_t)Q_WORDS * threads * sizeof(uint32_t);
  P.st_off = (uint32_t)off;
  off += (size_t)(W_SRV + S_WORDS * (int)a.cfg.n_servers) * NE * sizeof(uint32_t);
  // the softmax's partial maxima: past the exponentials where the activation rows reach
  P.red_off = (uint32_t)((size_t)(last + r4(m.n_actions)) * P.ld * sizeof(float));
  if (P.red_off + (size_t)threads * sizeof(float) > P.st_off) {
    P.red_off = (uint32_t)off;
    off += (size_t)threads * sizeof(float);
  }
  P.bias_off = (uint32_t)off;
  off += fwd_plan_biases(m, P);
  // Two stages, as large as keeps the blocks per SM that the registers allow: each chunk costs
  // about 500 cycles of waiting and pipeline fill, so fewer and larger ones win over more
  // stages (c4 at 65,536 envs: 2 x 32 KB 320 us per step, 4 x 16 KB 338, 8 x 8 KB 376; c3 at
  // 16,384: 2 x 10 KB 37.8, 3 x 6 KB 41.1, 6 x 2 KB 50.2)
  const int minb = P.big ? 2 : (threads > 128 ? 3 : 7) * (threads >= 128 ? 1 : 2);
  const int64_t blocks = ((int64_t)a.st.E + NE - 1) / NE;
  int64_t per_sm = (blocks + sm_count() - 1) / sm_count();
  if (per_sm > minb) per_sm = minb;
  const size_t budget = (size_t)(227 * 1024) / (size_t)per_sm - 1024;
  if (!fwd_plan_stages(m, off, budget, P)) return 0;
  P.sms = sm_count();
  // side work beside the deepest layer that leaves NE threads without tiles (the last warp apart)
  P.side_layer = -1;
  for (int l = 0; l < m.n_layers; ++l) {
    if (P.side_layer >= 0 && m.dims[l] <= m.dims[P.side_layer]) continue;
    const int nt = (NE / P.te[l]) * ((m.dims[l + 1] + P.to[l] - 1) / P.to[l]);
    const int nact = (nt + 31) & ~31;
    if (nact + (NE > 32 ? NE : 32) <= threads - 32) {
      P.side_layer = l;
      P.side_vt = nact;
    }
  }
  P.withheld = copies_withheld();
  P.on = 1;
  a.fwd = P;
  a.G = G;
  a.threads = threads;
  return fwd_smem(P);
}

cudaError_t launch_route(const RolloutArgs& a, size_t sh, cudaStream_t s) {
  const void* k = pick_kernel(a);
  if (const cudaError_t e = allow_smem(k, kMaxSmem)) return e;
  const int NE = a.threads / a.G;
  void* args[] = {const_cast<RolloutArgs*>(&a)};
  const cudaError_t e = cudaLaunchKernel(k, dim3((a.st.E + NE - 1) / NE), dim3(a.threads), args, sh, s);
  count_launches(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace simx
