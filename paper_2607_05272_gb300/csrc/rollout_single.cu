// rollout_single.cu — the single server's rollout (SINGLE mode, Sec. 3.1, 4.1) with a policy
// network (FP32 or grid): one thread per env runs the queue, the whole block the rest.
//
// A decision of the bursty single server takes in some sixty arrival candidates (up to a few
// hundred behind a long batch).  The lane-group kernel (rollout.cu) gave an env 8 to 32 lanes for
// everything: its warps ran their envs' candidate loops one after another where these differ, drew
// a step's last candidates again in the next, evaluated the policy with every warp loading every
// weight, and its code, inlined several times, missed the instruction cache (its largest stall).
// Here, per step of a block of NE = threads / G envs (state in shared memory):
//   - G threads per env write the observation; the forward runs on all threads (fwd_block.cuh),
//     with the weights resident in shared memory where they fit;
//   - the softmax, G threads per env; the env's thread draws the action and dispatches the batch;
//   - the warps take the envs in turn to their next decision, 32 candidates at a time, a lane
//     each, from a window of drawn candidates per env in shared memory, refilled 96 at a time.
// The requests' rings are in shared memory too where they fit and the horizon pays for the copy.
// What bounds it: the dependent chains between the barriers, above all a warp's through its envs'
// candidates, and the wait for the block's slowest (c2 at 4096 envs: 13.4 warps per SM issue in 38 %
// of the cycles; the barrier is the largest stall, 3.0 cycles an instruction, then fixed latencies,
// 1.8, and shared-memory loads, 1.1).  Measured against the lane-group kernel, us per step: c2 at
// 4096 envs 20.0 -> 17.0 (from a fresh reset 19.7 -> 16.4), at 30,000 196 -> 80; c2 with 65 actions
// at 65,000 421 -> 212; the paper's network at 4096 16.6 -> 14.4.
#include <cstdint>
#include <cstdlib>
#include <cstring>

#include "env_thread.cuh"
#include "fwd_block.cuh"
#include "kernels.h"

namespace simx {

using namespace envt;

namespace {

// Words of one env in shared memory: the header fields, then the server's.  Header fields of
// ROUTE mode, which a single server neither reads nor writes, stay in global memory; the places of
// five hold the end of the env's window of candidates (the first one not drawn, and the time of
// the last one drawn), whether the step advances the env (not when it was frozen), the requests it
// dispatched, and the policy draw's word.
enum : int { W_FJ = F_EP, W_TEND = F_EPO, W_GO = F_PT, W_N = F_PTY, W_U = F_PC };
enum : int { W_BUSY = F_COUNT, W_BSZ, W_QH0, W_QC0, W_QH1, W_QC1, W_WORDS };
__device__ __forceinline__ bool word_saved(int w) {
  return !(w == F_EP || w == F_EPO || w == F_PT || w == F_PTY || w == F_PC || w == F_RATE || w == W_BSZ);
}

// Word w's global array ([E]), or null (type 1 with one type).
__device__ __forceinline__ uint32_t* word_ptr(const DevState& st, int w) {
  const size_t E = st.E;
  switch (w) {
    case W_BUSY: return st.srv;
    case W_BSZ: return st.srv + E;
    case W_QH0: return st.qh;
    case W_QC0: return st.qc;
    case W_QH1: return st.T > 1 ? st.qh + E : nullptr;
    case W_QC1: return st.T > 1 ? st.qc + E : nullptr;
    default: return st.hdr + (size_t)w * E;
  }
}

struct SmEnv {
  uint32_t* b;
  int ne;
  __device__ __forceinline__ uint32_t& operator[](int w) const { return b[w * ne]; }
  __device__ __forceinline__ float f(int w) const { return __uint_as_float(b[w * ne]); }
};

// What a phase derives from the thread's place.
struct Who {
  int vt, NE, slot, part;
  uint32_t env;
  bool live;
  SmEnv S;
  unsigned char* sb;
  __device__ __forceinline__ explicit Who(const RolloutArgs& A, float* smem) {
    const FwdPlan& P = A.fwd;
    sb = reinterpret_cast<unsigned char*>(smem);
    vt = fwd::place_in_block(P.sms);
    NE = 1 << P.ne_shift;
    slot = vt & (NE - 1);
    part = vt >> P.ne_shift;
    env = blockIdx.x * (uint32_t)NE + (uint32_t)slot;
    live = env < A.st.E;
    S = SmEnv{reinterpret_cast<uint32_t*>(sb + P.st_off) + slot, NE};
  }
};

// The env's rings [T][cap] (and costs [cap] behind them): in shared memory, or the global ones.
__device__ __forceinline__ uint32_t* ring_of(const RolloutArgs& A, unsigned char* sb, int slot, uint32_t env) {
  const uint32_t per = A.cfg.n_types * A.cfg.queue_cap;
  if (A.fwd.ring_off)
    return reinterpret_cast<uint32_t*>(sb + A.fwd.ring_off) +
           (size_t)slot * (per + (A.st.cost ? A.cfg.queue_cap : 0u) + 1u);
  return A.st.ring + (size_t)env * per;
}
__device__ __forceinline__ uint32_t* cost_of(const RolloutArgs& A, uint32_t* ring, uint32_t env) {
  if (!A.st.cost) return nullptr;
  return A.fwd.ring_off ? ring + A.cfg.n_types * A.cfg.queue_cap : A.st.cost + (size_t)env * A.cfg.queue_cap;
}

// The windows: kWin candidates of env e, candidate j at e * kWin + j mod kWin: their times, meta
// words (bits 0 and 1: accepted in that state of the modulating chain; bit 2: type; bit 3: the
// time overflowed), and costs where a type has costs.
constexpr uint32_t kWin = 128;
constexpr int kRefill = 3;   // warps' worth of candidates per refill: 96 + 31 left fit the window
struct Window {
  uint32_t* T;
  uint32_t* meta;
  uint32_t* cost;
  __device__ __forceinline__ explicit Window(const RolloutArgs& A, unsigned char* sb) {
    const int n = (int)kWin << A.fwd.ne_shift;
    T = reinterpret_cast<uint32_t*>(sb + A.fwd.win_off);
    meta = T + n;
    cost = A.cfg.cost_type >= 0 ? meta + n : nullptr;
  }
};

// One warp draws the next 96 candidates from fj on into env e's window, three per lane, the chains
// of Philox rounds, logarithm and prefix sum interleaved (one after another a chunk of 32 took
// about 1400 cycles).
template <bool TR>
__device__ __forceinline__ void refill(const RolloutArgs& A, const Window& win, int e, uint32_t env,
                                       uint32_t lane, uint32_t fj, uint32_t& tend) {
  const simx_config& c = A.cfg;
  constexpr int Q = kRefill;
  U4 r[Q];
  uint32_t sum[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) r[q] = philox(fj + 32u * q + lane, env, kStreamArrival, 0u, A.key0, A.key1);
#pragma unroll
  for (int q = 0; q < Q; ++q)
    sum[q] = TR ? min(A.tr_gap[(fj + 32u * q + lane) % A.tr_n], kTimeLimit)
                : duration_us(__fmul_rn(c.cand_mean_gap_us, expo1(r[q].x)));
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    uint32_t y[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) y[q] = __shfl_up_sync(0xFFFFFFFFu, sum[q], d);
#pragma unroll
    for (int q = 0; q < Q; ++q)
      if (lane >= (uint32_t)d) {
        sum[q] += y[q];
        if (TR) sum[q] = min(sum[q], kTimeLimit);   // a trace's gaps may add up past 32 bits
      }
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const uint32_t j = fj + 32u * q + lane;
    const uint64_t t64 = (uint64_t)tend + sum[q];
    const bool over = t64 >= kTimeLimit;
    const uint32_t T = over ? kTimeLimit : (uint32_t)t64;
    const uint32_t ty = t_cand_type<TR>(A, j, r[q].y), z = r[q].z >> 8;
    const uint32_t at = (uint32_t)e * kWin + (j & (kWin - 1u));
    win.T[at] = T;
    win.meta[at] = (z < c.accept_thr[0] ? 1u : 0u) | (z < c.accept_thr[1] ? 2u : 0u) | (ty << 2) | (over ? 8u : 0u);
    if (win.cost) win.cost[at] = (int32_t)ty == c.cost_type ? t_cand_cost<TR>(A, j, r[q].w) : 0u;
    tend = __shfl_sync(0xFFFFFFFFu, T, 31);
  }
  __syncwarp();
}

// The observation (the SINGLE layout of rollout.cu), G threads per env: feature d is
// (num * mul) / den.  Into X's column (x not null) and out[d * ld] (out not null).
__device__ __forceinline__ void observe(const RolloutArgs& A, const Who& w, float* x, int ldx, float* out,
                                        int64_t ld) {
  if (!w.live) return;
  const simx_config& c = A.cfg;
  const SmEnv& S = w.S;
  const int T = (int)c.n_types, D = 2 * T + 6 + (c.obs_extra ? 6 : 0);
  const uint32_t* ring = ring_of(A, w.sb, w.slot, w.env);
  const uint32_t qc0 = S[W_QC0], qc1 = T > 1 ? S[W_QC1] : 0u;
  const uint32_t now = S[F_NOW];
  uint32_t dt = now - S[F_PREV];
  if (dt < 1u) dt = 1u;
  for (int d = w.part; d < D; d += A.G) {
    float num = 0.0f, mul = 1.0f, den = 1.0f;
    const int r = d - T;
    if (d < T) {
      num = __uint2float_rn(d ? qc1 : qc0);
      den = __uint2float_rn(c.queue_cap);
    } else if (r == 0) {
      num = __uint2float_rn(now - S[F_TLD]);
      den = c.t_window_us;
    } else if (r == 1 || r == 2 || (r >= 6 && r < 6 + T)) {
      const uint32_t h0 = qc0 > 0u ? ring[S[W_QH0]] : 0u, h1 = qc1 > 0u ? ring[c.queue_cap + S[W_QH1]] : 0u;
      if (r < 6) {
        const uint32_t head = qc0 > 0u ? ((qc1 > 0u && h1 < h0) ? 1u : 0u) : (qc1 > 0u ? 1u : kNone);
        num = head == (uint32_t)(r - 1) ? 1.0f : 0.0f;
      } else {
        const bool one = r != 6;
        num = (one ? qc1 : qc0) > 0u ? __uint2float_rn(now - (one ? h1 : h0)) : 0.0f;
        den = c.t_window_us;
      }
    } else if (r == 3) {
      num = 0.0f;   // server status: always free at a decision
    } else if (r == 4) {
      num = __uint2float_rn(S[F_NA0] + S[F_NA1]);
      mul = c.rate_scale;
      den = __uint2float_rn(dt);
    } else if (r == 5) {
      num = __uint2float_rn(S[F_NLAST]);
      den = 32.0f;
    } else {
      const int q = r - 6 - T;
      if (q < 2) {
        num = __uint2float_rn(q ? S[F_NA1] : S[F_NA0]);
        mul = c.rate_scale;
        den = __uint2float_rn(dt);
      } else if (q < 4) {
        num = S[F_TLAST] == (uint32_t)(q - 2) ? 1.0f : 0.0f;
      } else if (q == 4) {
        num = __uint2float_rn(S[F_ND0] + S[F_ND1]);
        den = 32.0f;
      } else {
        num = S.f(F_LMW);
        den = c.t_window_us;
      }
    }
    const float v = __fdiv_rn(__fmul_rn(num, mul), den);
    if (x) x[d * ldx] = v;
    if (out) out[(int64_t)d * ld] = v;
  }
}

// The env's thread: action `a` applied (the batch dispatched).
__device__ __forceinline__ void dispatch(const RolloutArgs& A, const Who& w, int a, uint32_t extra,
                                            float& reward, uint32_t& now0, uint32_t& n, uint64_t& Wt,
                                            uint32_t& qafter) {
  const simx_config& c = A.cfg;
  const SmEnv& S = w.S;
  const uint32_t cap = c.queue_cap;
  uint32_t* ring = ring_of(A, w.sb, w.slot, w.env);
  uint32_t* cost = cost_of(A, ring, w.env);
  uint32_t kk, b;
  if (c.action_layout == 1) {   // a = 0: Wait (batch 0); a >= 1: type, batch 1 .. n_bsizes
    kk = a == 0 ? 0u : (uint32_t)(a - 1) / c.n_bsizes;
    b = a == 0 ? 0u : (uint32_t)(a - 1) % c.n_bsizes + 1u;
  } else {
    kk = (uint32_t)a / c.n_bsizes;
    b = c.bsizes[(uint32_t)a % c.n_bsizes];
  }
  TScal s;
  s.status = S[F_STATUS] | extra;
  const bool frozen = s.status != 0u;
  now0 = S[F_NOW];
  uint32_t qc0 = S[W_QC0], qc1 = S[W_QC1], qh0 = S[W_QH0], qh1 = S[W_QH1];
  n = 0u;
  Wt = 0;
  if (!frozen) {
    const uint32_t q = kk ? qc1 : qc0, head = kk ? qh1 : qh0;
    uint64_t csum = 0;
    n = b < q ? b : q;
    const uint32_t* rk = ring + kk * cap;
    const bool costed = (int32_t)kk == c.cost_type;
    for (uint32_t j = 0; j < n; j += 4u) {
      uint32_t t4[4], c4[4];
#pragma unroll
      for (uint32_t i = 0; i < 4u; ++i) {
        const uint32_t at = (head + j + i) & (cap - 1u);
        t4[i] = j + i < n ? rk[at] : now0;
        c4[i] = costed && j + i < n ? cost[at] : 0u;
      }
#pragma unroll
      for (uint32_t i = 0; i < 4u; ++i) {
        Wt += (uint64_t)(now0 - t4[i]);
        csum += c4[i];
      }
    }
    if (kk) {
      qh1 = (head + n) & (cap - 1u);
      qc1 -= n;
    } else {
      qh0 = (head + n) & (cap - 1u);
      qc0 -= n;
    }
    if (n > 0u) {
      const uint64_t L = costed ? (uint64_t)c.alpha_us[kk] + csum
                                : (uint64_t)c.alpha_us[kk] + (uint64_t)c.beta_us[kk] * n;
      S[W_BUSY] = t_add(now0, t_speed(c, 0, L), s.status);
      S[F_NLAST] = n;
      S[F_TLAST] = kk;
      S[F_TLD] = now0;
      S[F_LMW] = __float_as_uint(__fdiv_rn(__ull2float_rn(Wt), __uint2float_rn(n)));
      S[F_NBAT] += 1u;
    }
    S[F_NDISP] += n;
    const uint64_t sw = ((uint64_t)S[F_SWLO] | ((uint64_t)S[F_SWHI] << 32)) + Wt;
    S[F_SWLO] = (uint32_t)sw;
    S[F_SWHI] = (uint32_t)(sw >> 32);
  }
  reward = __fsub_rn(__uint2float_rn(n), __fmul_rn(c.w_wait[kk], __ull2float_rn(Wt)));
  qafter = qc0 + qc1;
  S[F_PREV] = now0;
  S[F_TG] += 1u;
  S[F_NA0] = S[F_NA1] = S[F_ND0] = S[F_ND1] = 0u;
  S[F_STATUS] = s.status;
  S[W_GO] = frozen ? 0u : 1u;
  S[W_N] = n;
  S[W_QC0] = qc0;
  S[W_QC1] = qc1;
  S[W_QH0] = qh0;
  S[W_QH1] = qh1;
}

// The warps take the envs to their next decision point: to the batch's end, if one runs; then, or
// with nothing queued there, to the next accepted arrival and every candidate up to its time.
template <bool TR>
__device__ __forceinline__ void phase_advance(const RolloutArgs& A, float* smem) {
  const simx_config& c = A.cfg;
  const Who w(A, smem);
  const Window win(A, w.sb);
  const uint32_t lane = (uint32_t)w.vt & 31u, cap = c.queue_cap;
  constexpr uint32_t kAll = 0xFFFFFFFFu;
  // the next env from a counter: a long batch's env keeps its warp for many candidates
  uint32_t* next = reinterpret_cast<uint32_t*>(w.sb + A.fwd.part_off);
  for (;;) {
    int e = 0;
    if (lane == 0u) e = (int)atomicAdd(next, 1u);
    e = __shfl_sync(kAll, e, 0);
    if (e >= w.NE) break;
    const uint32_t env = blockIdx.x * (uint32_t)w.NE + (uint32_t)e;
    const SmEnv S{reinterpret_cast<uint32_t*>(w.sb + A.fwd.st_off) + e, w.NE};
    if (env >= A.st.E || S[W_GO] == 0u) continue;
    uint32_t* ring = ring_of(A, w.sb, e, env);
    uint32_t* cost = cost_of(A, ring, env);
    const Ctx x{A, env, nullptr, nullptr};
    TScal s;
    s.status = S[F_STATUS];
    s.cj = S[F_CJ];
    s.cT = S[F_CT];
    s.swi = S[F_SWI];
    s.swT = S[F_SWT];
    s.mst = S[F_MST];
    s.events = 0u;
    uint32_t fj = S[W_FJ], tend = S[W_TEND], now = S[F_NOW], target = S[W_BUSY];
    uint32_t qc0 = S[W_QC0], qc1 = S[W_QC1];
    const uint32_t qh0 = S[W_QH0], qh1 = S[W_QH1];
    uint32_t na0 = 0u, na1 = 0u, nd0 = 0u, nd1 = 0u;
    bool seek = S[W_N] == 0u, tied = false;
    for (;;) {
      if (fj - s.cj < 32u) {   // fewer than a warp's worth of candidates drawn
        refill<TR>(A, win, e, env, lane, fj, tend);
        fj += 32u * kRefill;
      }
      // the next 32 candidates
      const uint32_t at0 = (uint32_t)e * kWin + ((s.cj + lane) & (kWin - 1u));
      const uint32_t T = win.T[at0], meta = win.meta[at0];
      if (seek) {
        // the first accepted of them, the chain's switches walked tentatively
        uint32_t st = s.mst, ms = s.mst, si = s.swi, sT = s.swT, nsw = 0u, flag = 0u;
        const uint32_t Tmax = __shfl_sync(kAll, T, 31);
        if (c.n_mod_states == 2) {
          TScal v;
          v.status = 0u;
          while (sT <= Tmax && nsw <= kEventCap) {
            if (T >= sT) st ^= 1u;
            ms ^= 1u;
            si += 1u;
            sT = t_switch_time(x, si, sT, v.status);
            nsw += 1u;
          }
          flag = v.status;
        }
        const uint32_t bm = __ballot_sync(kAll, (meta >> st) & 1u);
        if (!bm) {
          if (__ballot_sync(kAll, meta & 8u)) s.status |= kStTime;
          s.status |= flag;
          s.mst = ms;
          s.swi = si;
          s.swT = sT;
          s.cj += 32u;
          s.cT = Tmax;
          s.events += 32u + nsw;
          if (s.events > kEventCap) {
            s.status |= kStEvent;
            break;
          }
          continue;
        }
        target = __shfl_sync(kAll, T, __ffs(bm) - 1);
        seek = false;
        tied = true;
      }
      // those up to the target
      const bool cons = T <= target;
      const uint32_t m = __popc(__ballot_sync(kAll, cons));
      if (__ballot_sync(kAll, lane <= m && (meta & 8u))) s.status |= kStTime;   // up to the first left
      if (m > 0u) {
        const uint32_t Tlast = __shfl_sync(kAll, T, (int)m - 1);
        uint32_t st = s.mst;
        bool full = false;
        if (c.n_mod_states == 2) {
          while (s.swT <= Tlast) {
            if (T >= s.swT) st ^= 1u;
            s.mst ^= 1u;
            s.swi += 1u;
            s.swT = t_switch_time(x, s.swi, s.swT, s.status);
            if (t_count(s)) {
              full = true;
              break;
            }
          }
        }
        if (full) {
          now = target;
          break;
        }
        const bool acc = cons && ((meta >> st) & 1u);
        const bool one = (meta & 4u) != 0u;
        const uint32_t b0 = __ballot_sync(kAll, acc && !one), b1 = __ballot_sync(kAll, acc && one);
        const uint32_t n0 = __popc(b0), n1 = __popc(b1), room0 = cap - qc0, room1 = cap - qc1;
        if (acc) {
          const uint32_t rank = __popc((one ? b1 : b0) & ((1u << lane) - 1u));
          if (rank < (one ? room1 : room0)) {
            const uint32_t at = ((one ? qh1 + qc1 : qh0 + qc0) + rank) & (cap - 1u);
            ring[(one ? cap : 0u) + at] = T;
            if ((int32_t)(one ? 1 : 0) == c.cost_type) cost[at] = win.cost[at0];
          }
        }
        const uint32_t a0 = n0 < room0 ? n0 : room0, a1 = n1 < room1 ? n1 : room1;
        qc0 += a0;
        qc1 += a1;
        na0 += n0;
        na1 += n1;
        nd0 += n0 - a0;
        nd1 += n1 - a1;
        s.cj += m;
        s.cT = Tlast;
        s.events += m;
        if (s.events > kEventCap) {
          s.status |= kStEvent;
          now = target;
          break;
        }
        if (m == 32u) continue;
      }
      if (c.n_mod_states == 2) {
        while (s.swT <= target) {
          s.mst ^= 1u;
          s.swi += 1u;
          s.swT = t_switch_time(x, s.swi, s.swT, s.status);
          if (t_count(s)) break;
        }
      }
      now = target;
      if (tied || qc0 + qc1 > 0u) break;
      seek = true;   // the server is free and idle
    }
    if (lane == 0u) {
      S[W_FJ] = fj;
      S[W_TEND] = tend;
      S[F_NOW] = now;
      S[F_CJ] = s.cj;
      S[F_CT] = s.cT;
      S[F_SWI] = s.swi;
      S[F_SWT] = s.swT;
      S[F_MST] = s.mst;
      S[F_STATUS] = s.status;
      S[F_NARR] += na0 + na1;
      S[F_NDROP] += nd0 + nd1;
      S[F_NA0] = na0;
      S[F_NA1] = na1;
      S[F_ND0] = nd0;
      S[F_ND1] = nd1;
      S[W_QC0] = qc0;
      S[W_QC1] = qc1;
    }
  }
}

// The action from the logits in X, the dispatch, the records of step t.
__device__ __forceinline__ void phase_step(const RolloutArgs& A, float* smem, int t) {
  const FwdPlan& P = A.fwd;
  const DevMlp& m = A.mlp;
  const Who w(A, smem);
  const int NA = m.n_actions, ld = P.ld;
  const float* z = smem + w.slot;
  float* ex = smem + (size_t)P.ex_row * ld + w.slot;
  const float mx = fwd::softmax_parts(z, ex, reinterpret_cast<float*>(w.sb + P.red_off), NA, ld, w.vt, w.part,
                                      w.slot, A.G, w.NE);
  if (w.part != 0 || !w.live) return;
  float sum;
  const int a = fwd::draw(z, ex, NA, ld, mx, A.policy_mode == SIMX_POLICY_ARGMAX, w.S[W_U], sum);
  const int64_t o = (int64_t)t * A.ld + w.env;
  if (A.action) A.action[o] = (uint8_t)a;
  if (A.logp) A.logp[o] = __fsub_rn(__fsub_rn(z[a * ld], mx), det_log(sum));
  if (A.value) A.value[o] = m.has_value ? z[NA * ld] : 0.0f;
  float reward;
  uint32_t now, n, qafter;
  uint64_t W;
  const fwd::Pipe p = fwd::pipe_at(w.sb, P);
  dispatch(A, w, a, *p.flag ? SIMX_DEV_COPY_TIMEOUT : 0u, reward, now, n, W, qafter);
  if (A.reward) A.reward[o] = reward;
  if (A.done) A.done[o] = (uint8_t)((w.S[F_TG] % A.cfg.episode_len) == 0u);
  if (A.trace) {
    int64_t* tr = A.trace + (int64_t)t * SIMX_TRACE_WIDTH * A.ld + w.env;
    tr[0] = now;
    tr[A.ld] = n;
    tr[2 * A.ld] = (int64_t)W;
    tr[3 * A.ld] = qafter;
  }
}

// The rings between global and shared memory, coalesced (in = true: into shared memory).
__device__ __forceinline__ void copy_rings(const RolloutArgs& A, float* smem, bool in) {
  if (!A.fwd.ring_off) return;
  const int NE = 1 << A.fwd.ne_shift;
  const uint32_t per = A.cfg.n_types * A.cfg.queue_cap, cap = A.cfg.queue_cap;
  unsigned char* sb = reinterpret_cast<unsigned char*>(smem);
  for (int e = 0; e < NE; ++e) {
    const uint32_t env = blockIdx.x * (uint32_t)NE + (uint32_t)e;
    if (env >= A.st.E) break;
    uint32_t* r = ring_of(A, sb, e, env);
    uint32_t* g = A.st.ring + (size_t)env * per;
    for (uint32_t i = threadIdx.x; i < per; i += blockDim.x)
      if (in) r[i] = g[i]; else g[i] = r[i];
    if (A.st.cost) {
      uint32_t* gc = A.st.cost + (size_t)env * cap;
      for (uint32_t i = threadIdx.x; i < cap; i += blockDim.x)
        if (in) r[per + i] = gc[i]; else gc[i] = r[per + i];
    }
  }
}

}  // namespace

template <bool TR, bool GRID>
__global__ void __launch_bounds__(256, 3) k_single(const __grid_constant__ RolloutArgs A) {
  extern __shared__ __align__(128) float smem[];
  const FwdPlan& P = A.fwd;
  const DevMlp& m = A.mlp;
  const DevState& st = A.st;
  const int NE = 1 << P.ne_shift, ld = P.ld;
  const int vt = fwd::place_in_block(P.sms), producer = (int)blockDim.x - 32;
  unsigned char* sb = reinterpret_cast<unsigned char*>(smem);
  const fwd::Pipe p = fwd::pipe_at(sb, P);
  fwd::Place at{0u, 0u};
  if (vt == producer) fwd::start<true>(m, P, p, P.resident ? (uint32_t)P.n : (uint32_t)A.H * (uint32_t)P.n);
  fwd::load_biases(m, P, p);
  uint32_t* words = reinterpret_cast<uint32_t*>(sb + P.st_off);
  const uint32_t env0 = blockIdx.x * (uint32_t)NE;
  for (int i = (int)threadIdx.x; i < W_WORDS * NE; i += (int)blockDim.x) {
    const int w = i >> P.ne_shift, e = i & (NE - 1);
    uint32_t v = 0u;
    if (env0 + (uint32_t)e < st.E) {
      // an empty window: it ends at the next candidate
      const uint32_t* g = w == W_FJ ? word_ptr(st, F_CJ) : w == W_TEND ? word_ptr(st, F_CT)
                          : word_saved(w) ? word_ptr(st, w) : nullptr;
      if (g) v = g[env0 + (uint32_t)e];
    }
    words[i] = v;
  }
  for (int i = (int)threadIdx.x; i < m.dims[0] * ld; i += (int)blockDim.x) smem[i] = 0.0f;  // envs past the last
  copy_rings(A, smem, true);
  __syncthreads();
  for (int t = 0; t < A.H; ++t) {
    {
      const Who w(A, smem);
      observe(A, w, smem + w.slot, ld, A.obs ? A.obs + (int64_t)t * A.obs_dim * A.ld + w.env : nullptr, A.ld);
      if (w.vt == 0) *reinterpret_cast<uint32_t*>(sb + P.part_off) = 0u;   // phase_advance's counter
      if (w.part == A.G - 1) w.S[W_U] = philox(w.S[F_TG], w.env, kStreamPolicy, 0u, A.key0, A.key1).x;
    }
    fwd::forward<false, GRID, true>(m, P, p, at, smem, NE, ld, vt, []() {});
    phase_step(A, smem, t);
    __syncthreads();
    phase_advance<TR>(A, smem);
    __syncthreads();
  }
  if (A.next_obs) {
    const Who w(A, smem);
    observe(A, w, nullptr, 0, A.next_obs + w.env, A.next_ld);
  }
  if (vt == producer && *p.flag) fwd::drain(P, p);
  for (int i = (int)threadIdx.x; i < W_WORDS * NE; i += (int)blockDim.x) {
    const int w = i >> P.ne_shift, e = i & (NE - 1);
    if (!word_saved(w) || env0 + (uint32_t)e >= st.E) continue;
    uint32_t* g = word_ptr(st, w);
    if (g) g[env0 + (uint32_t)e] = words[i];
  }
  copy_rings(A, smem, false);
}

// The plan of k_single for this launch: a.fwd.on when it applies (SINGLE mode and a policy network;
// SIMX_STAGE=0 turns it off); returns the dynamic shared memory.
size_t plan_single(RolloutArgs& a) {
  std::memset(&a.fwd, 0, sizeof(a.fwd));
  const DevMlp& m = a.mlp;
  const bool net = a.policy_mode == SIMX_POLICY_SAMPLE || a.policy_mode == SIMX_POLICY_ARGMAX;
  if (a.cfg.mode != SIMX_MODE_SINGLE || !net) return 0;
  const bool forced = getenv("SIMX_LANES") || getenv("SIMX_THREADS");
  if (m.grid && forced) return 0;   // the lane-group kernel's grid forwards are asked for by shape
  if (const char* f = getenv("SIMX_STAGE"))
    if (f[0] == '0') return 0;
  int maxd = 0;
  for (int l = 0; l <= m.n_layers; ++l) maxd = m.dims[l] > maxd ? m.dims[l] : maxd;
  int G = a.G, threads = a.threads;
  const int64_t E = a.st.E, sms = sm_count();
  size_t wbytes = 0;
  for (int l = 0; l < m.n_layers; ++l) wbytes += (size_t)m.dims[l] * m.npad[l + 1] * sizeof(float);
  if (!forced) {
    // Up to one env per warp slot the lane-group kernel's 32 lanes per env are faster (c2 at 512
    // envs 9.4 against 11.4 us per step, c1 at 1000 4.7 against 6.3), and so they are, with fewer
    // lanes, for a policy too small to share (c1's 450 weights at 8000 envs: 9.7 against 15.5;
    // at 65,000 62.0 against 56.5).  16 envs per block while two blocks per SM hold them all
    // (c2 at 4096: 17.1 against 21.4 with 32), then 32 (at 30,000: 80 against 114).
    if (E <= 16 * sms || (wbytes < 4096 && E <= 256 * sms)) return 0;
    threads = 256;
    G = E <= 32 * sms ? 16 : 8;
  }
  const int NE = threads / G;
  if (NE < 4) return 0;
  FwdPlan P;
  std::memset(&P, 0, sizeof(P));
  if (!fwd_pick_tiles(m, NE, threads, false, 75, P)) return 0;
  auto r4 = [](int v) { return (v + 3) / 4 * 4; };
  const int last = r4(m.dims[m.n_layers]);
  P.ld = NE + 4;
  P.ex_row = last;
  const int rows = r4(maxd) > last + r4(m.n_actions) ? r4(maxd) : last + r4(m.n_actions);
  size_t off = (size_t)rows * P.ld * sizeof(float);
  P.st_off = (uint32_t)off;
  off += (size_t)W_WORDS * NE * sizeof(uint32_t);
  P.red_off = (uint32_t)off;
  off += (size_t)threads * sizeof(float);
  P.bias_off = (uint32_t)off;
  off += fwd_plan_biases(m, P);
  off = (off + 15) / 16 * 16;
  P.part_off = (uint32_t)off;   // phase_advance's counter
  off += 16;
  P.win_off = (uint32_t)off;
  off += (size_t)(a.cfg.cost_type >= 0 ? 3 : 2) * kWin * NE * sizeof(uint32_t);
  // the rings, where they leave two blocks per SM and the horizon is long enough to pay
  const size_t rings = (size_t)NE * (a.cfg.n_types * a.cfg.queue_cap + (a.cfg.cost_type >= 0 ? a.cfg.queue_cap : 0u) + 1u) * sizeof(uint32_t);
  const size_t half = 113 * 1024 - 512;
  if (a.H >= 16 && off + rings + wbytes + 512 <= half) {
    P.ring_off = (uint32_t)off;
    off += rings;
  }
  if (!fwd_plan_resident(m, off, half, P) && !fwd_plan_stages(m, off, half, P)) return 0;
  P.side_layer = -1;
  P.sms = (int)sms;
  P.withheld = copies_withheld();
  P.on = 1;
  a.fwd = P;
  a.G = G;
  a.threads = threads;
  return fwd_smem(P);
}

cudaError_t launch_single(const RolloutArgs& a, size_t sh, cudaStream_t s) {
  const bool tr = a.cfg.arrival_kind == SIMX_ARR_TRACE;
  auto k = a.mlp.grid ? (tr ? k_single<true, true> : k_single<false, true>)
                      : (tr ? k_single<true, false> : k_single<false, false>);
  if (const cudaError_t e = allow_smem(k, kMaxSmem)) return e;
  const int NE = a.threads / a.G;
  k<<<(a.st.E + NE - 1) / NE, a.threads, sh, s>>>(a);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace simx
