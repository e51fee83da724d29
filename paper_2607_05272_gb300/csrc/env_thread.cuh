// env_thread.cuh — one environment per thread: the scalar state, the arrival process and
// the batch start of the simulator (Sec. 3.1, 3.2) as one thread runs them, shared by the
// policy-free step (step_thread.cu) and the router's rollout (rollout_route.cu).  The event
// semantics are those of the lane-group kernel (rollout.cu) and of the oracle, step for step.
#pragma once
#include <cstdint>

#include "kernels.h"

namespace simx {
namespace envt {

// One env's scalar state in a thread's registers.
struct TScal {
  uint32_t now, tg, cj, cT, swi, swT, mst, ep, epo, pt, pty, pc;
  uint32_t narr, ndrop, ndisp, nbat, tld, prev, nlast, tlast, na0, na1, nd0, nd1, status, events;
  uint64_t swait;
  float lmw, rate, ep_factor;
  uint32_t ep_cached;
};

__device__ __forceinline__ uint32_t t_add(uint32_t a, uint64_t b, uint32_t& status) {
  const uint64_t s = (uint64_t)a + b;
  if (s >= kTimeLimit) {
    status |= kStTime;
    return kTimeLimit;
  }
  return (uint32_t)s;
}

struct Ctx {
  const RolloutArgs& A;
  uint32_t env;
  uint32_t* ring;  // this env's rings [K][T][cap]
  uint32_t* cost;  // this env's cost rings [K][cap] or null
};

__device__ __forceinline__ uint32_t t_type(const simx_config& c, uint32_t w1) {
  return (c.n_types > 1 && (w1 >> 8) >= c.type0_thr) ? 1u : 0u;
}

__device__ __forceinline__ uint32_t t_cost(const simx_config& c, uint32_t w3) {
  const float E = expo1(w3);
  if (c.cost_kind == 0) return duration_us(__fmul_rn(c.cost_scale_us, det_exp(__fmul_rn(c.pareto_inv_alpha, E))));
  return duration_us(__fmul_rn(c.cost_scale_us, E));
}

__device__ __forceinline__ bool t_count(TScal& s) {
  if (++s.events > kEventCap) {
    s.status |= kStEvent;
    return true;
  }
  return false;
}

// Time of the modulating chain's switch i, given switch i - 1 at t.
__device__ __forceinline__ uint32_t t_switch_time(const Ctx& x, uint32_t i, uint32_t t, uint32_t& status) {
  if (x.A.cfg.dwell_kind == 1) return t_add(t, duration_us(x.A.cfg.dwell_mean_us), status);  // a square wave
  const U4 w = philox(i, x.env, kStreamSwitch, 0u, x.A.key0, x.A.key1);
  return t_add(t, duration_us(__fmul_rn(x.A.cfg.dwell_mean_us, expo1(w.x))), status);
}

static __device__ __forceinline__ void t_switches(const Ctx& x, TScal& s, uint32_t limit) {
  if (x.A.cfg.n_mod_states < 2) return;
  while (s.swT <= limit) {
    if (t_count(s)) return;
    s.mst ^= 1u;
    s.swi += 1u;
    s.swT = t_switch_time(x, s.swi, s.swT, s.status);
  }
}

// Candidate s.cj: its Philox words and its time (a drawn gap, or under trace replay,
// TR, entry cj mod n of the trace).  TR is a template parameter so that the generated-
// arrival kernels carry none of the trace code.
template <bool TR>
__device__ __forceinline__ uint32_t t_cand(const Ctx& x, TScal& s, U4& w) {
  w = philox(s.cj, x.env, kStreamArrival, 0u, x.A.key0, x.A.key1);
  const uint32_t gap = TR ? x.A.tr_gap[s.cj % x.A.tr_n]
                          : duration_us(__fmul_rn(x.A.cfg.cand_mean_gap_us, expo1(w.x)));
  return t_add(s.cT, gap, s.status);
}

// Type and cost of candidate j: the trace's when it has them, else drawn.
template <bool TR>
__device__ __forceinline__ uint32_t t_cand_type(const RolloutArgs& A, uint32_t j, uint32_t w1) {
  if (TR && A.tr_type) {
    const uint32_t t = A.tr_type[j % A.tr_n];
    return t < A.cfg.n_types ? t : A.cfg.n_types - 1u;
  }
  return t_type(A.cfg, w1);
}

template <bool TR>
__device__ __forceinline__ uint32_t t_cand_cost(const RolloutArgs& A, uint32_t j, uint32_t w3) {
  return (TR && A.tr_cost) ? A.tr_cost[j % A.tr_n] : t_cost(A.cfg, w3);
}

// ROUTE mode: the next arrival into the pending slot.
template <bool TR>
__device__ void t_next_arrival(const Ctx& x, TScal& s) {
  const simx_config& c = x.A.cfg;
  for (;;) {
    if (t_count(s)) return;
    U4 w;
    if (TR || c.arrival_kind != SIMX_ARR_DIURNAL) {  // THINNED or TRACE
      const uint32_t T = t_cand<TR>(x, s, w);
      t_switches(x, s, T);
      const bool acc = (w.z >> 8) < c.accept_thr[s.mst];
      const uint32_t j = s.cj;
      s.cj += 1u;
      s.cT = T;
      if (!acc) continue;
      s.pty = t_cand_type<TR>(x.A, j, w.y);
      s.pc = ((int32_t)s.pty == c.cost_type) ? t_cand_cost<TR>(x.A, j, w.w) : 0u;
      s.pt = T;
      s.narr += 1u;
      return;
    }
    if (s.ep_cached != s.ep) {
      const U4 we = philox(s.ep, x.env, kStreamEpoch, 0u, x.A.key0, x.A.key1);
      s.ep_factor = det_exp(__fmul_rn(c.burst_sigma, normal01(we.x, we.y)));
      s.ep_cached = s.ep;
    }
    const float rate = __fmul_rn(c.diurnal_rate[(s.ep + s.epo) % c.diurnal_len], s.ep_factor);
    const float mean = __fdiv_rn(1.0e6f, rate);
    w = philox(s.cj, x.env, kStreamArrival, 0u, x.A.key0, x.A.key1);
    const uint32_t gap = duration_us(__fmul_rn(mean, expo1(w.x)));
    s.cj += 1u;
    const uint64_t end = (uint64_t)(s.ep + 1u) * (uint64_t)c.epoch_us;
    if ((uint64_t)s.cT + gap < end) {
      s.cT = t_add(s.cT, gap, s.status);
      s.pt = s.cT;
      s.pty = t_type(c, w.y);
      s.pc = ((int32_t)s.pty == c.cost_type) ? t_cost(c, w.w) : 0u;
      s.narr += 1u;
      return;
    }
    if (end >= kTimeLimit) {
      s.status |= kStTime;
      s.cT = kTimeLimit;
    } else {
      s.cT = (uint32_t)end;
    }
    s.ep += 1u;
  }
}

// Batch time L on server k scaled by its speed s/16, rounded to the nearest microsecond.
__device__ __forceinline__ uint64_t t_speed(const simx_config& c, int k, uint64_t L) {
  const uint64_t s = c.srv_speed16[k] ? c.srv_speed16[k] : 16u;
  return (L * s + 8u) >> 4;
}

// ROUTE mode: one server's queue state.
struct TSrv {
  uint32_t busy, bsize, qh0, qc0, qh1, qc1;
};

// ROUTE mode: server i (state r) starts a batch at time st (the oldest-head type, tie:
// type 0).  U: requests of the batch whose ring loads are issued together (registers allowing:
// 4 spilled the policy-free step's 96-register form, 128 against 134 us at 1,048,576 envs).
template <uint32_t U>
__device__ __forceinline__ void t_start(const Ctx& x, TScal& s, TSrv& r, int srv, uint32_t st,
                                        uint32_t& stn, uint64_t& w0, uint64_t& w1) {
  const simx_config& c = x.A.cfg;
  const uint32_t cap = c.queue_cap, T = c.n_types;
  uint32_t* rs = x.ring + (size_t)srv * T * cap;
  uint32_t h;
  if (r.qc0 > 0u && r.qc1 > 0u) {
    h = rs[cap + r.qh1] < rs[r.qh0] ? 1u : 0u;
  } else if (r.qc0 > 0u) {
    h = 0u;
  } else if (r.qc1 > 0u) {
    h = 1u;
  } else {
    return;
  }
  const uint32_t qn = h ? r.qc1 : r.qc0;
  const uint32_t head = h ? r.qh1 : r.qh0;
  const uint32_t n = r.bsize < qn ? r.bsize : qn;
  const bool costed = (int32_t)h == c.cost_type;
  uint64_t W = 0, csum = 0;
  if constexpr (U == 1u) {
    for (uint32_t j = 0; j < n; ++j) {
      const uint32_t slot = (head + j) & (cap - 1u);
      W += (uint64_t)(st - rs[h * cap + slot]);
      if (costed) csum += x.cost[(size_t)srv * cap + slot];
    }
  } else {
    // U requests at a time, their loads in flight together
    for (uint32_t j = 0; j < n; j += U) {
      uint32_t tu[U], cu[U];
#pragma unroll
      for (uint32_t i = 0; i < U; ++i) {
        const uint32_t slot = (head + j + i) & (cap - 1u);
        tu[i] = j + i < n ? rs[h * cap + slot] : st;
        cu[i] = costed && j + i < n ? x.cost[(size_t)srv * cap + slot] : 0u;
      }
#pragma unroll
      for (uint32_t i = 0; i < U; ++i) {
        W += (uint64_t)(st - tu[i]);
        csum += cu[i];
      }
    }
  }
  if (h) {
    r.qh1 = (head + n) & (cap - 1u);
    r.qc1 -= n;
  } else {
    r.qh0 = (head + n) & (cap - 1u);
    r.qc0 -= n;
  }
  const uint64_t L = costed ? (uint64_t)c.alpha_us[h] + csum
                            : (uint64_t)c.alpha_us[h] + (uint64_t)c.beta_us[h] * n;
  r.busy = t_add(st, t_speed(c, srv, L), s.status);
  stn += n;
  if (h) w1 += W; else w0 += W;
  s.ndisp += n;
  s.swait += W;
  s.nbat += 1u;
}

// q / cap for a power-of-two capacity: multiplying by the exact reciprocal 2^-k gives
// the bits of the IEEE division (no rounding either way for these small integers).
__device__ __forceinline__ float over_cap(uint32_t q, float inv_cap) {
  return __fmul_rn(__uint2float_rn(q), inv_cap);
}

}  // namespace envt
}  // namespace simx
