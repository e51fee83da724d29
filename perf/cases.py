"""The work that a user of this engine has it do, as cases that can be timed.

Each case is one pass through the public Python entry points (``simx`` and ``train``):

* ``step``     one decision of every env of a running simulator (sim_step_batched): the
               gym-style loop of a caller with its own agent, or of a baseline;
* ``rollout``  reset and ``rollout_collect`` over a horizon with a policy network, on the
               FP32 policy or on the grid policy, or with a policy-free baseline;
* ``returns``  GAE, or REINFORCE returns with the mean baseline, over a rollout buffer;
* ``forward``  ``policy_forward`` over a batch of observations (bootstrap values, serving);
* ``loss``     ``ppo_loss_grad`` of one minibatch (or a whole buffer), FP32 or TF32;
* ``adam``     one optimiser step with norm clipping;
* ``train``    ``Trainer.iteration``: rollout, returns, every minibatch's loss and update.

Sizes are those of the repository's workloads (``workloads.CONFIGS``, ``MLP_SHAPES``, the
benchmark, the trainer's defaults); ``draw`` spreads them over the range around those.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_05272_gb300 import simx, train
from paper_2607_05272_gb300 import workloads as W


def listed():
    return [
        # An agent outside the library steps 1,000 router envs with its own actions: the
        # smallest call, where launch latency is everything.
        dict(name="step external c3 1000", kind="step", workload="c3", envs=1000, mode="external"),
        # The Shortest-Queue baseline on the scale sweep's largest env count: state traffic.
        dict(name="step sq c5 1048576", kind="step", workload="c5", envs=1048576, mode="sq"),
        # One 1000-step episode of the smallest workload (64 envs): a dependent chain of steps.
        dict(name="rollout c1 64x1000", kind="rollout", workload="c1", envs=64, horizon=1000,
             mode="sample", grid=False),
        # The bursty single-server workload at its own size: narrow policy, many arrivals.
        dict(name="rollout c2 4096x512", kind="rollout", workload="c2", envs=4096, horizon=512,
             mode="sample", grid=False),
        # The 4-server router at its own size: 128-wide policy with a value row.
        dict(name="rollout c3 16384x256", kind="rollout", workload="c3", envs=16384, horizon=256,
             mode="sample", grid=False),
        # The benchmark's workload (8 servers, 256-wide policy), a quarter of its horizon.
        dict(name="rollout c4 65536x128", kind="rollout", workload="c4", envs=65536, horizon=128,
             mode="sample", grid=False),
        # GAE over the router's rollout buffer.
        dict(name="gae 256x16384", kind="returns", T=256, E=16384, lam=0.95),
        # Bootstrap values and actions for the benchmark's env count.
        dict(name="forward c4 65536", kind="forward", workload="c4", n=65536, mode="sample"),
        # The benchmark's minibatch on the tensor cores, and the router's in FP32 (the
        # trainer's default precision).
        dict(name="loss c4 8192 tf32", kind="loss", workload="c4", rows=8192, buffer=262144,
             algo="ppo", precision="tf32"),
        dict(name="loss c3 8192 fp32", kind="loss", workload="c3", rows=8192, buffer=1048576,
             algo="ppo", precision="fp32"),
        # Whole training iterations, as the trainer runs them: PPO with four epochs of
        # minibatches on the benchmark's env, REINFORCE over the whole buffer on c2.
        dict(name="train c4 ppo 4096x64", kind="train", workload="c4", envs=4096, horizon=64,
             algo="ppo", minibatch=8192, precision="tf32"),
        dict(name="train c2 reinforce 4096x512", kind="train", workload="c2", envs=4096,
             horizon=512, algo="reinforce", minibatch=8192, precision="fp32"),
    ]


def _log(rng, lo, hi):
    """A whole number from lo to hi, even over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _params(name):
    dims, _ = W.mlp_dims(name)
    return sum(k * n + n for k, n in zip(dims[:-1], dims[1:]))


ROUTERS = ("c3", "c4", "c3h", "c3s", "c3t")
# Decisions x parameters of the largest listed rollout, which no drawn one exceeds.
MOST_ROLLOUT = 65536 * 128 * 84273


def draw(rng):
    kind = rng.choice(["step", "rollout", "rollout", "rollout", "returns", "forward", "loss",
                       "loss", "loss", "adam", "train", "train"])
    if kind == "step":
        # single-server envs take far more simulated time per decision and would reach the
        # simulator's time limit in a long run of steps: routers only
        wl = rng.choice(["c3", "c4", "c3h", "c3t"])
        hi = 1048576 if wl != "c4" else 131072
        return dict(kind=kind, workload=wl, envs=_log(rng, 100, hi),
                    mode=rng.choice(["external", "sq", "rr", "random"]))
    if kind == "rollout":
        wl = rng.choice(["c1", "c2", "c3", "c4", "c5", "burst", "c3h", "c1w", "c2w", "c1p", "c2t",
                         "c3t", "c3s"])
        mode = rng.choice(["sample", "sample", "sample", "argmax", "baseline"])
        if mode == "baseline":
            mode = rng.choice(["sq", "rr", "random"] if wl in ROUTERS + ("c5",) else ["static", "random"])
        grid = mode in ("sample", "argmax") and wl in ("c2", "c3", "c5", "c1p") and rng.random() < 0.3
        envs = _log(rng, 50, 65536)
        most = min(512, max(16, MOST_ROLLOUT // (2 * envs * max(_params(wl), 20000))))
        return dict(kind=kind, workload=wl, envs=envs, horizon=_log(rng, 16, max(17, most)),
                    mode=mode, grid=grid)
    if kind == "returns":
        T = _log(rng, 16, 2048)
        E = _log(rng, 50, min(262144, (1 << 26) // T))
        return dict(kind=kind, T=T, E=E, lam=rng.choice([0.95, 1.0, -1.0]))
    if kind == "forward":
        return dict(kind=kind, workload=rng.choice(["c2", "c3", "c4", "c1p", "c2w"]),
                    n=_log(rng, 100, 65536), mode=rng.choice(["sample", "argmax"]))
    if kind == "loss":
        wl = rng.choice(["c1", "c2", "c3", "c4", "c1p", "c3s", "c2w"])
        algo = rng.choice(["ppo", "reinforce"])
        rows = _log(rng, 500, 65536 if wl == "c4" else 262144)
        if rng.random() < 0.4:
            rows = rng.choice([1024, 4096, 8192, 16384])
        buffer = max(131072, 1 << rows.bit_length())
        if algo == "reinforce":  # over a whole buffer
            rows = buffer = 4096 * _log(rng, 1, 16 if wl == "c4" else 64)
        return dict(kind=kind, workload=wl, rows=rows, buffer=buffer, algo=algo,
                    precision=rng.choice(["fp32", "tf32"]))
    if kind == "adam":
        wl = rng.choice(["c1", "c2", "c3", "c4", "c1p", "c3s"])
        return dict(kind=kind, workload=wl, clip=rng.choice([0.0, 0.5, 0.5, 0.5]),
                    state=rng.randrange(1, 1000))
    wl = rng.choice(["c2", "c3", "c4", "c3s", "c1p"])
    algo = rng.choice(["reinforce", "ppo"]) if W.mlp_dims(wl)[1] else "reinforce"
    envs = _log(rng, 256, 4096)
    return dict(kind=kind, workload=wl, envs=envs, horizon=_log(rng, 32, 128), algo=algo,
                minibatch=rng.choice([1024, 4096, 8192]), precision=rng.choice(["fp32", "tf32"]))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _weights(name, seed):
    """Flat fp32 parameters of `name`'s policy (initial weights, small biases as after some
    updates), in the order W0, b0, W1, b1, ..., masked entries zero."""
    dims, hv = W.mlp_dims(name)
    Ws, bs = W.policy_weights(name, dims, int(seed))
    rng = np.random.default_rng([int(seed), 7])
    bs = [(b + 0.02 * rng.standard_normal(b.shape)).astype(np.float32) for b in bs]
    flat = np.concatenate([np.concatenate([w.ravel(), b.ravel()]) for w, b in zip(Ws, bs)])
    return torch.from_numpy(flat.astype(np.float32)).cuda(), dims, hv


def _obs(shape, D, g):
    """Observations [..., D, n] of the ranges the simulator gives: queue fractions in [0, 1],
    waits and busy times over their normaliser (heavy-tailed), indicators."""
    u = torch.rand(shape, device="cuda", generator=g)
    f = torch.arange(D, device="cuda") % 3
    f = f.view(-1, 1)
    tail = torch.where(u > 0.98, -40.0 * torch.log1p(-u), -torch.log1p(-u))
    return torch.where(f == 0, u * u, torch.where(f == 1, tail, (u > 0.5).float())).contiguous()


def _split(flat, dims):
    out, off = [], 0
    for k, n in zip(dims[:-1], dims[1:]):
        out.append((flat[off:off + n * k].view(n, k), flat[off + n * k:off + n * k + n]))
        off += n * k + n
    return out


def _mlp(X, layers, acts):
    """The policy network on rows X in the layers' own precision."""
    for l, (w, b) in enumerate(layers):
        X = X @ w.T + b
        if l + 1 < len(layers):
            a = acts[l]
            X = torch.tanh(X) if a == "tanh" else X if a == "identity" else \
                torch.nn.functional.gelu(X, approximate="tanh")
    return X


def _grid_policy(name, seed):
    dims, hv = W.mlp_dims(name)
    n = len(dims) - 1
    gx, ew = [4] + [7] * (n - 1), [6] * n
    Ws, bs = W.grid_weights(dims, int(seed), gx, ew)
    return simx.Policy([torch.from_numpy(w).cuda() for w in Ws],
                       [torch.from_numpy(b).cuda() for b in bs], hv, W.mlp_acts(name), grid=gx)


def _loss_inputs(case, seed):
    """A rollout buffer of `buffer` rows (E envs per step), the minibatch's rows, old
    log-probabilities of a policy a few updates older, and returns and advantages."""
    name, g = case["workload"], _gen(seed)
    flat, dims, hv = _weights(name, seed)
    E = 4096
    H = case["buffer"] // E
    obs = _obs((H, dims[0], E), dims[0], g)
    A = dims[-1] - (1 if hv else 0)
    acts = W.mlp_acts(name)
    layers = _split(flat, dims)
    action = torch.empty((H, E), dtype=torch.uint8, device="cuda")
    logp = torch.empty((H, E), device="cuda")
    for h in range(H):
        z = torch.log_softmax(_mlp(obs[h].T, layers, acts)[:, :A], dim=1)
        a = torch.argmax(z - torch.log(-torch.log(torch.rand(z.shape, device="cuda", generator=g)
                                                  .clamp_(1e-12, 1 - 1e-7))), dim=1)
        action[h] = a.to(torch.uint8)
        logp[h] = z.gather(1, a[:, None])[:, 0]
    logp += 0.1 * torch.randn((H, E), device="cuda", generator=g)
    adv = 4.0 * torch.randn((H, E), device="cuda", generator=g)
    ret = adv - 6.0 + 2.0 * torch.randn((H, E), device="cuda", generator=g)
    rows = case["rows"]
    # a whole buffer is passed without an index, a minibatch as rows of a permutation
    idx = None if rows == H * E else torch.randperm(H * E, device="cuda", generator=g)[:rows].clone()
    return flat, dims, hv, dict(obs=obs, action=action, logp=logp), ret, adv, idx


LOSS = dict(clip_eps=0.2, c_value=0.5, c_entropy=0.01)


def prepare(case, seed):
    kind, seed = case["kind"], int(seed) & 0x7FFFFFFF
    if kind in ("step", "rollout", "train"):
        name, E = case["workload"], case["envs"]
        cfg = W.CONFIGS[name](E)
    if kind == "step":
        sim = simx.Sim(cfg)
        sim.reset(seed)
        n = cfg["n_servers"] * cfg["n_bsizes"]
        s = dict(case=case, sim=sim, obs=torch.empty((sim.D, E), device="cuda"),
                 reward=torch.empty(E, device="cuda"),
                 done=torch.empty(E, dtype=torch.uint8, device="cuda"),
                 action=torch.empty(E, dtype=torch.uint8, device="cuda"), actions=None)
        if case["mode"] == "external":
            s["actions"] = torch.randint(0, n, (E,), dtype=torch.int32, device="cuda",
                                         generator=_gen(seed))
        return s
    if kind == "rollout":
        dims, hv = W.mlp_dims(name)
        pol = None
        if case["mode"] in ("sample", "argmax"):
            pol = _grid_policy(name, seed) if case["grid"] else \
                simx.Policy.from_flat(_weights(name, seed)[0], dims, hv, W.mlp_acts(name))
        sim = simx.Sim(cfg)
        buf = simx.alloc_rollout(E, sim.D, case["horizon"], has_value=hv and pol is not None)
        return dict(case=case, sim=sim, pol=pol, buf=buf, seed=seed)
    if kind == "returns":
        g, T, E = _gen(seed), case["T"], case["E"]
        rew = 2.0 * torch.rand((T, E), device="cuda", generator=g) - \
            0.5 * torch.empty((T, E), device="cuda").exponential_(generator=g)
        done = (torch.rand((T, E), device="cuda", generator=g) < 1.0 / 256).to(torch.uint8)
        s = dict(case=case, rew=rew, done=done, ret=torch.empty_like(rew),
                 adv=torch.empty_like(rew), val=None,
                 last=10.0 * torch.randn(E, device="cuda", generator=g))
        if case["lam"] >= 0:
            s["val"] = 10.0 * torch.randn((T, E), device="cuda", generator=g)
        else:
            s["mean"] = torch.empty(1, device="cuda")
            s["ws"] = torch.empty(simx.returns_baseline_workspace_size(T * E), dtype=torch.uint8,
                                  device="cuda")
        return s
    if kind == "forward":
        name, n = case["workload"], case["n"]
        flat, dims, hv = _weights(name, seed)
        pol = simx.Policy.from_flat(flat, dims, hv, W.mlp_acts(name))
        A = dims[-1] - (1 if hv else 0)
        return dict(case=case, pol=pol, obs=_obs((dims[0], n), dims[0], _gen(seed)), seed=seed,
                    logits=torch.empty((A, n), device="cuda"),
                    value=torch.empty(n, device="cuda") if hv else None,
                    action=torch.empty(n, dtype=torch.uint8, device="cuda"),
                    logp=torch.empty(n, device="cuda"),
                    ws=torch.empty(simx.policy_forward_workspace_size(pol), dtype=torch.uint8,
                                   device="cuda"))
    if kind == "loss":
        flat, dims, hv, buf, ret, adv, idx = _loss_inputs(case, seed)
        pol = simx.Policy.from_flat(flat, dims, hv, W.mlp_acts(case["workload"]))
        return dict(case=case, pol=pol, buf=buf, ret=ret, adv=adv, idx=idx,
                    grad=torch.empty(pol.n_params, device="cuda"),
                    stats=torch.empty(5, device="cuda"),
                    ws=torch.empty(simx.ppo_loss_grad_workspace_size(pol, case["rows"]),
                                   dtype=torch.uint8, device="cuda"))
    if kind == "adam":
        flat, grad, m, v, mask = _adam_inputs(case, seed)
        n = flat.numel()
        return dict(case=case, params=flat, grad=grad, m=m, v=v, mask=mask,
                    t=torch.full((1,), case["state"], dtype=torch.int64, device="cuda"),
                    ws=torch.empty(simx.adam_workspace_size(n), dtype=torch.uint8, device="cuda"))
    dims, hv = W.mlp_dims(name)
    tr = train.Trainer(cfg, dims, hv, W.mlp_acts(name), W.policy_weights(name, dims, seed),
                       W.param_mask(name, dims), algo=case["algo"], horizon=case["horizon"],
                       minibatch=case["minibatch"], seed=seed, precision=case["precision"],
                       graph=True)
    return dict(case=case, tr=tr)


def _adam_inputs(case, seed):
    name = case["workload"]
    flat, dims, _ = _weights(name, seed)
    n, g = flat.numel(), _gen(seed)
    scale = torch.exp(torch.randn(n, device="cuda", generator=g) - 4.0)
    grad = scale * torch.randn(n, device="cuda", generator=g)
    m = 0.3 * scale * torch.randn(n, device="cuda", generator=g)
    v = scale * scale * torch.rand(n, device="cuda", generator=g).add_(0.5)
    mask = W.param_mask(name, dims)
    mask = None if mask is None else torch.from_numpy(mask).cuda()
    return flat, grad, m, v, mask


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        s["sim"].step(case["mode"], actions=s["actions"], obs=s["obs"], reward=s["reward"],
                      done=s["done"], action=s["action"])
        return [s["obs"], s["reward"], s["done"], s["action"]]
    if kind == "rollout":
        # an evaluation or collection from a fresh start: the envs reset, then the horizon
        s["sim"].reset(s["seed"])
        s["sim"].rollout(case["mode"], case["horizon"], s["buf"], s["pol"])
        return s["buf"]
    if kind == "returns":
        if s["val"] is not None:
            simx.compute_returns_gae(s["rew"], s["done"], 0.99, case["lam"], s["ret"], adv=s["adv"],
                                     val=s["val"], last_val=s["last"])
            return dict(ret=s["ret"], adv=s["adv"])
        simx.compute_returns_gae(s["rew"], s["done"], 0.99, -1.0, s["ret"], last_val=s["last"])
        simx.returns_baseline(s["ret"], s["adv"], s["mean"], s["ws"])
        return dict(ret=s["ret"], adv=s["adv"], mean=s["mean"])
    if kind == "forward":
        simx.policy_forward(s["pol"], s["obs"], case["n"], case["mode"], s["seed"], 3,
                            logits=s["logits"], value=s["value"], action=s["action"],
                            logp=s["logp"], workspace=s["ws"])
        return dict(logits=s["logits"], value=s["value"], action=s["action"], logp=s["logp"])
    if kind == "loss":
        c_value = LOSS["c_value"] if s["pol"].has_value else 0.0
        simx.ppo_loss_grad(s["pol"], s["buf"], s["ret"], s["adv"], s["idx"], case["rows"],
                           case["algo"], LOSS["clip_eps"], c_value, LOSS["c_entropy"], s["grad"],
                           s["stats"], s["ws"], precision=case["precision"])
        return dict(grad=s["grad"], stats=s["stats"])
    if kind == "adam":
        simx.adam_step(s["params"], s["grad"], s["m"], s["v"], s["t"], 3e-4,
                       max_grad_norm=case["clip"], mask=s["mask"], workspace=s["ws"])
        return dict(params=s["params"], m=s["m"], v=s["v"])
    tr = s["tr"]
    tr.iteration()
    # the first moment is left out: near a minimum it is a difference of a few noisy gradients
    return dict(params=tr.params, v=tr.v)


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _rollout_work(name, envs, horizon, net, has_value):
    """Records written per decision, and the policy's multiply-adds (the simulator's integer
    work is not counted)."""
    cfg = W.CONFIGS[name](1)
    rec = 4 * cfg["obs_dim"] + 1 + 4 + 4 + 1 + (4 if has_value else 0)
    d = envs * horizon
    return dict(bytes=d * rec + 4 * _params(name) * net, flops=2 * d * _params(name) * net)


def _loss_work(name, rows):
    dims, hv = W.mlp_dims(name)
    P = _params(name)
    per = 4 * dims[0] + 1 + 4 + 4 + (4 if hv else 0) + 8
    # forward and weight gradient of every layer, input gradient of every layer but the first
    return dict(bytes=rows * per + 8 * P, flops=rows * (6 * P - 2 * dims[0] * dims[1]))


def work(case):
    kind = case["kind"]
    if kind == "step":
        cfg = W.CONFIGS[case["workload"]](1)
        K, T = cfg["n_servers"], cfg["n_types"]
        # the env's state words in and out, and the step's outputs
        words = 29 + 2 * K + 2 * K * T
        per = 8 * words + 4 * cfg["obs_dim"] + 6 + (4 if case["mode"] == "external" else 0)
        return dict(bytes=case["envs"] * per, flops=0)
    if kind == "rollout":
        hv = W.mlp_dims(case["workload"])[1]
        net = case["mode"] in ("sample", "argmax")
        return _rollout_work(case["workload"], case["envs"], case["horizon"], net, hv and net)
    if kind == "returns":
        n = case["T"] * case["E"]
        # reward, done (and value) in; returns and advantages out
        return dict(bytes=n * (17 if case["lam"] >= 0 else 13), flops=n * 8)
    if kind == "forward":
        dims, _ = W.mlp_dims(case["workload"])
        P = _params(case["workload"])
        return dict(bytes=case["n"] * (4 * dims[0] + 4 * dims[-1] + 5) + 4 * P,
                    flops=2 * case["n"] * P)
    if kind == "loss":
        return _loss_work(case["workload"], case["rows"])
    if kind == "adam":
        return dict(bytes=28 * _params(case["workload"]), flops=12 * _params(case["workload"]))
    name, rows = case["workload"], case["envs"] * case["horizon"]
    w = _rollout_work(name, case["envs"], case["horizon"], True, W.mlp_dims(name)[1])
    P = _params(name)
    if case["algo"] == "reinforce":
        mb, n = rows, 1
    else:
        mb, n = min(case["minibatch"], rows), 4 * (rows // case["minibatch"])
    lw = _loss_work(name, mb)
    return dict(bytes=w["bytes"] + rows * 17 + n * (lw["bytes"] + 28 * P),
                flops=w["flops"] + n * lw["flops"])


# ---------------------------------------------------------------------------
# What another correct implementation may differ by
# ---------------------------------------------------------------------------
def tolerance(case):
    kind = case["kind"]
    if kind in ("step", "rollout", "forward"):
        # the simulator, the policy's fp32 chains and the sampler are specified to the bit
        return "exact"
    if kind == "returns":
        return dict(rel=2e-6, max=2e-5)
    if kind == "loss":
        # TF32 inputs round at 2^-11, and in PPO rows at the clip's edge fall on either side of
        # it (measured 8e-4 typically, 8e-3 and 0.09 of the rms in one of 24); FP32 sums over
        # the rows measured 4e-7, with PPO's edge again the exception
        if case["precision"] == "tf32":
            return dict(rel=2e-2, max=0.3)
        return dict(rel=1e-4, max=1e-2) if case["algo"] == "ppo" else dict(rel=4e-6, max=1e-4)
    if kind == "adam":
        return dict(rel=2e-6, max=2e-5)
    # REINFORCE takes one update per iteration; PPO's many updates on few rows carry a
    # difference of rounding in one of them on (measured with the rows of every minibatch in
    # another order: parameters up to 5e-3, single values up to 0.15 of the rms)
    if case["algo"] == "ppo":
        return dict(rel=0.02, max=0.6)
    return dict(rel=1e-2, max=0.1) if case["precision"] == "tf32" else dict(rel=1e-5, max=1e-4)


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _exact_loss(case, seed):
    flat, dims, hv, buf, ret, adv, idx = _loss_inputs(case, seed)
    name, rows, E = case["workload"], case["rows"], buf["action"].shape[1]
    acts, A = W.mlp_acts(name), dims[-1] - (1 if hv else 0)
    p = flat.double().requires_grad_(True)
    layers = _split(p, dims)
    idx = torch.arange(rows, device="cuda") if idx is None else idx
    total, pol_s, val_s, ent_s, clip_s = 0.0, 0.0, 0.0, 0.0, 0.0
    c_value = LOSS["c_value"] if hv else 0.0
    for i in range(0, rows, 32768):
        r = idx[i:i + 32768]
        t, e = r // E, r % E
        Z = _mlp(buf["obs"][t, :, e].double(), layers, acts)
        lp = torch.log_softmax(Z[:, :A], dim=1)
        la = lp.gather(1, buf["action"][t, e].long()[:, None])[:, 0]
        a = adv[t, e].double()
        if case["algo"] == "ppo":
            rho = torch.exp(la - buf["logp"][t, e].double())
            lo, hi = 1.0 - float(np.float32(LOSS["clip_eps"])), 1.0 + float(np.float32(LOSS["clip_eps"]))
            pol = -torch.minimum(rho * a, rho.clamp(lo, hi) * a).sum()
            clip_s += float((((rho - 1.0).abs() > float(np.float32(LOSS["clip_eps"]))).sum()).item())
        else:
            pol = -(a * la).sum()
        ent = -(lp.exp() * lp).sum()
        val = ((Z[:, A] - ret[t, e].double()) ** 2).sum() if hv else torch.zeros((), device="cuda",
                                                                             dtype=torch.float64)
        L = (pol + c_value * val - LOSS["c_entropy"] * ent) / rows
        L.backward()
        total += float(L.item())
        pol_s += float(pol.item()) / rows
        val_s += float(val.item()) / rows
        ent_s += float(ent.item()) / rows
    # the clip fraction (last statistic) counts rows at a threshold and is left to the tolerance
    stats = torch.tensor([total, pol_s, val_s, ent_s, clip_s / rows], dtype=torch.float64)
    return dict(grad=p.grad, stats=stats)


def exact(case, seed):
    kind, seed = case["kind"], int(seed) & 0x7FFFFFFF
    if kind == "returns":
        s = prepare(case, seed)
        T = case["T"]
        rew, nd = s["rew"].double(), 1.0 - s["done"].double()
        g32 = float(np.float32(0.99))
        run_, last = torch.zeros_like(s["last"]).double(), s["last"].double()
        ret, adv = torch.empty_like(rew), torch.empty_like(rew)
        if s["val"] is not None:
            lam, val = float(np.float32(case["lam"])), s["val"].double()
            nxt = last
            for t in range(T - 1, -1, -1):
                delta = rew[t] + g32 * nd[t] * nxt - val[t]
                run_ = delta + g32 * lam * nd[t] * run_
                adv[t], ret[t], nxt = run_, run_ + val[t], val[t]
            return dict(ret=ret, adv=adv)
        run_ = last
        for t in range(T - 1, -1, -1):
            run_ = rew[t] + g32 * nd[t] * run_
            ret[t] = run_
        mean = ret.mean()
        return dict(ret=ret, adv=ret - mean, mean=mean.reshape(1))
    if kind == "forward":
        flat, dims, hv = _weights(case["workload"], seed)
        A = dims[-1] - (1 if hv else 0)
        Z = _mlp(_obs((dims[0], case["n"]), dims[0], _gen(seed)).double().T,
                 _split(flat.double(), dims), W.mlp_acts(case["workload"]))
        return dict(logits=Z[:, :A].T.contiguous(), value=Z[:, A].contiguous() if hv else None,
                    action=None, logp=None)
    if kind == "loss":
        return _exact_loss(case, seed)
    if kind == "adam":
        p, g, m, v, mask = (None if x is None else x.double() for x in _adam_inputs(case, seed))
        keep = torch.ones_like(p, dtype=torch.bool) if mask is None else mask > 0
        b1, b2, lr, eps = (float(np.float32(x)) for x in (0.9, 0.999, 3e-4, 1e-8))
        norm, t = float(torch.linalg.norm(g[keep]).item()), case["state"] + 1
        clip = min(1.0, case["clip"] / norm) if case["clip"] > 0 else 1.0
        m2 = b1 * m + (1 - b1) * clip * g
        v2 = b2 * v + (1 - b2) * (clip * g) ** 2
        step = (lr / (1 - b1 ** t)) * m2 / (torch.sqrt(v2) / math.sqrt(1 - b2 ** t) + eps)
        return dict(params=torch.where(keep, p - step, p), m=torch.where(keep, m2, m),
                    v=torch.where(keep, v2, v))
    # simulations are specified step by step in whole microseconds and fp32: no 64-bit value
    return None
