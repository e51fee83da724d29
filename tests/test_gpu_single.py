"""The single server's rollout with a thread per queue and a warp per env's arrivals (Sec. 3.1, 4.1,
4.2) at the sizes where its plan changes: 16 and 32 envs per block, ragged last blocks, rings in
shared memory and (short horizons) in global memory, policies resident in shared memory and
streamed, the Wait layout, per-request costs, trace replay, the square wave, full queues, windows
of candidates drawn many times over in one decision; and the lane-group kernel beside it at 32
lanes per env, whose chunk of candidates outlives the decision.

Every result is specified to the bit: the oracle's on sampled envs, and where both kernels take a
configuration (SIMX_STAGE=0) the same on every env."""
import numpy as np
import pytest

import oracle
from paper_2607_05272_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _with(cfg, **kw):
    cfg.update(kw)
    return cfg


# name, configuration, hidden widths, activations, mode, steps, by the new kernel
CASES = [
    ("lanes-32", W.c2(40), [64, 64], None, "sample", 60, False),
    ("lanes-32-wait", W.c1w(7), [32], None, "sample", 60, False),
    ("16-envs-ragged", W.c2(2451), [64, 64], None, "sample", 40, True),
    ("16-envs-global-rings", W.c2(2451), [64, 64], None, "argmax", 9, True),
    ("32-envs-ragged", W.c2(9777), [64, 64], None, "sample", 24, True),
    ("paper-net", W.c1p(2600), [4, 4, 4, 128], ["identity", "identity", "identity", "gelu"], "sample", 30, True),
    ("wide-streamed", W.c2w(2500), [256, 200], ["tanh", "gelu"], "sample", 24, True),
    ("costs", W.mm1(900.0, 2100.0, 2500), [40, 64], None, "sample", 40, True),
    ("trace", W.c2t(2500), [64, 64], None, "sample", 40, True),
    ("square-wave", W.burst(2500), [32, 200], None, "sample", 40, True),
    ("small-queue-overload", _with(W.c2(2500), queue_cap=4), [64, 64], None, "sample", 24, True),
    ("grid", W.c2(2500), [64, 64], None, "sample", 40, True),
    ("grid-gelu", W.c1p(2600), [4, 4, 4, 128], ["identity", "identity", "identity", "gelu"], "argmax", 30, True),
    ("long-batches", _with(W.c2(2500), alpha_us=[400000, 900000]), [64, 64], None, "sample", 6, True),
]


@pytest.mark.parametrize("cfg,hidden,acts,mode,H,new", [c[1:] for c in CASES], ids=[c[0] for c in CASES])
def test_single_rollout(cfg, hidden, acts, mode, H, new, request, monkeypatch):
    from paper_2607_05272_gb300 import build as B
    B.build()
    from paper_2607_05272_gb300 import simx
    for k in ("SIMX_LANES", "SIMX_THREADS"):
        monkeypatch.delenv(k, raising=False)
    E = cfg["n_envs"]
    n_act = cfg["n_types"] * cfg["n_bsizes"] + (1 if cfg["action_layout"] == 1 else 0)
    dims = [cfg["obs_dim"]] + hidden + [n_act + 1]
    Ws, bs = W.mlp_weights(dims, 5, sigma=0.3)
    gx = None
    if "grid" in request.node.callspec.id:
        gx, ew = [4] + [7] * len(hidden), [6] * (len(hidden) + 1)
        Ws, bs = W.grid_weights(dims, 5, gx, ew)
    got = []
    for stage in ("", "0"):
        monkeypatch.setenv("SIMX_STAGE", stage)
        pol = simx.Policy([torch.from_numpy(w).cuda() for w in Ws],
                          [torch.from_numpy(b).cuda() for b in bs], True, acts, grid=gx)
        sim = simx.Sim(cfg)
        sim.reset(0xB22)
        assert sim.launch_shape(mode, pol)["staged"] == (new and stage == "")
        kernel, weights = sim.rollout_kernel(mode, pol)
        assert kernel == ("single" if new and stage == "" else "lanes")
        if kernel == "single":
            assert weights == ("streamed" if "streamed" in request.node.callspec.id else "resident")
        buf = simx.alloc_rollout(E, sim.D, H, has_value=True, trace=True)
        sim.rollout(mode, H, buf, pol)
        nxt = torch.empty((sim.D, E), device="cuda")
        sim.step(mode, pol, obs=nxt)
        torch.cuda.synchronize()
        assert sim.last_status() == (0, 0)
        got.append((buf, nxt, sim.save()))
        sim.close()
    (a, na, sa), (b, nb, sb) = got
    for k in a:
        assert torch.equal(a[k], b[k]), k
    assert torch.equal(na, nb) and np.array_equal(sa, sb)
    envs = sorted({0, E // 2, E - 1} | {e for e in (15, 16, 31, 33) if e < E})
    ref = oracle.rollout(cfg, (Ws, bs, True, acts or ["tanh"] * len(hidden), gx), 0xB22,
                         {"sample": 0, "argmax": 1}[mode], envs, H)
    sel = torch.tensor(envs, device="cuda")
    col = {k: v.index_select(v.dim() - 1, sel).cpu().numpy() for k, v in a.items()}
    assert np.array_equal(col["action"], ref["action"].astype(np.uint8))
    assert np.array_equal(col["trace"], ref["trace"])
    for k in ("obs", "reward", "logp", "value"):
        assert np.array_equal(col[k].view(np.uint32), ref[k].view(np.uint32)), k


@pytest.mark.parametrize("gap,H", [((1 << 27) + 7, 12), (1 << 28, 5)])
@pytest.mark.parametrize("name,E", [("c2t", 2500), ("c2t", 40), ("c3t", 300)])
@pytest.mark.parametrize("stage", ["", "0"], ids=["default", "lanes"])
def test_long_gaps(name, E, gap, H, stage, monkeypatch):
    """A trace whose gaps add up past 32 bits within one group of candidates: their times end at the
    limit, which no decision here reaches, and none starts over."""
    from paper_2607_05272_gb300 import build as B
    B.build()
    from paper_2607_05272_gb300 import simx
    for k in ("SIMX_LANES", "SIMX_THREADS"):
        monkeypatch.delenv(k, raising=False)
    monkeypatch.setenv("SIMX_STAGE", stage)
    cfg = W.CONFIGS[name](E)
    cfg["trace"] = (np.full(64, gap, np.uint32), None, None)
    dims, hv = W.mlp_dims(name)
    Ws, bs = W.policy_weights(name, dims, 7)
    acts = W.mlp_acts(name)
    pol = simx.Policy([torch.from_numpy(w).cuda() for w in Ws], [torch.from_numpy(b).cuda() for b in bs],
                      hv, acts)
    sim = simx.Sim(cfg)
    sim.reset(0xB23)
    buf = simx.alloc_rollout(E, sim.D, H, has_value=hv, trace=True)
    sim.rollout("sample", H, buf, pol)
    torch.cuda.synchronize()
    envs = sorted({0, 7, E // 2, E - 1})
    sel = torch.tensor(envs, device="cuda")
    ref = oracle.rollout(cfg, (Ws, bs, hv, acts), 0xB23, 0, envs, H)
    col = {k: v.index_select(v.dim() - 1, sel).cpu().numpy() for k, v in buf.items()}
    assert np.array_equal(col["action"], ref["action"].astype(np.uint8))
    assert np.array_equal(col["trace"], ref["trace"])
    for k in ("obs", "reward", "logp"):
        assert np.array_equal(col[k].view(np.uint32), ref[k].view(np.uint32)), k
    assert np.array_equal(sim.save()[envs], ref["state"])
    assert sim.last_status() == (0, 0)
    sim.close()
