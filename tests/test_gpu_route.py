"""The router's rollout with one simulator thread per env (Sec. 3.1, 4.1, 4.2) at the sizes
where its plan changes: 8, 16 and 32 envs per 256-thread block, 16 per 128-thread block, ragged
last blocks, one to eight servers, one request type, trace replay and diurnal arrivals, policies
whose widths are no multiple of its register tiles, with GELU and identity layers.

Every result is specified to the bit, so each rollout must equal the lane-group kernel's
(SIMX_STAGE=0) on every env, and the oracle's on sampled envs.
"""
import numpy as np
import pytest

import oracle
from paper_2607_05272_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _router(K, T, E):
    c = W.c3(E)
    c.update(n_servers=K, n_types=T, obs_dim=3 * K + 1, episode_len=7)
    if T == 1:
        c.update(type0_thr=W.TWO24)
    return c


def _dims(cfg, hidden):
    return [cfg["obs_dim"]] + hidden + [cfg["n_servers"] * cfg["n_bsizes"] + 1]


# name, configuration, hidden widths, activations, mode, steps
CASES = [
    ("one-env", W.c3(1), [128, 128], None, "sample", 40),
    ("8-envs-per-block-ragged", W.c3(1001), [128, 128], None, "sample", 40),
    ("16-envs-per-block-ragged", W.c4(2131), [256, 256], None, "sample", 24),
    ("32-envs-per-block-ragged", W.c3(4999), [128, 128], None, "argmax", 24),
    ("128-threads-ragged", W.c3(14701), [128, 128], None, "sample", 16),
    ("wide-8-envs", W.c4(130), [256, 256], None, "argmax", 24),
    ("odd-widths-gelu", W.c4(517), [100, 130, 61], ["gelu", "identity", "tanh"], "sample", 24),
    ("three-servers-one-type", _router(3, 1, 700), [64, 33], None, "sample", 40),
    ("one-server", _router(1, 2, 300), [40], None, "sample", 40),
    ("five-servers-deep", _router(5, 2, 2500), [31, 64, 17, 128], ["tanh"] * 4, "sample", 24),
    ("grid-128-threads", W.c3(14701), [128, 128], None, "sample", 16),
    ("grid-wide", W.c4(2131), [256, 255], ["tanh", "gelu"], "argmax", 16),
    ("trace", W.c3t(900), [128, 128], None, "sample", 40),
]


@pytest.mark.parametrize("cfg,hidden,acts,mode,H", [c[1:] for c in CASES], ids=[c[0] for c in CASES])
def test_route_rollout(cfg, hidden, acts, mode, H, request, monkeypatch):
    from paper_2607_05272_gb300 import build as B
    B.build()
    from paper_2607_05272_gb300 import simx
    monkeypatch.delenv("SIMX_LANES", raising=False)
    monkeypatch.delenv("SIMX_THREADS", raising=False)
    E, dims = cfg["n_envs"], _dims(cfg, hidden)
    Ws, bs = W.mlp_weights(dims, 11, sigma=0.2)
    bs = [b + np.float32(0.05) * np.arange(len(b), dtype=np.float32) / len(b) for b in bs]
    gx = None
    if "grid" in request.node.callspec.id:
        gx, ew = [4] + [7] * len(hidden), [6] * (len(hidden) + 1)
        Ws, bs = W.grid_weights(dims, 5, gx, ew)
    got = []
    for stage in ("1", "0"):
        monkeypatch.setenv("SIMX_STAGE", stage)
        pol = simx.Policy([torch.from_numpy(w).cuda() for w in Ws],
                          [torch.from_numpy(b).cuda() for b in bs], True, acts, grid=gx)
        sim = simx.Sim(cfg)
        sim.reset(0xA11)
        shape = sim.launch_shape(mode, pol)
        assert shape["staged"] == (stage == "1") and shape["kernel"] == "fused"
        kernel, weights = sim.rollout_kernel(mode, pol)
        assert (kernel, weights) == ("route", "streamed") if stage == "1" else kernel == "lanes"
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
    envs = sorted({0, E // 2, E - 1} | {e for e in (31, 32, 127) if e < E})
    ref = oracle.rollout(cfg, (Ws, bs, True, acts or ["tanh"] * len(hidden), gx), 0xA11,
                         {"sample": 0, "argmax": 1}[mode], envs, H)
    sel = torch.tensor(envs, device="cuda")
    col = {k: v.index_select(v.dim() - 1, sel).cpu().numpy() for k, v in a.items()}
    assert np.array_equal(col["action"], ref["action"].astype(np.uint8))
    assert np.array_equal(col["trace"], ref["trace"])
    for k in ("obs", "reward", "logp", "value"):
        assert np.array_equal(col[k].view(np.uint32), ref[k].view(np.uint32)), k
