"""Returns and GAE (Sec. 4.3) at the edges of the kernel that reads each input once (GAE from 16,384
envs): horizons of one step, of one chunk and around it, of one window and around it, several
windows, env counts off the block's 32; returns past its line of 24 Mi samples; and at the same
horizons the kernel of fewer envs; and the mean baseline at its block edges, on sums that overflow
fp32 and on values that cancel."""
import math

import numpy as np
import pytest

from oracle import rl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _simx():
    from paper_2607_05272_gb300 import build as B
    B.build()
    from paper_2607_05272_gb300 import simx
    return simx


@pytest.mark.parametrize("T,E", [(1, 1), (7, 33), (8, 32), (9, 31), (63, 100), (255, 17), (256, 5),
                                 (257, 5), (300, 16384), (64, 16391), (129, 40001),
                                 (1, 16384), (8, 16385), (9, 16390), (65, 16384), (513, 50001)])
@pytest.mark.parametrize("gae", [False, True], ids=["reinforce", "gae"])
def test_returns(T, E, gae):
    simx = _simx()
    rng = np.random.default_rng(T * 7 + E)
    r = (rng.standard_normal((T, E)) * 2.0 - 0.5).astype(np.float32)
    v = rng.standard_normal((T, E)).astype(np.float32)
    d = (rng.random((T, E)) < 0.05).astype(np.uint8)
    last = rng.standard_normal(E).astype(np.float32)
    dev = lambda x: torch.from_numpy(x).cuda()
    ret, adv = torch.empty((T, E), device="cuda"), torch.empty((T, E), device="cuda")
    if gae:
        simx.compute_returns_gae(dev(r), dev(d), 0.99, 0.95, ret, adv=adv, val=dev(v), last_val=dev(last))
        A, R = rl.gae(r, v, d, 0.99, 0.95, last)
        vn = np.vstack([v[1:], last[None]]).astype(np.float64)
        scale = rl.returns(np.abs(r) + 0.99 * np.abs(vn) + np.abs(v), d, 0.99 * 0.95)
        pairs = [(adv, A, scale), (ret, R, scale + np.abs(v))]
    else:
        simx.compute_returns_gae(dev(r), dev(d), 0.99, -1.0, ret, adv=adv, last_val=dev(last))
        pairs = [(ret, rl.returns(r, d, 0.99, last), rl.returns(np.abs(r), d, 0.99, np.abs(last)))]
        assert torch.equal(ret, adv)
    for got, ref, s in pairs:
        # the recurrence's rounding: a few units of 2^-24 of the sum of the absolute terms per step
        # of the effective horizon (1 / (1 - 0.99) steps)
        assert np.all(np.abs(got.cpu().numpy() - ref) <= 1e-5 * (np.abs(ref) + s) + 1e-30)


@pytest.mark.parametrize("n", [1, 255, 2048, 2049, 1000003])
@pytest.mark.parametrize("kind", ["plain", "cancel", "huge", "inf"])
def test_baseline(n, kind):
    simx = _simx()
    rng = np.random.default_rng(n)
    x = rng.standard_normal(n).astype(np.float32)
    if kind == "cancel":
        x = (x + np.where(np.arange(n) % 2 == 0, 1e6, -1e6)).astype(np.float32)
    elif kind == "huge":
        x = np.full(n, 3e38, np.float32)
    elif kind == "inf":
        x[n // 2] = np.inf
    adv, mean = torch.empty(n, device="cuda"), torch.empty(1, device="cuda")
    ws = torch.empty(simx.returns_baseline_workspace_size(n), dtype=torch.uint8, device="cuda")
    simx.returns_baseline(torch.from_numpy(x).cuda(), adv, mean, ws)
    m = x.astype(np.float64).mean()
    got, gm = adv.cpu().numpy(), mean.item()
    if kind == "inf":
        assert gm == np.inf
        with np.errstate(invalid="ignore"):
            assert np.array_equal(got, (x.astype(np.float64) - np.inf).astype(np.float32), equal_nan=True)
        return
    # the mean to fp64 rounding of n additions, the centred value rounded once more
    tol = 1e-14 * np.abs(x).astype(np.float64).mean() * max(1.0, np.log2(n + 1))
    assert abs(gm - m) <= 6e-8 * abs(m) + tol
    ref = x.astype(np.float64) - m
    assert np.all(np.abs(got - ref) <= 1.2e-7 * np.abs(ref) + tol)


def test_baseline_sums_in_64_bits():
    """Every element of a thread's sum is a whole multiple of 2^-23 and every partial sum below 2^28,
    so that fp64 holds each exactly and the mean is the exact one, rounded once; 2^25 against values
    of about 2 is more than fp32 pairs keep."""
    simx = _simx()
    M, stride = 256, 1024 * 256   # elements per thread, threads
    v = np.random.default_rng(2).uniform(1.5, 1.99, (M - 8) // 2).astype(np.float32)
    back = np.random.default_rng(3).permutation(v) + np.float32(2.0 ** -12)
    big = np.full(4, 2.0 ** 25, np.float32)
    seq = np.concatenate([big, v, -back, -big]).astype(np.float32)
    n = M * stride
    assert simx.returns_baseline_workspace_size(n) == 1024 * 8
    x = torch.from_numpy(seq).cuda().repeat_interleave(stride)
    adv, mean = torch.empty(n, device="cuda"), torch.empty(1, device="cuda")
    ws = torch.empty(1024 * 8, dtype=torch.uint8, device="cuda")
    simx.returns_baseline(x, adv, mean, ws)
    m = math.fsum(seq.tolist()) / M
    assert m != 0.0 and mean.item() == np.float32(m)
    want = torch.from_numpy((seq.astype(np.float64) - m).astype(np.float32)).cuda()
    assert torch.equal(adv.view(M, stride), want[:, None].expand(M, stride))
