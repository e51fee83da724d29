"""The order in which returns and GAE (Sec. 4.3) of fewer than 16,384 envs (and returns up to 24 Mi
samples) are composed: S chunks of ceil(T / S) steps, S doubled while chunks of 16 steps or more
remain (and threads are wanted), each chunk's affine map in fp32 from the right, the maps
chained, the chunks replayed.  A training run amplifies a last bit of an advantage, so the order is
part of what the entry point returns; it is followed here on the host (every multiplication and
addition rounds once: none is contracted)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

f32 = np.float32


def _composed(r, v, d, last, gamma, lam, S):
    T, E = r.shape
    gae = v is not None
    cm = f32(gamma) * f32(lam) if gae else f32(gamma)
    L = -(-T // S)
    delta = r.copy()
    if gae:
        vn = np.vstack([v[1:], last[None]])
        delta = r + f32(gamma) * (1 - d).astype(f32) * vn - v
    c = cm * (1 - d).astype(f32)
    carry = np.zeros(E, f32) if gae else last.copy()
    x = np.empty((T, E), f32)
    for j in range(S - 1, -1, -1):
        t0, t1 = j * L, min(j * L + L, T)
        a, b, y = np.ones(E, f32), np.zeros(E, f32), carry
        for t in range(t1 - 1, t0 - 1, -1):
            b = delta[t] + c[t] * b
            a = c[t] * a
            y = delta[t] + c[t] * y
            x[t] = y
        carry = b + a * carry
    return x


@pytest.mark.parametrize("T,E,S", [
    (64, 4096, 4), (256, 100, 16), (31, 33, 1), (100, 16383, 4), (1, 1, 1), (33, 5, 2),
    (255, 16380, 8), (511, 3, 16), (512, 40, 32), (513, 9, 32)])
@pytest.mark.parametrize("gae", [False, True], ids=["reinforce", "gae"])
def test_chunks_are_composed_in_order(T, E, S, gae):
    from paper_2607_05272_gb300 import build as B
    B.build()
    from paper_2607_05272_gb300 import simx
    rng = np.random.default_rng(T * 5 + E)
    r = (rng.standard_normal((T, E)) * 2.0 - 0.5).astype(f32)
    v = (10.0 * rng.standard_normal((T, E))).astype(f32)
    d = (rng.random((T, E)) < 0.05).astype(np.uint8)
    last = rng.standard_normal(E).astype(f32)
    dev = lambda x: torch.from_numpy(x).cuda()
    ret, adv = torch.empty((T, E), device="cuda"), torch.empty((T, E), device="cuda")
    if gae:
        simx.compute_returns_gae(dev(r), dev(d), 0.99, 0.95, ret, adv=adv, val=dev(v), last_val=dev(last))
        A = _composed(r, v, d, last, 0.99, 0.95, S)
        assert np.array_equal(adv.cpu().numpy(), A) and np.array_equal(ret.cpu().numpy(), A + v)
    else:
        simx.compute_returns_gae(dev(r), dev(d), 0.99, -1.0, ret, adv=adv, last_val=dev(last))
        assert np.array_equal(ret.cpu().numpy(), _composed(r, None, d, last, 0.99, 0.0, S))
        assert torch.equal(ret, adv)
