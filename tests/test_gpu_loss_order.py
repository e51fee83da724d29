"""The order of the FP32 loss gradient's sums (Sec. 4.3): dW sums a tile's rows in order, one fma a
row.  A training run amplifies it (a last bit of an update changes a sampled action some iterations
later), so the order is part of what the entry point returns.

One layer without hidden units, zero weights and a power of two of actions: every probability is
1 / A exactly, and with small whole advantages dZ is exact.  Each product has at most 30 bits then
and each sum of the chain is exact in fp64 before its one rounding to fp32, so the chain can be
followed on the host to the bit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# observation width, actions, rows: one tile of 64 rows with resident weights, one of 32 rows
@pytest.mark.parametrize("D,A,n", [(64, 64, 64), (64, 128, 32)])
def test_weight_gradient_sums_rows_in_order(D, A, n):
    from paper_2607_05272_gb300 import build as B
    B.build()
    from paper_2607_05272_gb300 import simx
    rng = np.random.default_rng(D + n)
    X = (rng.integers(-32767, 32768, (D, n)) / 4096.0).astype(np.float32)
    adv = rng.integers(1, 200, n).astype(np.float32)
    action = rng.integers(0, A, n).astype(np.uint8)
    pol = simx.Policy([torch.zeros((A, D), device="cuda")], [torch.zeros(A, device="cuda")], False)
    buf = dict(obs=torch.from_numpy(X[None]).cuda(), action=torch.from_numpy(action[None]).cuda(),
               logp=torch.zeros((1, n), device="cuda"))
    grad, stats = torch.empty(pol.n_params, device="cuda"), torch.empty(5, device="cuda")
    ws = torch.empty(simx.ppo_loss_grad_workspace_size(pol, n), dtype=torch.uint8, device="cuda")
    simx.ppo_loss_grad(pol, buf, None, torch.from_numpy(adv[None]).cuda(), None, n, "reinforce", 0.2,
                       0.0, 0.0, grad, stats, ws)
    dz = -adv * ((np.arange(A)[:, None] == action) - 1.0 / A) / n   # exact
    assert np.array_equal(dz, dz.astype(np.float32))
    acc = np.zeros((A, D), np.float32)
    for r in range(n):
        acc = (acc.astype(np.float64) + np.outer(dz[:, r], X[:, r].astype(np.float64))).astype(np.float32)
    got = grad.cpu().numpy()[:A * D].reshape(A, D)
    assert np.array_equal(got, acc)
    # the inputs tell orders apart: even and odd rows summed on their own give other bits
    half = [np.zeros((A, D), np.float32) for _ in range(2)]
    for r in range(n):
        half[r % 2] = (half[r % 2].astype(np.float64) +
                       np.outer(dz[:, r], X[:, r].astype(np.float64))).astype(np.float32)
    assert not np.array_equal(half[0] + half[1], acc)
