"""FP32 loss gradient over minibatches of one tile per SM: the block kernel's range and the sizes
beside it, against the fp64 oracle with the tolerances of the other FP32 paths.  The range follows
the SM count; each case asserts the kernel it means to cover."""
import numpy as np
import pytest

from paper_2607_05272_gb300 import workloads as W
from test_gpu_rl import _check_grad, _loss_case, _simx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _kernel(simx, name, hidden, n):
    dims, hv = W.mlp_dims(name)
    if hidden is not None:
        dims = [dims[0]] + [hidden] * (len(dims) - 2) + [dims[-1]]
    pol = simx.Policy([torch.zeros((b, a), device="cuda") for a, b in zip(dims[:-1], dims[1:])],
                      [torch.zeros(b, device="cuda") for b in dims[1:]], hv, W.mlp_acts(name))
    return simx.loss_kernel(pol, n)


def _check(simx, name, algo, E, H, nmb, hidden, kernel):
    assert _kernel(simx, name, hidden, nmb or E * H) == kernel
    g, s, g_ref, st, layers, n = _loss_case(simx, name, algo, E, H, nmb, "fp32", hidden)
    _check_grad(g, g_ref, layers)
    assert np.all(np.abs(s[:4] - st[:4]) <= 1e-5 * (np.abs(st[:4]) + 1.0))
    assert abs(s[4] - st[4]) <= 1.0 / n


# rows: per SM, and over that in all
@pytest.mark.parametrize("name,algo,per_sm,over,kernel", [
    ("c3", "ppo", 32, 0, "fused"),          # 32 rows per SM on either: the fused kernel
    ("c3", "ppo", 32, 1, "block"),          # first of the range: 40-row tiles, the last ragged
    ("c3", "reinforce", 40, 1, "block"),    # 48 rows, the last tile one row
    ("c3", "ppo", 56, 0, "block"),          # last of the range: 56 rows on every SM
    ("c3", "ppo", 56, 1, "fused"),          # past it: 64 rows on either
    ("c3s", "ppo", 50, 592, "block"),       # two-tower policy
])
def test_block_loss_gradient_matches_oracle(name, algo, per_sm, over, kernel):
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + over
    _check(_simx(), name, algo, -(-n // 256), 256, n, None, kernel)


@pytest.mark.parametrize("n,kernel", [(1, "block"), (8, "block"), (9, "fused")])
def test_block_loss_gradient_of_few_rows(n, kernel):
    _check(_simx(), "c3", "ppo", 4, 64, n, None, kernel)


def test_block_loss_gradient_of_odd_widths():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    _check(_simx(), "c3", "reinforce", -(-47 * sms // 101), 101, None, 100, "block")   # every row


@pytest.mark.parametrize("name,algo,E,H,nmb,hidden,kernel", [
    ("c2", "reinforce", 1, 1, None, None, "fused"),   # one row
    ("c2", "ppo", 4, 2, 8, None, "fused"),
    ("c2", "ppo", 16, 64, 64, None, "fused"),         # one full tile
    ("c2", "ppo", 16, 64, 65, None, "fused"),
    ("c2", "reinforce", 40, 512, 19457, None, "fused"),  # one block walks two tiles
    ("c2", "ppo", 16, 64, 333, 60, "fused"),          # widths off the tiles
    ("c2", "ppo", 16, 64, 333, 68, "fused"),          # the weights no longer fit beside two blocks
    ("c1", "ppo", 64, 400, 20000, None, "fused"),
])
def test_resident_weights_loss_gradient_matches_oracle(name, algo, E, H, nmb, hidden, kernel):
    """The fused kernel with every weight in shared memory, dZ over the activations."""
    _check(_simx(), name, algo, E, H, nmb, hidden, kernel)
