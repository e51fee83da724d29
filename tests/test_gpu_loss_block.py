"""FP32 loss gradient over minibatches of one tile per SM: the block kernel's range and the sizes
beside it, against the fp64 oracle with the tolerances of the other FP32 paths."""
import numpy as np
import pytest

from test_gpu_rl import _check_grad, _loss_case, _simx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,algo,E,H,nmb,hidden", [
    ("c3", "ppo", 40, 256, 4864, None),         # 32 rows per SM: the fused kernel
    ("c3", "ppo", 40, 256, 4865, None),         # first of the range: 40-row tiles, the last ragged
    ("c3", "reinforce", 40, 256, 6081, None),   # 48 rows, the last tile one row
    ("c3", "ppo", 40, 256, 8512, None),         # last of the range: 56 rows on every SM
    ("c3", "ppo", 40, 256, 8513, None),         # past it: 64 rows on either kernel
    ("c3", "reinforce", 71, 101, None, 100),    # every row, widths off the tiles of 8
    ("c3s", "ppo", 32, 256, 8192, None),        # two-tower policy
])
def test_block_loss_gradient_matches_oracle(name, algo, E, H, nmb, hidden):
    g, s, g_ref, st, layers, n = _loss_case(_simx(), name, algo, E, H, nmb, "fp32", hidden)
    _check_grad(g, g_ref, layers)
    assert np.all(np.abs(s[:4] - st[:4]) <= 1e-5 * (np.abs(st[:4]) + 1.0))
    assert abs(s[4] - st[4]) <= 1.0 / n


@pytest.mark.parametrize("name,algo,E,H,nmb,hidden", [
    ("c2", "reinforce", 1, 1, None, None),      # one row
    ("c2", "ppo", 16, 64, 64, None),            # one full tile
    ("c2", "ppo", 16, 64, 65, None),
    ("c2", "reinforce", 40, 512, 19457, None),  # one block walks two tiles
    ("c2", "ppo", 16, 64, 333, 60),             # widths off the tiles
    ("c2", "ppo", 16, 64, 333, 68),             # the weights no longer fit beside two blocks
    ("c1", "ppo", 64, 400, 20000, None),
])
def test_resident_weights_loss_gradient_matches_oracle(name, algo, E, H, nmb, hidden):
    """The fused kernel with every weight in shared memory, dZ over the activations."""
    g, s, g_ref, st, layers, n = _loss_case(_simx(), name, algo, E, H, nmb, "fp32", hidden)
    _check_grad(g, g_ref, layers)
    assert np.all(np.abs(s[:4] - st[:4]) <= 1e-5 * (np.abs(st[:4]) + 1.0))
    assert abs(s[4] - st[4]) <= 1.0 / n
