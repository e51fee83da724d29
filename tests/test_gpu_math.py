"""The branch-free tanh and exp of the block forward (Sec. 4.2) have the bits of the library's defining
ones on every input: every rollout, forward and FP32 loss evaluates them, and the tanh replaces an
IEEE division by an estimate, a Newton step and the exact remainder, whose rounding the reachable
activations of the other tests would only sample.  All 2^32 patterns (exp: those not above zero)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", ["tanh", "exp"])
def test_branch_free_form_has_the_same_bits(which):
    from paper_2607_05272_gb300 import build as B
    B.build()
    from paper_2607_05272_gb300 import simx
    count = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    simx.math_check(which, count)
    assert int(count) == 0
    with pytest.raises(KeyError):
        simx.math_check("log", count)
