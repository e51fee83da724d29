"""What a call reports when a wait for a bulk copy of the policy's weights runs out.  The copies that
SIMX_WITHHOLD_COPIES names are never issued, so the bounded waits for them (about a second) end by
themselves and the kernels return: the batched forward writes NaN, the rollouts flag their envs."""
import pytest

from paper_2607_05272_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _simx():
    from paper_2607_05272_gb300 import build as B
    B.build()
    from paper_2607_05272_gb300 import simx
    return simx


def _policy(simx, name, hidden=None):
    dims, hv = W.mlp_dims(name)
    dims = [dims[0]] + (hidden or dims[1:-1]) + [dims[-1]]
    Ws, bs = W.mlp_weights(dims, 7, sigma=0.2)
    return simx.Policy([torch.from_numpy(w).cuda() for w in Ws], [torch.from_numpy(b).cuda() for b in bs], hv)


# one tile of columns per block; several, of which the last is concerned
@pytest.mark.parametrize("n", [100, 60000])
@pytest.mark.parametrize("mode", ["sample", "argmax"])
def test_forward_says_nan(n, mode, monkeypatch):
    simx = _simx()
    pol = _policy(simx, "c4")
    obs = torch.randn((28, n), device="cuda", generator=torch.Generator("cuda").manual_seed(n))

    def call():
        out = dict(logits=torch.zeros((48, n), device="cuda"), value=torch.zeros(n, device="cuda"),
                   action=torch.zeros(n, dtype=torch.uint8, device="cuda"), logp=torch.zeros(n, device="cuda"))
        simx.policy_forward(pol, obs, n, mode, 3, 4, **out)
        torch.cuda.synchronize()
        return out

    good = call()
    monkeypatch.setenv("SIMX_WITHHOLD_COPIES", "1")
    bad = call()
    monkeypatch.delenv("SIMX_WITHHOLD_COPIES")
    again = call()
    for k in good:
        assert torch.equal(good[k], again[k]), k
    void = torch.isnan(bad["value"])
    assert bool(void.all()) if n == 100 else 0 < int(void.sum()) < n
    assert bool(torch.isnan(bad["logits"][:, void]).all()) and bool(torch.isnan(bad["logp"][void]).all())
    assert int(bad["action"].max()) < 48
    for k in good:
        assert torch.equal(good[k][..., ~void], bad[k][..., ~void]), k


@pytest.mark.parametrize("name,E,hidden", [("c3", 300, None), ("c2", 2500, None), ("c2", 2500, [256, 200])],
                         ids=["route", "single-resident", "single-streamed"])
def test_rollout_flags_its_envs(name, E, hidden, monkeypatch):
    simx = _simx()
    pol = _policy(simx, name, hidden)
    sim = simx.Sim(W.CONFIGS[name](E))
    sim.reset(1)
    buf = simx.alloc_rollout(E, sim.D, 3, has_value=pol.has_value)
    monkeypatch.setenv("SIMX_WITHHOLD_COPIES", "1")
    sim.rollout("sample", 3, buf, pol)
    torch.cuda.synchronize()
    st, code = sim.last_status()
    assert st != 0 and code == 16   # SIMX_DEV_COPY_TIMEOUT
    assert int(buf["action"].max()) < pol.n_actions
    sim.close()


def test_loss_gradient_says_nan(monkeypatch):
    """The FP32 loss of one tile per SM: gradient and statistics, so that no optimiser step takes a
    gradient of unloaded weights for a finite one."""
    simx = _simx()
    pol = _policy(simx, "c3")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 32 * sms + 1   # the first size of the block kernel
    g = torch.Generator("cuda").manual_seed(2)
    buf = dict(obs=torch.randn((1, 13, n), device="cuda", generator=g),
               action=torch.randint(0, 16, (1, n), device="cuda", generator=g, dtype=torch.uint8),
               logp=torch.full((1, n), -2.7, device="cuda"))
    adv, ret = torch.randn((2, 1, n), device="cuda", generator=g)
    ws = torch.empty(simx.ppo_loss_grad_workspace_size(pol, n), dtype=torch.uint8, device="cuda")

    def call():
        grad, stats = torch.zeros(pol.n_params, device="cuda"), torch.zeros(5, device="cuda")
        simx.ppo_loss_grad(pol, buf, ret, adv, None, n, "ppo", 0.2, 0.5, 0.01, grad, stats, ws)
        torch.cuda.synchronize()
        return grad, stats

    good = call()
    monkeypatch.setenv("SIMX_WITHHOLD_COPIES", "1")
    grad, stats = call()
    monkeypatch.delenv("SIMX_WITHHOLD_COPIES")
    assert bool(torch.isnan(grad).all()) and bool(torch.isnan(stats[:4]).all())
    assert all(torch.equal(a, b) for a, b in zip(good, call())) and bool(torch.isfinite(good[0]).all())
