"""The batched policy forward (Sec. 4.2) at the sizes where its plan changes: 8, 16, 32 and 64
columns per block, ragged last blocks, several tiles per block, widths that are no multiple of
the register tiles, every activation, and an output layer too wide for the tiles (the lane-group
kernel).  Specified to the bit: every output must equal the oracle's on sampled columns, and a
column's outputs must not depend on how many columns the call has."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# n columns, widths (last: actions + value row), activations
CASES = [
    (1, [13, 128, 128, 17], None),
    (1003, [28, 256, 256, 49], None),
    (2200, [16, 64, 64, 13], None),
    (4999, [28, 256, 100, 49], ["gelu", "tanh"]),
    (7301, [8, 4, 4, 4, 128, 34], ["identity", "identity", "identity", "gelu"]),
    (45001, [28, 256, 256, 49], None),
    (8000, [5, 61, 3], ["tanh"]),
    (7300, [12, 40, 251], None),
]


@pytest.mark.parametrize("n,dims,acts", CASES, ids=["%d-%s" % (c[0], "-".join(map(str, c[1]))) for c in CASES])
@pytest.mark.parametrize("mode", ["sample", "argmax"])
def test_policy_forward(n, dims, acts, mode):
    from paper_2607_05272_gb300 import build as B
    B.build()
    from paper_2607_05272_gb300 import simx
    rng = np.random.default_rng(n + len(dims))
    Ws = [(0.3 * rng.standard_normal((b, a))).astype(np.float32) for a, b in zip(dims[:-1], dims[1:])]
    bs = [(0.1 * rng.standard_normal(b)).astype(np.float32) for b in dims[1:]]
    obs = (rng.standard_normal((dims[0], n)) * np.exp(rng.uniform(-8, 4, (dims[0], n)))).astype(np.float32)
    pol = simx.Policy([torch.from_numpy(w).cuda() for w in Ws], [torch.from_numpy(b).cuda() for b in bs],
                      True, acts)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    block = 64 if n > 48 * sms else 32 if n > 32 * sms else 16 if n > 14 * sms else 8
    assert simx.forward_columns(pol, n) == (0 if dims[-1] == 251 else block)
    A = dims[-1] - 1
    ld = n + 5

    def call(n):
        x = torch.zeros((dims[0], ld), device="cuda")
        x[:, :n] = torch.from_numpy(obs[:, :n]).cuda()
        out = dict(logits=torch.zeros((A, ld), device="cuda"), value=torch.zeros(ld, device="cuda"),
                   action=torch.zeros(ld, dtype=torch.uint8, device="cuda"), logp=torch.zeros(ld, device="cuda"))
        simx.policy_forward(pol, x, n, mode, 77, 9, env_base=40, **out)
        torch.cuda.synchronize()
        return {k: v.cpu().numpy() for k, v in out.items()}

    got = call(n)
    assert all(np.all(v[..., n:] == 0) for v in got.values())  # nothing past the last column
    few = min(n, 37)
    part = call(few)
    for k in got:
        assert np.array_equal(got[k][..., :few], part[k][..., :few]), k
    cols = sorted({0, n // 2, n - 1} | {int(c) for c in rng.integers(0, n, 24)})
    for i in cols:
        lg, v, a, lp = oracle.policy((Ws, bs, True, acts or ["tanh"] * (len(dims) - 2)), obs[:, i],
                                     {"sample": 0, "argmax": 1}[mode], 77, 9, 40 + i)
        assert np.array_equal(got["logits"][:, i].view(np.uint32), lg.view(np.uint32))
        assert got["value"][i] == v and got["action"][i] == a and got["logp"][i] == lp


def test_host_threads_with_plans_of_different_sizes():
    """policy_forward_ws shares no state between calls: two host threads whose launches of one kernel
    ask for different amounts of shared memory, on streams and workspaces of their own."""
    import threading
    from paper_2607_05272_gb300 import build as B
    B.build()
    from paper_2607_05272_gb300 import simx
    rng = np.random.default_rng(5)

    def make(dims, n):
        Ws = [torch.from_numpy((0.3 * rng.standard_normal((b, a))).astype(np.float32)).cuda()
              for a, b in zip(dims[:-1], dims[1:])]
        pol = simx.Policy(Ws, [torch.zeros(b, device="cuda") for b in dims[1:]], True)
        return dict(pol=pol, obs=torch.randn((dims[0], n), device="cuda"), n=n,
                    ws=torch.empty(simx.policy_forward_workspace_size(pol), dtype=torch.uint8, device="cuda"),
                    logits=torch.empty((dims[-1] - 1, n), device="cuda"), stream=torch.cuda.Stream())

    def call(s):
        simx.policy_forward(s["pol"], s["obs"], s["n"], "sample", 1, 2, logits=s["logits"],
                            workspace=s["ws"], stream=s["stream"].cuda_stream)

    # both take the kernel with 8 x 8 tiles, one with small and one with large activations and stages
    jobs = [make([8, 132, 5], 12000), make([28, 256, 256, 49], 12000)]
    want, errors = [], []
    for s in jobs:
        call(s)
        torch.cuda.synchronize()
        want.append(s["logits"].clone())
    start = threading.Barrier(2)

    def work(s):
        try:
            start.wait()
            for _ in range(1500):
                call(s)
        except Exception as e:   # noqa: BLE001 (reported below)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(s,)) for s in jobs]
    torch.cuda.synchronize()
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for s, w in zip(jobs, want):
        assert torch.equal(s["logits"], w)
