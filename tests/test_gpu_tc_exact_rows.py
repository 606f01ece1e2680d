"""Batched tensor-core searches whose certificate fails (few consumers sharing
the FP32 tiles, then cache rows of exact keys): many equal keys, few consumers,
short lists, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2401_07378_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def dev(a, dt):
    return torch.from_numpy(np.ascontiguousarray(a)).to(device="cuda", dtype=dt)


@pytest.mark.parametrize("precision,rk", [("fp8", 0), ("fp8", 1), ("fp16", 3), ("bf16", 0)])
@pytest.mark.parametrize("d", [9, 48])
def test_uncertified_searches(d, precision, rk):
    from paper_2401_07378_gb300 import nnsemd
    ctx = nnsemd.Context(0)
    pairs = []
    for k, (m, n) in enumerate([(1500, 1), (900, 5), (2048, 64), (600, 65), (700, 129), (530, 600), (1, 700), (6, 900)]):
        p = wl.uniform_pair(m, n, d, 5 * d + k, "dirichlet")
        if k % 2 == 0:  # far more equal keys than a list holds
            p.x[:], p.y[:] = np.round(p.x), np.round(p.y)
        else:           # keys closer together than the operand precision tells apart
            p.x[:], p.y[:] = 1.0 + 1e-3 * p.x, 1.0 + 1e-3 * p.y
        if k % 3 == 0 and m > 5:
            p.a[::5] = 0.0
        pairs.append(p)
    ref = [oracle.solve_pair(p, "sql2") for p in pairs]
    b = wl.Batch.pack(pairs)
    costs, stats = ctx.solve_batched(dev(b.x, torch.float32), dev(b.a, torch.float64), b.x_off, dev(b.y, torch.float32),
                                     dev(b.b, torch.float64), b.y_off, metric="sql2", precision=precision, rerank_k=rk)
    assert costs.cpu().numpy().tolist() == [r.cost for r in ref]
    assert stats["rounds"] == sum(r.rounds for r in ref)
    assert stats["certified"] + stats["fallbacks"] == sum(int(r.n_t.sum()) for r in ref)
    ctx.close()
