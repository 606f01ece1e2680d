"""One-CTA solves (d <= 8) with few consumers, a warp each, and the sizes around
where the chunked scan takes over, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2401_07378_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def dev(a, dt):
    return torch.from_numpy(np.ascontiguousarray(a)).to(device="cuda", dtype=dt)


@pytest.mark.parametrize("metric", ["l2", "l1"])
@pytest.mark.parametrize("d", [1, 3, 8])
def test_few_consumers(d, metric):
    from paper_2401_07378_gb300 import nnsemd
    ctx = nnsemd.Context(0)
    pairs = []
    for k, (m, n) in enumerate([(1000, 1), (900, 2), (1024, 31), (700, 32), (1000, 33), (512, 1), (400, 7), (511, 8),
                                (90, 9), (31, 5), (1500, 3), (2000, 16), (1700, 17), (600, 20)]):
        p = wl.uniform_pair(m, n, d, 9 * d + k, "dirichlet")
        if k % 2:
            p.x[:], p.y[:] = np.round(4 * p.x), np.round(4 * p.y)  # equal keys
        if k == 13:
            p.y[::2] *= 1e25  # keys all infinite
        pairs.append(p)
    ref = [oracle.solve_pair(p, metric) for p in pairs]
    for p, r in zip(pairs, ref):
        got = ctx.solve(dev(p.x, torch.float32), dev(p.a, torch.float64), dev(p.y, torch.float32),
                        dev(p.b, torch.float64), metric=metric)
        assert got.cost == r.cost and got.stats["rounds"] == r.rounds
    b = wl.Batch.pack(pairs)
    costs, _ = ctx.solve_batched(dev(b.x, torch.float32), dev(b.a, torch.float64), b.x_off, dev(b.y, torch.float32),
                                 dev(b.b, torch.float64), b.y_off, metric=metric)
    assert costs.cpu().numpy().tolist() == [r.cost for r in ref]
    ctx.close()
