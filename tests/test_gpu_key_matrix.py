"""The packed 64 x 64 x 32 distance tiles (d > 8, FP32) and the batched
solvers' key matrices, at the edges of tiles, vectors and capacities, against
the oracle: costs and rounds bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2401_07378_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2401_07378_gb300 import nnsemd
    c = nnsemd.Context(0)
    yield c
    c.close()


def dev(a, dt):
    return torch.from_numpy(np.ascontiguousarray(a)).to(device="cuda", dtype=dt)


def shifted(a):
    """The same values at a base that is not 16-byte aligned."""
    buf = torch.empty(a.size + 1, dtype=torch.float32, device="cuda")
    buf[1:] = dev(a.ravel(), torch.float32)
    return buf[1:].view(a.shape)


SIZES = [(1, 1), (1, 70), (63, 65), (64, 64), (65, 129), (512, 512), (513, 30), (511, 513), (700, 1000)]


@pytest.mark.parametrize("metric", ["l2", "l1"])
@pytest.mark.parametrize("d", [9, 12, 31, 40, 64])
def test_batched_fp32_equals_oracle(ctx, d, metric):
    pairs = []
    for k, (m, n) in enumerate(SIZES):
        p = wl.uniform_pair(m, n, d, 100 * d + k, "dirichlet")
        if m > 4:
            p.a[::3] = 0.0  # zero weights take no part (rows of the matrix that are never active)
        if n > 4:
            p.y[: n // 2] = np.round(p.y[: n // 2] * 2) / 2  # equal keys
            p.x[: m // 2] = np.round(p.x[: m // 2] * 2) / 2
        pairs.append(p)
    batch = wl.Batch.pack(pairs)
    ref = [oracle.solve_pair(p, metric) for p in pairs]
    for make in (lambda v: dev(v, torch.float32), shifted):
        costs, stats = ctx.solve_batched(make(batch.x), dev(batch.a, torch.float64), batch.x_off, make(batch.y),
                                         dev(batch.b, torch.float64), batch.y_off, metric=metric)
        assert costs.cpu().numpy().tolist() == [r.cost for r in ref]
        assert stats["rounds"] == sum(r.rounds for r in ref)
        assert stats["pair_evals"] == sum(r.pair_evals for r in ref)


@pytest.mark.parametrize("m,n,d", [(2100, 65, 9), (129, 2300, 31), (2049, 2113, 12)])
def test_single_pair_tiles_equal_oracle(ctx, m, n, d):
    p = wl.uniform_pair(m, n, d, 7 * m + n, "dirichlet")
    r = oracle.solve_pair(p, "l2", threads=0)
    for make in (lambda v: dev(v, torch.float32), shifted):
        got = ctx.solve(make(p.x), dev(p.a, torch.float64), make(p.y), dev(p.b, torch.float64), metric="l2")
        assert got.cost == r.cost and got.stats["rounds"] == r.rounds
