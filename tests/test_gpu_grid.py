"""The spatially ordered NNS step of large rounds (d <= 3) on distributions that
stretch its order, bounds and rule, against the oracle bit for bit."""
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


def points(kind, n, d, rng):
    if kind == "uniform":
        return rng.random((n, d))
    if kind == "clusters":
        c = np.random.default_rng(5).random((6, d))
        return c[rng.integers(0, 6, n)] + rng.normal(0, 0.01, (n, d))
    if kind == "lattice":  # many equal points and keys
        return rng.integers(0, 40, (n, d)) - 20.0
    if kind == "outlier":  # one far point: every other one in a single cell
        p = rng.random((n, d)) * 1e-3
        p[0] = 1e6
        return p
    if kind == "line":  # an axis without extent
        p = rng.random((n, d))
        p[:, -1] = 0.25
        return p
    if kind == "tiny":  # squares in the subnormal range
        return rng.random((n, d)) * 1e-20
    if kind == "huge":  # squares overflow
        return (rng.random((n, d)) - 0.5) * 1e20
    raise ValueError(kind)


CASES = [("uniform", 1), ("uniform", 2), ("uniform", 3), ("clusters", 2), ("clusters", 3), ("lattice", 1), ("lattice", 2),
         ("lattice", 3), ("outlier", 3), ("line", 2), ("line", 3), ("tiny", 3), ("huge", 3)]


@pytest.mark.parametrize("kind,d", CASES)
def test_grid_step_equals_oracle(ctx, kind, d):
    rng = np.random.default_rng(len(kind) + d)
    m, n = (8193, 8200) if kind != "uniform" else (20011, 5003)
    p = wl.Pair(points(kind, m, d, rng).astype(np.float32), rng.exponential(1.0, m),
                points(kind, n, d, rng).astype(np.float32), rng.exponential(1.0, n))
    p.a[::11] = 0.0
    for metric in ("l2",) if kind in ("tiny", "huge") else ("l2", "l1"):
        r = oracle.solve_pair(p, metric, threads=0)
        got = ctx.solve(dev(p.x, torch.float32), dev(p.a, torch.float64), dev(p.y, torch.float32),
                        dev(p.b, torch.float64), metric=metric, plan=True)
        assert got.cost == r.cost and got.stats["rounds"] == r.rounds and got.stats["pair_evals"] == r.pair_evals
        assert sorted(zip(got.plan_i.tolist(), got.plan_j.tolist(), got.plan_f.tolist())) == sorted(
            zip(r.plan_i.tolist(), r.plan_j.tolist(), r.plan_f.tolist()))
