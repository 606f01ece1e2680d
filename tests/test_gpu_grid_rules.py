"""Which rounds take the spatially ordered NNS step (d <= 3, both sides large),
told from the launches a solve makes, and its results at those sizes against the
oracle."""
import numpy as np
import pytest

import oracle
from paper_2401_07378_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIDE = 1 << 14       # the smaller side from which a round takes the step
ROUND, GRID = 7, 5   # launches of a round with K1; what the step adds to it


@pytest.fixture(scope="module")
def ctx():
    from paper_2401_07378_gb300 import nnsemd
    c = nnsemd.Context(0)
    yield c
    c.close()


def dev(a, dt):
    return torch.from_numpy(np.ascontiguousarray(a)).to(device="cuda", dtype=dt)


def solve(ctx, p, metric="l2"):
    return ctx.solve(dev(p.x, torch.float32), dev(p.a, torch.float64), dev(p.y, torch.float32),
                     dev(p.b, torch.float64), metric=metric)


def grid_rounds(stats):
    """Rounds that took the step: the launches beside the rounds' own are 4 to set
    up, 2 to finish, the tail if one ran, and for the step its own and the box."""
    return (stats["kernel_launches"] - ROUND * stats["nns_kernel_launches"] - 6) // GRID


def cloud(n, d, rng):
    return rng.random((n, d)).astype(np.float32)


@pytest.mark.parametrize("m,n,d,want", [(SIDE, SIDE, 1, True), (SIDE, SIDE + 77, 2, True), (20011, SIDE, 3, True),
                                        (SIDE - 1, 30000, 3, False), (30000, SIDE - 1, 2, False),
                                        (100000, 1000, 3, False)])
def test_size_rule(ctx, m, n, d, want):
    rng = np.random.default_rng(m + n)
    p = wl.Pair(cloud(m, d, rng), rng.exponential(1.0, m), cloud(n, d, rng), rng.exponential(1.0, n))
    for metric in ("l2", "l1"):
        r = oracle.solve_pair(p, metric, threads=0)
        got = solve(ctx, p, metric)
        assert got.cost == r.cost and got.stats["rounds"] == r.rounds and got.stats["pair_evals"] == r.pair_evals
        assert (grid_rounds(got.stats) > 0) == want, got.stats
