"""Which rounds take the spatially ordered NNS step (d <= 3, both sides large),
told from the launches a solve makes, and its results at those sizes against the
oracle."""
import numpy as np
import pytest

import oracle
from paper_2401_07378_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIDE = 7 << 11       # the smaller side from which a round takes the step
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


def points(kind, n, d, rng, consumers):
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
    if kind == "ring":  # every supplier about as near as any other
        p = rng.normal(size=(n, d))
        return 1e-3 * p if consumers else p / np.linalg.norm(p, axis=1, keepdims=True)
    if kind == "line":  # an axis without extent
        p = rng.random((n, d))
        p[:, -1] = 0.25
        return p
    if kind == "tiny":  # squares in the subnormal range
        return rng.random((n, d)) * 1e-20
    if kind == "huge":  # squares overflow
        return (rng.random((n, d)) - 0.5) * 1e20
    raise ValueError(kind)


# want: rounds with the step (None: not told); one where it refuses the points
@pytest.mark.parametrize("kind,d,want", [("uniform", 3, None), ("clusters", 2, None), ("lattice", 3, None),
                                         ("line", 2, None), ("tiny", 3, None), ("huge", 3, None),
                                         ("outlier", 1, 1), ("outlier", 3, 1), ("ring", 2, 1),
                                         ("ring", 3, 1)])
def test_refused_points_try_the_step_once(ctx, kind, d, want):
    rng = np.random.default_rng(len(kind) + d)
    m, n = (34000, 33900) if want else (SIDE + 1, SIDE + 16)  # (more than one round of that size where it matters)
    p = wl.Pair(points(kind, m, d, rng, False).astype(np.float32), rng.exponential(1.0, m),
                points(kind, n, d, rng, True).astype(np.float32), rng.exponential(1.0, n))
    if not want:
        p.a[::11 * SIDE] = 0.0
    for metric in ("l2",) if kind in ("tiny", "huge") or want else ("l2", "l1"):
        r = oracle.solve_pair(p, metric, threads=0)
        got = solve(ctx, p, metric)
        assert got.cost == r.cost and got.stats["rounds"] == r.rounds and got.stats["pair_evals"] == r.pair_evals
        took = grid_rounds(got.stats)
        assert took >= 1
        if want:
            assert took == want and int((np.minimum(r.m_t, r.n_t) >= SIDE).sum()) > want
