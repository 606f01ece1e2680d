"""Cluster tails whose rounds all run inside each CTA (few points: no barrier
between the CTAs from the opening one to the last): cost, rounds and pair
evaluations of many solves in a row, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2401_07378_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,d", [(2, 1, 9), (1, 2, 16), (64, 64, 50), (30, 9, 300), (2000, 8, 3), (5, 1500, 2)])
def test_many_small_tails(m, n, d):
    from paper_2401_07378_gb300 import nnsemd
    ctx = nnsemd.Context(0)
    p = wl.uniform_pair(m, n, d, 11 * m + n, "dirichlet")
    r = oracle.solve_pair(p, "l2")
    args = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (p.x, p.a, p.y, p.b)]
    for _ in range(200):
        got = ctx.solve(*args, metric="l2")
        assert got.cost == r.cost
        assert got.stats["rounds"] == r.rounds and got.stats["pair_evals"] == r.pair_evals
    ctx.close()
