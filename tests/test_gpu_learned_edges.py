"""Solves with a proposal at the edges of its passes' tiles and selections
(128 x 128 blocks of rows and cells, rows of 256 and of 4,096 columns, 64 cells
kept), against the oracle bit for bit."""
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


@pytest.mark.parametrize("d,hidden", [(64, 256), (48, 80), (32, 16), (128, 32)])
@pytest.mark.parametrize("cells,n", [(64, 2100), (129, 2177), (256, 2049), (263, 2500), (512, 2560), (1030, 4097),
                                     (4096, 4500), (6400, 6500)])
def test_solve_with_proposal_equals_oracle(ctx, d, hidden, cells, n):
    from paper_2401_07378_gb300 import nnsemd
    p = wl.gmm_pair(cells + d, n=n, d=d, components=50)
    p.x[:] = np.round(p.x * 8) / 8  # equal keys, equal rows
    p.y[:] = np.round(p.y * 8) / 8
    t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()
    prop = nnsemd.Proposal(ctx, d, cells=cells, hidden=hidden, seed=5)
    prop.fit(t(p.x), iters=2, seed=1)
    ref = oracle.solve_pair(p, "l2", threads=0)
    for precision in ("fp32", "bf16"):
        res = ctx.solve(t(p.x), t(p.a), t(p.y), t(p.b), metric="l2", precision=precision, plan=True, proposal=prop)
        assert res.cost == ref.cost and res.stats["rounds"] == ref.rounds
        assert sorted(zip(res.plan_i.tolist(), res.plan_j.tolist(), res.plan_f.tolist())) == sorted(
            zip(ref.plan_i.tolist(), ref.plan_j.tolist(), ref.plan_f.tolist()))
    prop.close()
