"""One-CTA solves of small low-dimensional pairs at the edges of their
capacities and of the rounds of a few warps (64 points), single and batched, against
the oracle bit for bit."""
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


SIZES = [(1, 1), (3, 64), (64, 3), (65, 64), (63, 66), (129, 300), (512, 511), (511, 513), (513, 64), (1024, 700)]


def pairs_of(d):
    out = []
    for k, (m, n) in enumerate(SIZES):
        p = wl.uniform_pair(m, n, d, 31 * d + k, "dirichlet" if k % 2 else "uniform")
        if k % 3 == 0:  # equal keys and zero weights
            p.x[:], p.y[:] = np.round(p.x * 4) / 4, np.round(p.y * 4) / 4
            p.a[1::3] = 0.0
        # weights whose sums span many exponents
        if k % 4 == 1:
            p.a *= 10.0 ** np.random.default_rng(k).uniform(-30, 3, m)
        out.append(p)
    return out


@pytest.mark.parametrize("metric", ["l2", "sql2", "l1"])
@pytest.mark.parametrize("d", [1, 2, 3, 5, 8])
def test_small_pairs_equal_oracle(ctx, d, metric):
    pairs = pairs_of(d)
    ref = [oracle.solve_pair(p, metric) for p in pairs]
    for p, r in zip(pairs, ref):
        got = ctx.solve(dev(p.x, torch.float32), dev(p.a, torch.float64), dev(p.y, torch.float32),
                        dev(p.b, torch.float64), metric=metric, plan=True)
        assert got.cost == r.cost and got.stats["rounds"] == r.rounds
        assert sorted(zip(got.plan_i.tolist(), got.plan_j.tolist(), got.plan_f.tolist())) == sorted(
            zip(r.plan_i.tolist(), r.plan_j.tolist(), r.plan_f.tolist()))
    b = wl.Batch.pack(pairs)
    costs, stats = ctx.solve_batched(dev(b.x, torch.float32), dev(b.a, torch.float64), b.x_off,
                                     dev(b.y, torch.float32), dev(b.b, torch.float64), b.y_off, metric=metric)
    assert costs.cpu().numpy().tolist() == [r.cost for r in ref]
    assert stats["rounds"] == sum(r.rounds for r in ref)


@pytest.mark.parametrize("side,value,status", [("x", float("nan"), 2), ("y", float("inf"), 2), ("a", -1.0, 3),
                                               ("b", float("nan"), 2), ("both", -1.0, 3)])
def test_first_sides_error_is_reported(ctx, side, value, status):
    from paper_2401_07378_gb300 import nnsemd
    p = wl.uniform_pair(100, 90, 2, 5)
    t = dict(x=dev(p.x, torch.float32), a=dev(p.a, torch.float64), y=dev(p.y, torch.float32),
             b=dev(p.b, torch.float64))
    if side == "both":  # a negative weight of the first side before a coordinate of the second
        t["a"][7] = value
        t["y"][3, 0] = float("nan")
    else:
        t[side].view(-1)[7] = value
    with pytest.raises(nnsemd.NNSEMDError) as e:
        ctx.solve(t["x"], t["a"], t["y"], t["b"])
    assert e.value.status == status
