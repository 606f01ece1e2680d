"""Batched pairs (d > 8) of which only some points have weight: the key matrices
and the tensor-core kernel's distance cache hold those alone, by original index;
costs, rounds and searches against the oracle."""
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


def keep(w, share, rng):
    """Weights of which about this share is not zero (one at least)."""
    out = np.where(rng.random(w.size) < share, w, 0.0)
    out[rng.integers(w.size)] = 1.0
    return out


def pairs_of(sizes, d, seed):
    out = []
    for k, (m, n, sa, sb) in enumerate(sizes):
        rng = np.random.default_rng(seed + k)
        p = wl.uniform_pair(m, n, d, seed + 31 * k, "dirichlet")
        p.a[:], p.b[:] = keep(p.a, sa, rng), keep(p.b, sb, rng)
        if k % 2:  # equal keys
            p.x[:], p.y[:] = np.round(3 * p.x), np.round(3 * p.y)
        out.append(p)
    return out


SIZES = [(70, 61, 0.2, 0.3), (512, 500, 0.02, 0.5), (300, 512, 1.0, 0.05), (512, 64, 0.3, 1.0),
         (900, 1100, 0.05, 0.04), (2048, 2047, 0.3, 0.004), (1300, 700, 0.01, 1.0), (700, 1300, 1.0, 0.6),
         (1025, 1023, 0.5, 0.5)]


@pytest.mark.parametrize("metric,precision", [("l2", "fp32"), ("l1", "fp32"), ("l2", "fp16"), ("sql2", "bf16x3"),
                                              ("l2", "fp8")])
@pytest.mark.parametrize("d", [9, 64])
def test_few_points_with_weight(ctx, d, metric, precision):
    pairs = pairs_of(SIZES, d, 1000 + d)
    ref = [oracle.solve_pair(p, metric) for p in pairs]
    b = wl.Batch.pack(pairs)
    costs, stats = ctx.solve_batched(dev(b.x, torch.float32), dev(b.a, torch.float64), b.x_off, dev(b.y, torch.float32),
                                     dev(b.b, torch.float64), b.y_off, metric=metric, precision=precision)
    assert costs.cpu().numpy().tolist() == [r.cost for r in ref]
    assert stats["rounds"] == sum(r.rounds for r in ref) and stats["pair_evals"] == sum(r.pair_evals for r in ref)
    if precision != "fp32":
        assert stats["certified"] + stats["fallbacks"] == sum(int(r.n_t.sum()) for r in ref)
