"""Finite points so far out that FP32 squared distances, or the squared norms
of the reduced-precision passes, overflow (d > 8): costs and rounds against the
oracle, whose first position wins among infinite keys."""
import numpy as np
import pytest

import oracle
from paper_2401_07378_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FAR = 1e20  # its square is above FP32's range


@pytest.fixture(scope="module")
def ctx():
    from paper_2401_07378_gb300 import nnsemd
    c = nnsemd.Context(0)
    yield c
    c.close()


def dev(a, dt):
    return torch.from_numpy(np.ascontiguousarray(a)).to(device="cuda", dtype=dt)


def batch_args(pairs):
    b = wl.Batch.pack(pairs)
    return (dev(b.x, torch.float32), dev(b.a, torch.float64), b.x_off, dev(b.y, torch.float32),
            dev(b.b, torch.float64), b.y_off)


def pair_args(p):
    return dev(p.x, torch.float32), dev(p.a, torch.float64), dev(p.y, torch.float32), dev(p.b, torch.float64)


def far_consumers(m, n, d, seed, every=7):
    """Consumers (every so many, the first among them) whose keys are all +inf."""
    p = wl.uniform_pair(m, n, d, seed, "dirichlet")
    p.y[::every] *= FAR
    p.y[::every, 0] = FAR
    return p


def far_suppliers(m, n, d, seed):
    """Every other supplier so far out that its squared norm overflows, some
    consumers beside those, and little weight on the first supplier."""
    p = wl.uniform_pair(m, n, d, seed, "dirichlet")
    p.x[1::2] *= FAR
    p.x[1::2, 0] = FAR
    far = p.x[1::2]
    k = p.y[::3].shape[0]
    p.y[::3] = far[np.arange(k) % far.shape[0]] * np.float32(1 + 2 ** -12)
    p.a[0] = 1e-3 * p.a.min()
    return p


@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp16", "fp8", "bf16x3"])
@pytest.mark.parametrize("d", [9, 64])
def test_batched_far_consumers(ctx, d, precision):
    pairs = [far_consumers(m, n, d, 5 * d + k, every)
             for k, (m, n, every) in enumerate([(513, 12, 1), (5, 600, 3), (700, 515, 7), (300, 200, 2), (530, 900, 1)])]
    ref = [oracle.solve_pair(p, "l2") for p in pairs]
    costs, stats = ctx.solve_batched(*batch_args(pairs), metric="l2", precision=precision)
    assert costs.cpu().numpy().tolist() == [r.cost for r in ref]
    assert stats["rounds"] == sum(r.rounds for r in ref)


@pytest.mark.parametrize("rk", [0, 3])
@pytest.mark.parametrize("precision", ["bf16", "fp16", "fp8", "bf16x3"])
@pytest.mark.parametrize("d", [9, 64])
def test_batched_far_suppliers(ctx, d, precision, rk):
    pairs = [far_suppliers(m, n, d, 3 * d + k)
             for k, (m, n) in enumerate([(2, 513), (5, 600), (8, 700), (9, 530), (24, 1025), (520, 7), (600, 640)])]
    ref = [oracle.solve_pair(p, "l2") for p in pairs]
    costs, stats = ctx.solve_batched(*batch_args(pairs), metric="l2", precision=precision, rerank_k=rk)
    assert costs.cpu().numpy().tolist() == [r.cost for r in ref]
    assert stats["rounds"] == sum(r.rounds for r in ref)
    assert stats["certified"] + stats["fallbacks"] == sum(int(r.n_t.sum()) for r in ref)


@pytest.mark.parametrize("metric", ["l2", "sql2"])
def test_large_far_consumers_fp32(ctx, metric):
    p = far_consumers(3000, 2500, 40, 3)
    r = oracle.solve_pair(p, metric, threads=0)
    got = ctx.solve(*pair_args(p), metric=metric)
    assert got.cost == r.cost and got.stats["rounds"] == r.rounds


@pytest.mark.parametrize("precision", ["bf16", "fp16", "fp8", "bf16x3"])
@pytest.mark.parametrize("m,n,d", [(3000, 2500, 40), (40, 4000, 64), (17, 9000, 64)])
def test_large_reduced_precision(ctx, m, n, d, precision):
    for p in (far_consumers(m, n, d, m), far_suppliers(m, n, d, n)):
        r = oracle.solve_pair(p, "l2", threads=0)
        for rk in (0, 8):
            got = ctx.solve(*pair_args(p), metric="l2", precision=precision, rerank_k=rk)
            assert got.cost == r.cost and got.stats["rounds"] == r.rounds
            assert got.stats["certified"] + got.stats["fallbacks"] <= int(r.n_t.sum())
