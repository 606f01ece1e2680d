"""The batched tensor-core solver's candidate lists and cache (pairs above 512
points per side), and the key-matrix route of smaller pairs, on inputs with
equal keys, zero weights and odd dimensions: costs, rounds and the number of
searches against the oracle."""
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


def pairs_of(d):
    out = []
    for k, (m, n) in enumerate([(513, 12), (5, 600), (640, 515), (530, 900), (300, 512), (64, 70), (1025, 513)]):
        p = wl.uniform_pair(m, n, d, 17 * d + k, "dirichlet")
        if k % 2 == 0:  # coarse grid: many equal keys, more than a list holds
            p.x[:], p.y[:] = np.round(p.x), np.round(p.y)
        if k in (2, 4):  # zero weights: the scan path from the first list on
            p.a[::4] = 0.0
            p.b[1::5] = 0.0
        if k == 3:  # nearly equal distances: the certificate fails at low precision
            p.x[:] = 1.0 + 1e-3 * p.x
            p.y[:] = 1.0 + 1e-3 * p.y
        out.append(p)
    return out


@pytest.mark.parametrize("d", [9, 50, 64])
def test_lists_equal_oracle(ctx, d):
    pairs = pairs_of(d)
    ref = [oracle.solve_pair(p, "l2") for p in pairs]
    b = wl.Batch.pack(pairs)
    args = (dev(b.x, torch.float32), dev(b.a, torch.float64), b.x_off, dev(b.y, torch.float32),
            dev(b.b, torch.float64), b.y_off)
    searches = sum(int(r.n_t.sum()) for r in ref)
    for precision in ("bf16", "fp16", "fp8", "bf16x3"):
        for rk in (0, 1, 3):
            costs, stats = ctx.solve_batched(*args, metric="l2", precision=precision, rerank_k=rk)
            assert costs.cpu().numpy().tolist() == [r.cost for r in ref], (precision, rk)
            assert stats["rounds"] == sum(r.rounds for r in ref)
            assert stats["certified"] + stats["fallbacks"] == searches, (precision, rk, stats)
