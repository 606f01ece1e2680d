"""The statistics of the multi-CTA rounds' NNS steps: rounds, the pairs their
durations stand for, and a duration for every round that evaluated any."""
import numpy as np
import pytest

import oracle
from paper_2401_07378_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def dev(a, dt):
    return torch.from_numpy(np.ascontiguousarray(a)).to(device="cuda", dtype=dt)


@pytest.mark.parametrize("n,d,precision", [(20000, 3, "fp32"), (5000, 5, "fp32"), (4000, 40, "fp32"),
                                           (6000, 64, "bf16x3"), (6000, 33, "fp16"), (3000, 200, "bf16")])
def test_rounds_pairs_and_time(n, d, precision):
    from paper_2401_07378_gb300 import nnsemd
    ctx = nnsemd.Context(0)
    p = wl.gmm_pair(2, n=n, d=d, components=30)
    r = oracle.solve_pair(p, "l2", threads=0)
    st = ctx.solve(dev(p.x, torch.float32), dev(p.a, torch.float64), dev(p.y, torch.float32), dev(p.b, torch.float64),
                   metric="l2", precision=precision, flags=nnsemd.FLAG_TIME_KERNELS).stats
    rounds = st["nns_kernel_launches"]
    full = int((r.m_t[:rounds] * r.n_t[:rounds]).sum())
    assert rounds >= 1 and st["pair_evals"] == r.pair_evals and st["nns_kernel_ms"] > 0.0
    if precision == "fp32":
        assert st["nns_kernel_pairs"] == full
    else:
        first = int(r.m_t[0] * r.n_t[0])
        assert first <= st["nns_kernel_pairs"] <= full
        assert st["certified"] + st["fallbacks"] == int(r.n_t[:rounds].sum())
    ctx.close()
