"""NNSEMD_FLAG_GRAPH with the same buffers split into pairs in more ways than a
context keeps graphs: every call gives the result of the call without it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,precision", [(2, "fp32"), (16, "fp32"), (32, "fp16")])
def test_many_splits(d, precision):
    from paper_2401_07378_gb300 import nnsemd
    ctx = nnsemd.Context(0)
    g = torch.Generator(device="cuda").manual_seed(d)
    total = 6000
    x, y = (torch.rand(total, d, generator=g, device="cuda") for _ in range(2))
    a, b = (torch.rand(total, generator=g, device="cuda", dtype=torch.float64) + 0.1 for _ in range(2))
    rng = np.random.default_rng(d)
    splits = []
    for _ in range(40):
        cut = np.sort(rng.choice(np.arange(100, total, 100), rng.integers(8, 14), replace=False))
        splits.append(np.concatenate([[0], cut, [total]]).astype(np.int64))
    for off in splits + splits[:3]:
        want, _ = ctx.solve_batched(x, a, off, y, b, off, precision=precision)
        got = torch.full_like(want, float("nan"))
        ctx.solve_batched(x, a, off, y, b, off, precision=precision, costs=got, flags=nnsemd.FLAG_GRAPH)
        assert torch.equal(got, want)
    ctx.close()
