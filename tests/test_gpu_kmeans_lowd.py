"""The one-pass k-means of low-dimensional points (assignment, narrow exact
sums, sizes) at the edges of its tiles and rules, and the barycentric map's
rounding for any d, bit for bit against the oracle and exact sums."""
import math

import numpy as np
import pytest

from oracle import colour

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2401_07378_gb300 import nnsemd
    c = nnsemd.Context(0)
    yield c
    c.close()


# k at group and tile edges; k * d beyond the shared-memory sums; more
# centroids than one staged tile; N below and above four points per thread
@pytest.mark.parametrize("n,d,k,iters", [(1, 1, 1, 2), (777, 2, 7, 3), (4001, 3, 8, 3), (4001, 3, 9, 0),
                                         (5003, 4, 512, 2), (6001, 5, 31, 2), (3001, 8, 256, 2), (3001, 8, 257, 2),
                                         (5001, 3, 1030, 2), (4099, 1, 2048, 1), (160001, 3, 5, 2)])
def test_kmeans_equals_oracle(ctx, n, d, k, iters):
    rng = np.random.default_rng(n + d)
    pts = rng.random((n, d)).astype(np.float32)
    pts[::5] = np.round(pts[::5] * 8) / 8           # equal keys
    pts[::7] *= np.float32(1e-38)                   # subnormal products and values
    pts[3::11] *= np.float32(2.0 ** 40)             # far exponents in one sum
    cent, lab, cnt = ctx.kmeans(torch.from_numpy(pts).cuda(), k, iters)
    rc, rl, rn = colour.kmeans(pts, k, iters)
    assert np.array_equal(cent.cpu().numpy(), rc)
    assert np.array_equal(lab.cpu().numpy(), rl)
    assert np.array_equal(cnt.cpu().numpy(), rn)


@pytest.mark.parametrize("bad", [-1e-3, float("nan"), float("inf")])
def test_refused_points_leave_the_context_usable(ctx, bad):
    from paper_2401_07378_gb300 import nnsemd
    pts = torch.rand(3000, 3, device="cuda")
    pts[1234, 1] = bad
    with pytest.raises(nnsemd.NNSEMDError) as e:
        ctx.kmeans(pts, 16, 2)
    assert e.value.status == 2
    pts[1234, 1] = 0.5
    assert int(ctx.kmeans(pts, 16, 2)[2].sum()) == 3000


@pytest.mark.parametrize("d", [1, 7, 8, 12])
def test_barycentric_equals_exact_sums(ctx, d):
    rng = np.random.default_rng(d)
    m, n, nnz = 40, 33, 200
    x, y = rng.random((m, d)).astype(np.float32), rng.random((n, d)).astype(np.float32)
    i, j = rng.integers(0, m, nnz).astype(np.int32), rng.integers(0, n - 1, nnz).astype(np.int32)
    f = rng.exponential(1.0, nnz)
    t = lambda v: torch.from_numpy(v).cuda()
    got = ctx.barycentric(t(i), t(j), t(f), t(x), t(y)).cpu().numpy()
    for q in range(n):
        at = np.nonzero(j == q)[0]
        w = math.fsum(f[at])
        want = [np.float32(math.fsum(f[at] * x[i[at], c].astype(np.float64)) / w) if at.size else y[q, c]
                for c in range(d)]
        assert got[q].tolist() == [float(v) for v in want]
