"""Solves whose workspace does not fit with the buffers of the faster steps (key
matrices, candidate lists, the grid): they run without those, to the same
results.  The refusal comes from a fake cudaMalloc preloaded into a child
process."""
import os
import shutil
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "native", "fake_cuda_malloc.c")

CHILD = r'''
import ctypes, sys
import numpy as np, torch
sys.path.insert(0, sys.argv[1])
import oracle
from paper_2401_07378_gb300 import nnsemd, workloads as wl

fake = ctypes.CDLL(sys.argv[2])
fake.fake_malloc_limit.argtypes = [ctypes.c_size_t]
fake.fake_malloc_asked.restype = ctypes.c_size_t
dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()

def twice(run, want):
    """With all the memory, then with less than the first workspace (on a fresh
    context, and again on it): the same results in a smaller workspace."""
    asked = []
    for limit in (0, None):
        torch.cuda.synchronize()
        fake.fake_malloc_asked()
        ctx = nnsemd.Context(0)
        fake.fake_malloc_limit(asked[0] - 1 if limit is None else 0)
        got = run(ctx)
        fake.fake_malloc_limit(0)
        asked.append(fake.fake_malloc_asked())
        assert got == want, (limit, got, want)
        if limit is None:
            assert run(ctx) == want
        ctx.close()
    assert asked[1] == asked[0], asked  # the large layout was asked for first, and refused

def single(m, n, d, metric="l2", **kw):
    p = wl.uniform_pair(m, n, d, m + n + d, "dirichlet")
    t = [dev(v) for v in (p.x, p.a, p.y, p.b)]
    r = oracle.solve_pair(p, metric, threads=0)
    def run(ctx):
        got = ctx.solve(*t, metric=metric, **kw)
        return got.cost, got.stats["rounds"]
    twice(run, (r.cost, r.rounds))
    def host(ctx):
        got = ctx.solve_host(p.x, p.a, p.y, p.b, metric=metric, **kw)
        return got.cost, got.stats["rounds"]
    twice(host, (r.cost, r.rounds))

def batch(sizes, d, metric="l2", **kw):
    pairs = [wl.uniform_pair(m, n, d, 7 * k + d, "dirichlet") for k, (m, n) in enumerate(sizes)]
    for p in pairs[::2]:
        p.x[:], p.y[:] = np.round(3 * p.x), np.round(3 * p.y)
    pairs[0].y[::3] *= 1e20  # every key of theirs is infinite
    b = wl.Batch.pack(pairs)
    t = [dev(b.x), dev(b.a), b.x_off, dev(b.y), dev(b.b), b.y_off]
    want = [oracle.solve_pair(p, metric, threads=0).cost for p in pairs]
    def run(ctx):
        return ctx.solve_batched(*t, metric=metric, **kw)[0].cpu().tolist()
    twice(run, want)

torch.zeros(1, device="cuda")
single(20000, 19000, 3)
single(2500, 2300, 40)
single(1800, 900, 20, metric="l1")
single(3000, 2800, 64, precision="fp16")
single(300, 200, 16)
batch([(600, 700), (100, 90), (512, 512), (2048, 1500), (64, 65), (1, 30)], 33)
batch([(600, 700), (100, 90), (513, 20)], 16, metric="l1")
batch([(600, 700), (100, 90), (2500, 2100), (512, 300)], 32, precision="bf16")
print("child ok")
'''


def test_without_the_faster_steps(tmp_path):
    cc = shutil.which("gcc")
    if cc is None:
        pytest.skip("no C compiler")
    so = str(tmp_path / "fake_cuda_malloc.so")
    subprocess.run([cc, "-shared", "-fPIC", "-O1", "-o", so, SRC, "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=so)
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT, so], capture_output=True, text=True, env=env, timeout=300)
    assert r.returncode == 0 and "child ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
