"""Contexts on several host threads at once, in the entry points whose launches
differ in shared memory from call to call: every call succeeds with the results
of the same call alone."""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def run_threads(jobs, repeats):
    """jobs: functions of a context.  Each on its own thread, stream and context."""
    from paper_2401_07378_gb300 import nnsemd
    want = []
    for job in jobs:
        c = nnsemd.Context(0)
        want.append(job(c))
        c.close()
    torch.cuda.synchronize()
    start = threading.Barrier(len(jobs))
    failed = []

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                c = nnsemd.Context(0)
                start.wait()
                for _ in range(repeats):
                    got = jobs[k](c)
                    assert all(torch.equal(g, w) for g, w in zip(got, want[k]))
                c.close()
        except Exception as e:  # noqa: BLE001 (reported by the test)
            failed.append((k, repr(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[:3]


def test_kmeans_of_different_sizes():
    g = torch.Generator(device="cuda").manual_seed(5)
    pts = torch.rand(4000, 3, generator=g, device="cuda")
    torch.cuda.synchronize()
    run_threads([lambda c, k=k: c.kmeans(pts, k, 3) for k in (512, 8, 600, 64)], 200)


def test_reduced_precision_rows_of_different_lengths():
    g = torch.Generator(device="cuda").manual_seed(6)
    jobs = []
    for d in (390, 500, 700):
        x, y = (torch.randn(2300, d, generator=g, device="cuda") for _ in range(2))
        a, b = (torch.rand(2300, generator=g, device="cuda", dtype=torch.float64) + 0.1 for _ in range(2))
        jobs.append(lambda c, v=(x, a, y, b): (torch.tensor(c.solve(*v, precision="fp8").cost),))
    torch.cuda.synchronize()
    run_threads(jobs, 20)


def test_batched_reduced_precision_rows_of_different_lengths():
    g = torch.Generator(device="cuda").manual_seed(7)
    off = torch.arange(0, 9 * 600, 600).numpy()
    jobs = []
    for d, precision in ((16, "fp16"), (150, "fp16"), (90, "fp16"), (200, "bf16")):
        x, y = (torch.randn(8 * 600, d, generator=g, device="cuda") for _ in range(2))
        a, b = (torch.rand(8 * 600, generator=g, device="cuda", dtype=torch.float64) + 0.1 for _ in range(2))
        jobs.append(lambda c, v=(x, a, off, y, b, off), p=precision: (c.solve_batched(*v, precision=p)[0],))
    torch.cuda.synchronize()
    run_threads(jobs, 20)
