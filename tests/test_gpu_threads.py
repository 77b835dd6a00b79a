"""Host threads working on handles of their own at the same time, on streams of their own.
Each asks the same kernels for another amount of dynamic shared memory, call after call; every
call succeeds and its results are those of the thread alone."""
import threading

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
msp = pytest.importorskip("paper_1807_08848_gb300")


def run_together(jobs):
    """Every job (a callable) in a thread; the exceptions they ended with."""
    failures = []
    start = threading.Barrier(len(jobs))

    def body(job):
        try:
            start.wait()
            job()
        except Exception as e:      # reported by the caller
            failures.append(e)

    threads = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return failures


def test_operator_tiles_of_different_sizes():
    """Tiles of 21 to 41 nodes a side: one instance of the streaming kernel, 8 buffers of each."""
    jobs = []
    for N in (32, 48, 64, 72):
        med = msp.Medium(synth.lognormal(N, 4.0 / N, 16, 3), synth.uniform_patches(N, 2, 2, 4, 4))
        rows, cols = med.tile_shape()
        x = torch.randn((med.n_patches, 3, rows, (cols + 3) // 4 * 4), device="cuda")
        ref = med.apply_operator(x, "mixed")
        torch.cuda.synchronize()

        def job(med=med, x=x, ref=ref):
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                y = torch.empty_like(x)
                for _ in range(2000):
                    med.apply_operator(x, "mixed", y=y)
                s.synchronize()
                assert torch.equal(y, ref)

        jobs.append(job)
    assert run_together(jobs) == []


def test_extractions_of_different_orders():
    jobs = []
    for samples in (6, 20, 60, 150):
        med = msp.Medium(synth.lognormal(48, 1 / 12, 16, 3), synth.uniform_patches(48, 2, 2, 4, samples))
        med.sample(2, "mixed", tol=1e-10, max_iter=20000)
        ref = med.extract(1e-6)
        Q = [ref.Q(m).clone() for m in range(4)]
        torch.cuda.synchronize()

        def job(med=med, Q=Q):
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for _ in range(25):
                    basis = med.extract(1e-6)
                    for m in range(4):
                        assert torch.equal(basis.Q(m), Q[m])

        jobs.append(job)
    assert run_together(jobs) == []
