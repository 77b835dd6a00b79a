"""Handles dropped while a call that only enqueues is still running on the stream:
the results are those of the same calls with a synchronisation in between."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
msp = pytest.importorskip("paper_1807_08848_gb300")


def test_handles_destroyed_with_work_in_flight():
    N = 128
    ms, ps = synth.lognormal(N, 1 / 16, 32, 3), synth.uniform_patches(N, 4, 4, 8, 40)
    phi = torch.tensor(synth.phi_fourier(N, 16, 5, batch=32), device="cuda")

    def one(wait):
        med = msp.Medium(ms, ps)
        med.sample(1, "fp64", tol=1e-12, max_iter=20000)
        snap = med.snapshots(5)
        basis = med.extract(1e-6, "fp64")
        u, _ = basis.solve(phi, tol=1e-10, want_iters=False)
        if wait:
            torch.cuda.synchronize()
        del basis, med
        return u, snap

    ref, rsnap = (t.clone() for t in one(True))
    for _ in range(3):
        u, snap = one(False)
        assert torch.equal(u, ref) and torch.equal(snap, rsnap)
