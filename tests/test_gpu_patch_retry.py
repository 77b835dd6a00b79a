"""Cholesky-QR of snapshot blocks whose Gram matrices need a second try: columns that are
zero or repeat earlier ones leave non-positive pivots after the first, shifted pass.  The
first such column moves over the 16-column panels (and so over the CTAs that own them) from
patch to patch, for patches on one CTA, on a cluster, and on a cluster out of global memory.

Reference: numpy's SVD of the blocks.  Tolerances as for the full-rank blocks of
test_gpu_patch_dense.py: singular values to 1e-10 sigma_1, bases orthonormal to 1e-10, and
the leading subspace to 1e-10 (its gap is 1e-2 sigma_1)."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
msp = pytest.importorskip("paper_1807_08848_gb300")


@pytest.mark.parametrize("side,buffer,samples,rank", [(12, 2, 18, 10), (12, 2, 20, 10), (32, 4, 88, 60), (32, 4, 250, 60),
                                                      (32, 4, 527, 60)])
def test_dependent_columns(side, buffer, samples, rank):
    N, tau = 2 * side, 1e-6
    med = msp.Medium(synth.lognormal(N, 4.0 / N, 16, 3), synth.uniform_patches(N, 2, 2, buffer, samples))
    rng = np.random.Generator(np.random.PCG64(5))
    blocks = []
    for m in range(med.n_patches):
        n, c = med.patch(m).n_k, med.patch(m).cols
        U, _ = np.linalg.qr(rng.standard_normal((n, rank)))
        V, _ = np.linalg.qr(rng.standard_normal((c, rank)))
        R = (U * np.linspace(1.0, 1e-2, rank)) @ V.T
        first = [0, 15, c // 2, c - 2][m]           # first zero column, then a repeated one
        R[:, first] = 0.0
        R[:, c - 1] = R[:, 1]
        blocks.append(R)
        med.set_snapshots(m, torch.tensor(R, device="cuda"))
    basis = med.extract(tau, "fp64")
    assert basis.stats()["max_cholqr_tries"] >= 2
    for m, R in enumerate(blocks):
        U, s, _ = np.linalg.svd(R, full_matrices=False)
        k = int(np.sum(s > tau * s[0]))
        assert basis.k(m) == k, m
        got, Q = basis.sigma(m), basis.Q(m).cpu().numpy()
        assert np.max(np.abs(got[:k] - s[:k])) <= 1e-10 * s[0], m
        assert np.all(got[k:] < tau * s[0]), m
        assert np.max(np.abs(Q.T @ Q - np.eye(k))) <= 1e-10, m
        assert np.linalg.norm(U[:, :k] - Q @ (Q.T @ U[:, :k]), 2) <= 1e-10, m
