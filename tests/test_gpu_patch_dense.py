"""The per-patch dense kernels of the extraction at the orders where their layouts
change: panel edges (15..17 columns), the line between one CTA and a cluster per patch
(47..49 and 160, 161), and orders beyond a cluster's shared memory (600).

Reference: numpy's SVD of the snapshot blocks the device holds.  Tolerances: singular
values to 1e-10 sigma_1 where the sweeps resolve them (0.1 tau sigma_1 and above; the
shifted Cholesky-QR3 is backward stable to about 1e-12 sigma_1), bases orthonormal to
1e-10 and spanning the leading left singular vectors to 1e-11 sigma_1 / gap (Wedin),
the bounds the tensor-core product tests use."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
msp = pytest.importorskip("paper_1807_08848_gb300")

# (cells per patch side, buffer, samples): 2 x 2 patches, columns = samples + 2 (side + buffer) + 1
CASES = [(4, 2, 2), (4, 2, 3), (4, 2, 4), (12, 2, 18), (12, 2, 19), (12, 2, 20), (32, 4, 87), (32, 4, 88), (32, 4, 250),
         (32, 4, 527)]


@pytest.mark.parametrize("side,buffer,samples", CASES)
def test_bases_at_layout_edges(side, buffer, samples):
    N, tau = 2 * side, 1e-6
    med = msp.Medium(synth.lognormal(N, 4.0 / N, 16, 3), synth.uniform_patches(N, 2, 2, buffer, samples))
    med.sample(11, "fp64", tol=1e-12, max_iter=20000)
    basis = med.extract(tau, "fp64")
    for m in range(med.n_patches):
        R = med.snapshots(m).cpu().numpy()
        assert R.shape[1] == samples + 2 * (side + buffer) + 1
        U, s, _ = np.linalg.svd(R, full_matrices=False)
        got, Q = basis.sigma(m), basis.Q(m).cpu().numpy()
        res = s >= 0.1 * tau * s[0]
        assert np.max(np.abs(got[: len(s)] - s)[res]) <= 1e-10 * s[0], m
        assert np.all(got[: len(s)][~res] < tau * s[0]), m
        if np.min(np.abs(s / s[0] / tau - 1.0)) > 1e-3:
            assert basis.k(m) == int(np.sum(s > tau * s[0])), m
        assert np.max(np.abs(Q.T @ Q - np.eye(Q.shape[1]))) <= 1e-10, m
        for j in range(1, Q.shape[1]):
            gap = s[j - 1] - s[j]
            if gap > 1e-3 * s[0]:
                assert np.linalg.norm(U[:, :j] - Q[:, :j] @ (Q[:, :j].T @ U[:, :j]), 2) <= 1e-11 * s[0] / gap + 1e-10


@pytest.mark.parametrize("side,samples", [(4, 2), (4, 3), (4, 4), (12, 3), (12, 18), (12, 20)])
def test_many_patches(side, samples):
    """81 patches: from 1216 columns on (at 152 SMs) a warp of the triangular inverse takes
    four columns, here with one to three of them beyond the block's order."""
    N = 9 * side
    med = msp.Medium(synth.lognormal(N, 4.0 / N, 16, 3), synth.uniform_patches(N, 9, 9, 2, samples))
    med.sample(12, "fp64", tol=1e-12, max_iter=20000)
    basis = med.extract(1e-6, "fp64")
    for m in range(0, 81, 8):
        R = med.snapshots(m).cpu().numpy()
        s = np.linalg.svd(R, compute_uv=False)
        got, Q = basis.sigma(m), basis.Q(m).cpu().numpy()
        res = s >= 1e-7 * s[0]
        assert np.max(np.abs(got[: len(s)] - s)[res]) <= 1e-10 * s[0], m
        assert np.max(np.abs(Q.T @ Q - np.eye(Q.shape[1]))) <= 1e-10, m
        assert np.linalg.norm(R - Q @ (Q.T @ R), 2) <= 1.01e-6 * s[0] + 1e-10 * s[0], m
