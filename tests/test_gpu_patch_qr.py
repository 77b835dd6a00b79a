"""The two forms of the pivoted QR and of the Jacobi sweeps (a cluster per patch, one CTA per
patch) on the same blocks: one snapshot block extracted as a patch of a 2 x 2 partition, whose
few patches take clusters, and as an inner patch of a 12 x 12 partition, whose many patches
take a CTA each, in shared memory or beyond it (164 columns).  Every step's arithmetic is that of a patch by itself, so
singular values and bases are the same bits; the SVD of the block is checked against numpy as
in test_gpu_patch_dense.py."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
msp = pytest.importorskip("paper_1807_08848_gb300")

SIDE, BUFFER, TAU = 6, 2, 1e-6
DELTAS = 2 * (SIDE + BUFFER) + 1     # boundary columns of a corner patch


@pytest.mark.parametrize("cols", [20, 48, 80, 81, 161, 163, 164, 200, 260])
def test_forms_agree(cols):
    few = msp.Medium(synth.lognormal(2 * SIDE, 1 / 3, 16, 3), synth.uniform_patches(2 * SIDE, 2, 2, BUFFER, cols - DELTAS))
    many = msp.Medium(synth.lognormal(12 * SIDE, 1 / 12, 16, 3),
                      synth.uniform_patches(12 * SIDE, 12, 12, BUFFER, cols))
    few.sample(1, "fp64", tol=1e-12, max_iter=20000)
    many.sample(1, "fp64", tol=1e-12, max_iter=20000)
    m = 6 + 12 * 5
    assert few.patch(0).cols == many.patch(m).cols == cols
    rng, rank = np.random.Generator(np.random.PCG64(cols)), 16
    R = (rng.standard_normal((few.patch(0).n_k, rank)) * np.logspace(0, -3, rank)) @ rng.standard_normal((rank, cols))
    block = torch.tensor(R, device="cuda")
    few.set_snapshots(0, block)
    many.set_snapshots(m, block)
    a, b = few.extract(TAU, "fp64"), many.extract(TAU, "fp64")
    assert a.k(0) == b.k(m) == rank
    assert np.array_equal(a.sigma(0), b.sigma(m))
    assert torch.equal(a.Q(0), b.Q(m))
    s = np.linalg.svd(R, compute_uv=False)
    Q = b.Q(m).cpu().numpy()
    res = s >= 0.1 * TAU * s[0]
    assert np.max(np.abs(b.sigma(m)[: len(s)] - s)[res]) <= 1e-10 * s[0]
    assert np.max(np.abs(Q.T @ Q - np.eye(Q.shape[1]))) <= 1e-10
    assert np.linalg.norm(R - Q @ (Q.T @ R), 2) <= 1.01 * TAU * s[0] + 1e-10 * s[0]
