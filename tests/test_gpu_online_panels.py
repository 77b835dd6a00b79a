"""The online factor over block rows from one partial tile to more panel rows than a warp per
row takes (one CTA of eight rows per SM in FP64, two in FP32): the solution's normal-equation
residual, formed on the host from the exported rows, a hundred times the solve's tolerance, and
the iteration count, which a wrong factor would raise far above a right one's few steps."""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

import synth

pytestmark = pytest.mark.gpu
msp = pytest.importorskip("paper_1807_08848_gb300")


@pytest.mark.parametrize("columns,samples", [(2, 5), (4, 20), (8, 30), (24, 30), (32, 40), (48, 44)])
def test_block_rows(columns, samples):
    """columns x 2 patches of 8 cells' width: block rows of about columns x samples unknowns."""
    N = 8 * columns
    x = np.arange(columns + 1) * 8
    ps = synth.PatchSpec(x, np.array([0, N // 2, N]), np.full(2 * columns, 4), np.full(2 * columns, samples))
    med = msp.Medium(synth.lognormal(N, 8.0 / N, 16, 3), ps)
    med.sample(5, "mixed", tol=1e-11, max_iter=20000)
    basis = med.extract(1e-6)
    phi = synth.phi_sin_cos(N)
    u, iters, c = basis.solve(torch.tensor(phi, device="cuda"), tol=1e-11, max_iter=50, want_c=True)
    assert int(iters[0]) <= 8
    r, q, v, d = basis.online_system(phi)
    P = sp.csr_matrix((v, (r, q)), shape=(basis.n_rows, basis.n_unknowns))
    c = c.cpu().numpy().ravel()
    assert np.linalg.norm(P.T @ (P @ c - d)) <= 1e-9 * np.linalg.norm(P.T @ d)
