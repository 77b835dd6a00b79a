"""Slabs on both sides of the lines between the online stage's forms: one launch per solve or
one per phase (64 columns over the patches), and the factor's chain on one CTA or a cluster
(8 columns), against the CPU oracle's global solve (1e-8, full local spaces, as in
test_gpu_kinetic_shapes.py); a batch gives each data set the bits of the set alone."""
import numpy as np
import pytest
import torch

from oracle import kinetic as K

pytestmark = pytest.mark.gpu
msp = pytest.importorskip("paper_1807_08848_gb300")


@pytest.mark.parametrize("n_v,patches,cells", [(2, 1, 4), (2, 32, 4), (2, 33, 4), (4, 16, 6), (4, 17, 6), (6, 3, 8), (8, 8, 6),
                                               (8, 9, 6), (8, 4, 512), (64, 1, 12), (66, 1, 12)])
def test_forms(n_v, patches, cells):
    n, eps, g = patches * cells, 1.0, 0.4
    km = msp.KineticMedium(n_cells=n, eps=eps, n_v=n_v, n_patches=patches, buffer=2, samples=n_v + 4, g=g)
    assert km.sample(9, tol=1e-13, max_iter=16, precision="fp64").n_not_converged == 0
    kb = km.extract(1e-12)
    v, _ = K.velocities(n_v)
    data = np.stack([[1 + 0.5 * np.sin(np.pi * v), 0.5 + v ** 2], [v, 1 - v], [v * v, v]])
    f = kb.solve(torch.tensor(data, device="cuda"))
    for b in range(3):
        ref = K.global_reference(n, eps, n_v, data[b][0], data[b][1], g)
        assert np.linalg.norm(f[b].cpu().numpy() - ref) <= 1e-8 * np.linalg.norm(ref), b
        assert torch.equal(kb.solve(torch.tensor(data[b:b + 1], device="cuda"))[0], f[b]), b
