"""Edges of the kinetic kernels against the CPU oracle: velocity halves around the
16-wide thread grid and its register blocks, sample counts around the 16 lanes of a
half-warp, slabs of one to three patches (first and last node in one patch, a chain of
one block), and patch spaces on both sides of the width at which the online chain
leaves the cluster's shared memory (170 basis columns).

Tolerances: the refined snapshots 1e-9 relative, the stop being a scaled residual of
1e-13 on an operator whose inverse is bounded by about 1e3 at these sizes; full local
spaces reproduce the global solve within 1e-8.
"""
import numpy as np
import pytest
import torch

from oracle import kinetic as K

pytestmark = pytest.mark.gpu
msp = pytest.importorskip("paper_1807_08848_gb300")


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n_v,samples", [(2, 1), (4, 15), (30, 16), (32, 17), (34, 33), (62, 1), (64, 40), (66, 16), (128, 7)])
def test_local_solver(n_v, samples, precision):
    n, patches, buffer, g, eps = 18, 3, 2, 0.3, 1 / 8
    km = msp.KineticMedium(n_cells=n, eps=eps, n_v=n_v, n_patches=patches, buffer=buffer, samples=samples, g=g)
    st = km.sample(5, tol=1e-13, max_iter=16, precision=precision)
    assert st.n_not_converged == 0
    for m, p in enumerate(K.patches(n, patches, buffer, samples)):
        assert rel(km.snapshots(m).cpu().numpy(), K.snapshots(n, eps, n_v, p, 5, g)) <= 1e-9, m


@pytest.mark.parametrize("n_v,patches", [(2, 1), (2, 3), (34, 1), (34, 2), (128, 3), (170, 1), (170, 3)])
def test_online_chain(n_v, patches):
    g = 0.4 if n_v <= 128 else 0.0
    n, eps = 12 * patches, 1.0
    km = msp.KineticMedium(n_cells=n, eps=eps, n_v=n_v, n_patches=patches, buffer=2, samples=n_v + 4, g=g)
    st = km.sample(9, tol=1e-13, max_iter=16 if g else 20000, precision="fp64")
    assert st.n_not_converged == 0
    kb = km.extract(1e-12)
    v, _ = K.velocities(n_v)
    data = np.stack([[1 + 0.5 * np.sin(np.pi * v), 0.5 + v ** 2], [v, 1 - v]])
    f = kb.solve(torch.tensor(data, device="cuda")).cpu().numpy()
    for b in range(2):
        assert rel(f[b], K.global_reference(n, eps, n_v, data[b][0], data[b][1], g)) <= 1e-8, b
