"""The direct kinetic solver beyond 65535 patches and beyond 65535 chunks of 16 samples, the
end of a grid's second dimension, against the CPU oracle's solves of single patches (1e-9
relative, the bound of the refined snapshots in test_gpu_kinetic_shapes.py)."""
import numpy as np
import pytest

from oracle import kinetic as K

pytestmark = pytest.mark.gpu
msp = pytest.importorskip("paper_1807_08848_gb300")


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_many_patches(precision):
    n, n_v, buffer, eps, g = 65537, 2, 1, 1.0, 0.2
    km = msp.KineticMedium(n_cells=n, eps=eps, n_v=n_v, n_patches=n, buffer=buffer, samples=1, g=g)
    st = km.sample(5, tol=1e-13, max_iter=16, precision=precision)
    assert st.n_not_converged == 0
    for m in (0, 1, 65534, 65535, 65536):
        p = K.KPatch(m, m, m + 1, max(0, m - buffer), min(n, m + 1 + buffer), 1)
        R = K.snapshots(n, eps, n_v, p, 5, g)
        assert np.linalg.norm(km.snapshots(m).cpu().numpy() - R) <= 1e-9 * np.linalg.norm(R), m


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_many_samples(precision):
    n, n_v, samples, eps, g = 4, 2, 16 * 65535 + 1, 1.0, 0.2
    km = msp.KineticMedium(n_cells=n, eps=eps, n_v=n_v, n_patches=1, buffer=0, samples=samples, g=g)
    st = km.sample(6, tol=1e-13, max_iter=16, precision=precision)
    assert st.n_not_converged == 0
    R = K.snapshots(n, eps, n_v, K.KPatch(0, 0, n, 0, n, samples), 6, g)
    got = km.snapshots(0).cpu().numpy()
    scale = np.linalg.norm(R) / np.sqrt(samples)
    assert np.max(np.linalg.norm(got - R, axis=0)) <= 1e-9 * scale
