"""Edges of the direct local solver's tiles against the oracle's sparse solves: interior
row widths around the factor's 16-wide thread grid, the sweeps' 32-row groups (one to
five of them) and the widest row taken, each with column counts around the 32- and
64-column CTAs, and two patches so that both patch groups hold work.

Tolerance: 1e-9 relative, as for the other refined solves of the direct solver at a
residual of 1e-12 on media of this contrast.
"""
import numpy as np
import pytest

import synth
from oracle import elliptic as E

pytestmark = pytest.mark.gpu
msp = pytest.importorskip("paper_1807_08848_gb300")


@pytest.mark.parametrize("width,samples", [
    (2, 5), (15, 31), (16, 32), (17, 33), (31, 64), (32, 65), (33, 1), (48, 97), (63, 40), (64, 64), (65, 70),
    (95, 33), (96, 64), (97, 20), (127, 65), (128, 32), (129, 40), (143, 33), (145, 64), (160, 66)])
def test_row_widths(width, samples):
    n = width + 9   # interior widths of the two patches: `width` and 13
    ps = synth.PatchSpec(np.array([0, width - 2, n]) if width > 2 else np.array([0, 1, n]), np.array([0, n]),
                         np.array([3, 3]) if width > 2 else np.array([2, 1]), np.array([samples, 9]))
    ms = synth.hou_wu(n, 1 / 6)
    med = msp.Medium(ms, ps)
    med.set_launch("mixed", "direct")
    st = med.sample(17, "mixed", tol=1e-12, max_iter=20000)
    assert st.n_not_converged == 0
    aE, aN = E.face_coefficients(ms)
    boxes = E.patch_boxes(n, ps)
    assert boxes[0].X1 - boxes[0].X0 - 1 == width
    for m, p in enumerate(boxes):
        R = E.snapshots(aE, aN, p, 17, n)
        d = med.snapshots(m).cpu().numpy() - R
        assert np.linalg.norm(d) <= 1e-9 * np.linalg.norm(R), m
