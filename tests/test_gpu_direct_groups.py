"""The direct local solver with enough patches for its wide sweeps (64 columns per CTA, from two
CTAs per SM on) and for two groups of patches on two streams (from four per SM on): rows of
one to five groups of 32 nodes; a CTA whose second chunk holds one column, a full one, a chunk
left over and a CTA with one chunk.  Patches at the ends and on both sides of the split
against the oracle's sparse solves, to 1e-9 as in test_gpu_direct_shapes.py (whose two patches
stay below both lines); the first patch against the same patch of a 2 x 2 medium, which takes
the narrow sweeps, bit for bit; replayed from a graph, and with phase timing, which runs the
groups one after the other, the snapshots are the same bits."""
import numpy as np
import pytest
import torch

import synth
from oracle import elliptic as E

pytestmark = pytest.mark.gpu
msp = pytest.importorskip("paper_1807_08848_gb300")


def medium(m, width, buffer, samples):
    n = m * width
    ms, ps = synth.hou_wu(n, 1 / 6), synth.uniform_patches(n, m, m, buffer, samples)
    med = msp.Medium(ms, ps)
    med.set_launch("mixed", "direct")
    return med, ms, ps, n


@pytest.mark.parametrize("m,width,buffer,samples", [(26, 8, 2, 33), (26, 8, 2, 64), (26, 8, 2, 65), (26, 8, 2, 20),
                                                    (26, 24, 8, 33), (26, 24, 8, 65), (26, 48, 20, 33), (18, 64, 24, 40)])
def test_wide_and_grouped(m, width, buffer, samples):
    med, ms, ps, n = medium(m, width, buffer, samples)
    st = med.sample(17, "mixed", tol=1e-12, max_iter=20000)
    assert st.n_not_converged == 0
    aE, aN = E.face_coefficients(ms)
    boxes = E.patch_boxes(n, ps)
    cols = np.cumsum([med.patch(q).cols for q in range(m * m)])
    half = int(np.searchsorted(cols, cols[-1] / 2))
    for q in sorted({0, half - 1, half, half + 1, half + 2, m * m - 1}):
        R = E.snapshots(aE, aN, boxes[q], 17, n)
        d = med.snapshots(q).cpu().numpy() - R
        assert np.linalg.norm(d) <= 1e-9 * np.linalg.norm(R), q


@pytest.mark.parametrize("m,width,buffer,samples", [(26, 8, 2, 33), (26, 24, 8, 64), (18, 48, 20, 65), (18, 64, 24, 40),
                                                    (18, 100, 28, 33)])
def test_same_bits_as_the_narrow_sweeps(m, width, buffer, samples):
    n, k = m * width, 2 * width
    rng = np.random.Generator(np.random.PCG64(3))
    aE, aN = np.exp(0.5 * rng.standard_normal((n + 1, n))), np.exp(0.5 * rng.standard_normal((n, n + 1)))
    out = []
    for size, parts, e, v in ((n, m, aE, aN), (k, 2, aE[:k + 1, :k], aN[:k, :k + 1])):
        med = msp.Medium(synth.user_medium(e, v), synth.uniform_patches(size, parts, parts, buffer, samples))
        med.set_launch("mixed", "direct")
        assert med.sample(23, "mixed", tol=1e-12, max_iter=20000).n_not_converged == 0
        out.append(med.snapshots(0))
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("samples", [33, 64])
def test_graph_and_timing(samples):
    med, _, _, _ = medium(26, 8, 2, samples)
    med.sample(17, "mixed", tol=1e-12, max_iter=20000)
    ref = [med.snapshots(q).clone() for q in range(0, 26 * 26, 25)]

    def same():
        return all(torch.equal(med.snapshots(q), r) for q, r in zip(range(0, 26 * 26, 25), ref))

    med.set_graph(True)
    for seed in (17, 18, 17, 17):      # captured, captured for another seed, captured again, replayed
        med.sample(seed, "mixed", tol=1e-12, max_iter=20000)
    assert same()
    med.set_graph(False)
    med.set_timing(True)
    med.sample(17, "mixed", tol=1e-12, max_iter=20000)
    assert same() and med.direct_timing()["solve"]["ms"] > 0
