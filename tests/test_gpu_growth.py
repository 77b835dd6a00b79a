"""A work space that grows while the call before it, which only enqueued, is still running:
the memory it gives up must not reach another stream's allocations before that call is done.

One patch too large for the on-chip kernel keeps its columns in a scratch buffer that FP64
solves need 48 / 28 as much of as mixed ones; media built at once on another stream take
their coefficients from whatever the pool has free."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
msp = pytest.importorskip("paper_1807_08848_gb300")


def test_scratch_grows_with_work_in_flight():
    N = 160
    big = msp.Medium(synth.lognormal(N, 1 / 16, 32, 3), synth.uniform_patches(N, 1, 1, 0, 8))
    spec, ps = synth.lognormal(512, 1 / 32, 16, 4), synth.uniform_patches(512, 4, 4, 8, 4)
    ref = msp.Medium(spec, ps).coefficients()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    big.sample(1, "mixed", tol=1e-10, max_iter=20000, stream=s1, stats=False)
    big.sample(1, "fp64", tol=1e-10, max_iter=200, stream=s1, stats=False)
    others = [msp.Medium(spec, ps, stream=s2) for _ in range(8)]
    torch.cuda.synchronize()
    for med in others:
        for a, b in zip(med.coefficients(), ref):
            assert torch.equal(a, b)
    # the grown work space holds a whole run
    st = big.sample(1, "fp64", tol=1e-10, max_iter=20000)
    assert st.n_not_converged == 0
