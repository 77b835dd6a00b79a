"""Memory that the library's pool keeps between calls goes back to the device on request."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
msp = pytest.importorskip("paper_1807_08848_gb300")


def test_trim_gives_the_pool_back():
    spec, ps = synth.lognormal(1024, 1 / 32, 16, 3), synth.uniform_patches(1024, 16, 16, 8, 64)
    msp.trim_memory()
    free0 = torch.cuda.mem_get_info()[0]
    med = msp.Medium(spec, ps)
    held = 8 * med.snapshot_elems
    aE = med.coefficients()[0].cpu()
    kept = msp.Medium(synth.lognormal(64, 1 / 8, 16, 3), synth.uniform_patches(64, 2, 2, 4, 8))
    small = kept.coefficients()[0].cpu()
    del med
    assert free0 - torch.cuda.mem_get_info()[0] >= held      # the pool keeps the dropped medium's buffers
    msp.trim_memory(1 << 40)                                 # more than it holds: nothing goes
    assert free0 - torch.cuda.mem_get_info()[0] >= held
    msp.trim_memory()
    torch.cuda.empty_cache()
    assert free0 - torch.cuda.mem_get_info()[0] <= held // 4
    assert torch.equal(kept.coefficients()[0].cpu(), small)  # live handles are untouched
    assert torch.equal(msp.Medium(spec, ps).coefficients()[0].cpu(), aE)


def test_negative_size_is_refused():
    with pytest.raises(msp.MspError) as e:
        msp.trim_memory(-1)
    assert e.value.status == -1
