"""The FP32 streaming operator over the strip layouts its tile shapes select (1 to 8 rows a
strip, and tiles too wide for strips), with rows and pitch beyond the boxes and uneven
counts of samples, against the same operator in FP64.

Tolerance: faces and data rounded to FP32 and a five-term sum, 1e-5 of the largest term
(the bound of the operator's other tests)."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
msp = pytest.importorskip("paper_1807_08848_gb300")

# (cells, patches per side, buffer, rows beyond, columns of pitch beyond, samples)
SHAPES = [(24, 2, 2, 0, 0, 1), (64, 2, 4, 1, 4, 7), (96, 2, 6, 0, 8, 3), (128, 2, 9, 0, 0, 5), (160, 2, 12, 3, 0, 2),
          (170, 2, 14, 0, 4, 9), (24, 2, 2, 0, 640, 3), (20, 2, 1, 700, 0, 3)]


@pytest.mark.parametrize("N,m,buffer,more_rows,more_cols,S", SHAPES)
def test_strip_layouts(N, m, buffer, more_rows, more_cols, S):
    ps = synth.uniform_patches(N, m, m, buffer, 4)
    med = msp.Medium(synth.lognormal(N, 4.0 / N, 16, 3), ps)
    rows, cols = med.tile_shape()
    H, P = rows + more_rows, (cols + 3) // 4 * 4 + more_cols
    g = torch.Generator(device="cpu").manual_seed(1)
    x = torch.randn((med.n_patches, S, H, P), generator=g, dtype=torch.float64).cuda()
    y = med.apply_operator(x.float(), "mixed", y=torch.full((med.n_patches, S, H, P), 7.0, device="cuda")).double()
    aE, aN = med.coefficients()
    top = float(max(aE.max(), aN.max())) * float(x.abs().max()) * 8
    for k in range(med.n_patches):
        p = med.patch(k)
        h, w = p.Y1 - p.Y0 + 1, p.X1 - p.X0 + 1
        t = x[k, :, :h, :w].float().double()
        e, n = aE[p.Y0:p.Y1 + 1, p.X0:p.X1], aN[p.Y0:p.Y1, p.X0:p.X1 + 1]
        ref = torch.zeros((S, H, P), dtype=torch.float64, device="cuda")
        c = t[:, 1:-1, 1:-1]
        ref[:, 1:h - 1, 1:w - 1] = (e[1:-1, 1:] * (c - t[:, 1:-1, 2:]) + e[1:-1, :-1] * (c - t[:, 1:-1, :-2]) +
                                    n[1:, 1:-1] * (c - t[:, 2:, 1:-1]) + n[:-1, 1:-1] * (c - t[:, :-2, 1:-1]))
        assert float((y[k] - ref).abs().max()) <= 1e-5 * top, k
        inside = torch.zeros((H, P), dtype=torch.bool, device="cuda")
        inside[1:h - 1, 1:w - 1] = True
        assert bool((y[k][:, ~inside] == 0).all()), k
