"""The far-field kernel at the edges of its split: one to several thousand wavevectors
(4, 8 and 16 per CTA, clusters of 1 to 8 CTAs over the rows), windows of fewer rows than
a tile, of one cell, of more cells than the phase table, apodised rows.

Bounds relative to the largest |U|: FP64 1e-12 as in the other far-field test.  FP32
sums of n products in lanes and a tree of 5 levels carry at most (n/32 + 6) 2^-24 sum |F|
<= 2e-6 max|U| for these random windows (|U| ~ sqrt(cells) over the wavevectors)."""
import numpy as np
import pytest

from gpu_helpers import ensure_lib
from oracle import farfield as off
from paper_1608_05739_gb300 import capi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nk,wx,wy,window", [
    (1, 1, 1, "none"), (3, 33, 7, "xy"), (5, 64, 600, "x"), (17, 513, 9, "none"), (33, 1100, 40, "xy"),
    (1300, 70, 130, "x"), (2433, 40, 66, "xy"),
])
def test_split(nk, wx, wy, window, prec):
    import torch
    ensure_lib()
    g = np.random.default_rng(nk)
    nx, ny, d, x0, y0 = wx + 9, wy + 5, (0.5, 0.25), 4, 2
    F = g.standard_normal((ny, nx))
    if prec == "fp32":
        F = F.astype(np.float32).astype(np.float64)
    k = g.uniform(-6.0, 6.0, (nk, 2))
    want = off.fraunhofer(F, d, k, x_range=(x0, x0 + wx), y_range=(y0, y0 + wy), window=window)
    Ft = torch.from_numpy(F).to("cuda", torch.float64 if prec == "fp64" else torch.float32)
    got = capi.farfield((nx, ny), d, Ft, torch.from_numpy(k).to("cuda"), x_range=(x0, x0 + wx), y_range=(y0, y0 + wy),
                        window=window).cpu().numpy()
    assert np.abs(got - want).max() < (1e-12 if prec == "fp64" else 2e-6) * max(np.abs(want).max(), 1e-30)
