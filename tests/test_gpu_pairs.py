"""The FP32 passes in packed pairs (two rows, or two components of a line, per thread).

Every count of components makes another mix of pairs and single components, and the
smallest and odd-shaped grids run the edges of the rules that pick rows per CTA, lines
per CTA and component groups: lines of 1 to 4 threads, blocks of few lines, one row per
CTA.  One step against the FP64 oracle at the FP32 bound of the other parity tests (2e-6:
about 16 roundings of 2^-24 along the transforms, RMS of some 3e-7, with a margin of six
for the smallest grids), and one row per CTA against the built-in shape bitwise (the
packed halves round as the scalar operations, so the shape changes no bit)."""
import numpy as np
import pytest

from gpu_helpers import ensure_lib, mask_layout, psatd_gpu, rel_l2_fields, rounded
from oracle import psatd as orc
from paper_1608_05739_gb300 import capi, synth

pytestmark = pytest.mark.gpu

CASES = [
    ((8, 16), "te", "J"), ((8, 16), "2d6", "rho"), ((16, 32), "tm", "J"), ((48, 96), "te", "rho"),
    ((80, 160), "2d6", "none"), ((80, 192), "te", "J"), ((64, 96), "tm", "none"), ((8, 8, 16), "3d6", "none"),
    ((48, 80, 96), "3d6", "J"), ((16, 8, 160), "3d6", "rho"), ((1024, 32), "te", "none"), ((1024, 16), "2d6", "rho"),
    ((4096, 16), "te", "J"), ((16, 4096), "tm", "J"), ((512, 96), "te", "rho"), ((1280, 16), "te", "J"),
]


@pytest.mark.parametrize("shape,layout,src", CASES)
def test_pairs_match_oracle(shape, layout, src):
    ensure_lib()
    d, dt = (1.0, 0.9, 1.1)[:len(shape)], 0.4
    E = rounded(mask_layout(synth.random_fields(shape, 3, 61), layout, "E"), "fp32")
    B = rounded(mask_layout(synth.random_fields(shape, 3, 62), layout, "B"), "fp32")
    J = rounded(mask_layout(synth.random_fields(shape, 3, 63), layout, "J"), "fp32")
    r0, r1 = (rounded(synth.random_fields(shape, 1, s)[0], "fp32") for s in (64, 65))
    Eo, Bo = orc.psatd_step(E, B, J if src != "none" else None, r0 if src == "rho" else None,
                            r1 if src == "rho" else None, d=d, dt=dt, form=src)
    Eo, Bo = mask_layout(Eo, layout, "E"), mask_layout(Bo, layout, "B")
    plan = capi.Plan(tuple(reversed(shape)), d, dt, layout=layout, prec="fp32", src=src)
    Eg, Bg = psatd_gpu(shape, d, dt, E, B, J, r0, r1, layout=layout, prec="fp32", src=src, plan=plan)
    assert rel_l2_fields(Eg, Bg, Eo, Bo) < 2e-6
    plan.set_launch([0, -1 if len(shape) == 2 else 0, -1 if len(shape) == 2 else 0, 0, -1, -1])
    plan.set_push_groups(1)
    E1, B1 = psatd_gpu(shape, d, dt, E, B, J, r0, r1, layout=layout, prec="fp32", src=src, plan=plan)
    assert np.array_equal(E1, Eg) and np.array_equal(B1, Bg)
    plan.destroy()
