"""FDTD kernels at the edges of their row and plane split: rows of whole 16-byte blocks
and ragged ones, fewer cells than a block, rows and planes that the marching does not
divide, grids large enough that it is used.

A call of several steps subtracts the two half steps between two E updates in one pass;
they are the same two roundings, so it must equal single-step calls bitwise.  The single
step is compared with the FP64 oracle at the bounds of the other FDTD tests (1e-12; 1e-6
from FP32-rounded inputs)."""
import numpy as np
import pytest

from gpu_helpers import fdtd_gpu, mask_layout, rel_l2_fields, rounded
from oracle import fdtd as ofd
from paper_1608_05739_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = [
    ("yee", "te", (2, 2)), ("ckc", "2d6", (3, 5)), ("ckc", "te", (7, 130)), ("yee", "tm", (65, 4)),
    ("ckc", "tm", (1030, 1028)), ("ckc", "te", (1027, 1030)), ("yee", "2d6", (1026, 1024)),
    ("yee", "3d6", (2, 3, 2)), ("yee", "3d6", (5, 7, 132)), ("yee", "3d6", (70, 130, 132)), ("yee", "3d6", (67, 129, 130)),
]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("scheme,layout,shape", CASES)
def test_rows_and_planes(scheme, layout, shape, prec):
    d, dt = (1.0, 0.9, 1.1)[:len(shape)], 0.45
    E = rounded(mask_layout(synth.random_fields(shape, 3, 71), layout, "E"), prec)
    B = rounded(mask_layout(synth.random_fields(shape, 3, 72), layout, "B"), prec)
    J = rounded(mask_layout(synth.random_fields(shape, 3, 73), layout, "J"), prec)
    E1, B1 = fdtd_gpu(shape, d, dt, E, B, J, layout=layout, prec=prec, scheme=scheme)
    Eo, Bo = ofd.fdtd_step(E, B, J, d=d, dt=dt, scheme=scheme)
    tol = 1e-12 if prec == "fp64" else 1e-6
    assert rel_l2_fields(E1, B1, mask_layout(Eo, layout, "E"), mask_layout(Bo, layout, "B")) < tol
    for _ in range(2):
        E1, B1 = fdtd_gpu(shape, d, dt, E1, B1, J, layout=layout, prec=prec, scheme=scheme)
    E3, B3 = fdtd_gpu(shape, d, dt, E, B, J, layout=layout, prec=prec, scheme=scheme, nsteps=3)
    assert np.array_equal(E3, E1) and np.array_equal(B3, B1)
