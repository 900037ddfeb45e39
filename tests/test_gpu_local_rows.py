"""The local decomposition's x passes on the global grid: guard rows and columns read in
place, interiors written in place.  Odd guards (pairs of cells not aligned), one patch,
guards wider than a patch and than the whole grid (rows that wrap several times), every
precision; against the local oracle at each precision's one-step bound (1e-12, 2e-6, 4e-6),
several steps in one call against single-step calls and a checked plan against an
unchecked one, bitwise."""
import numpy as np
import pytest

from gpu_helpers import ensure_lib, mask_layout, rel_l2_fields, rounded, torch_dev
from oracle import local as ol
from paper_1608_05739_gb300 import capi, synth

pytestmark = pytest.mark.gpu

CASES = [  # interior (ix, iy), patches (px, py), guard
    ("fp32", (30, 30), (2, 3), 1), ("fp32", (26, 42), (1, 1), 3), ("fp32", (6, 6), (2, 2), 5), ("fp32", (2, 2), (1, 1), 7),
    ("fp32", (80, 32), (3, 2), 8), ("fp32", (64, 64), (2, 2), 0), ("fp64", (26, 58), (2, 2), 3), ("fp64", (48, 48), (2, 3), 8),
    ("mixed_fp16", (118, 22), (2, 2), 5), ("mixed_bf16", (112, 48), (2, 2), 8),
]


@pytest.mark.parametrize("order", [0, 8])
@pytest.mark.parametrize("prec,inner,patches,guard", CASES)
def test_global_rows(prec, inner, patches, guard, order):
    ensure_lib()
    (ix, iy), (px, py) = inner, patches
    shape, d, dt, layout = (py * iy, px * ix), (1.0, 0.9), 0.4, "te"
    E = rounded(mask_layout(synth.random_fields(shape, 3, 91), layout, "E"), prec)
    B = rounded(mask_layout(synth.random_fields(shape, 3, 92), layout, "B"), prec)
    J = rounded(mask_layout(synth.random_fields(shape, 3, 93), layout, "J"), prec)

    def run(nsteps, calls):
        loc = capi.Local((px * ix, py * iy), d, dt, px=px, py=py, guard=guard, layout=layout, prec=prec, src="J",
                         order=order)
        t = [torch_dev(a, prec) for a in (E[0], E[1], B[2], J[0], J[1])]
        for _ in range(calls):
            loc.step([t[0], t[1], None], [None, None, t[2]], [t[3], t[4], None], nsteps=nsteps)
        loc.sync()
        Eg, Bg = np.zeros((3,) + shape), np.zeros((3,) + shape)
        Eg[0], Eg[1], Bg[2] = (a.double().cpu().numpy() for a in t[:3])
        assert np.array_equal(t[3].double().cpu().numpy(), J[0])   # the sources are read only
        loc.destroy()
        return Eg, Bg

    Eg, Bg = run(1, 1)
    Eo, Bo = ol.local_step(E, B, J, d=d, dt=dt, px=px, py=py, guard=guard, form="J", order=order)
    tol = {"fp64": 1e-12, "fp32": 2e-6}.get(prec, 4e-6)
    assert rel_l2_fields(Eg, Bg, mask_layout(Eo, layout, "E"), mask_layout(Bo, layout, "B")) < tol
    a, b = run(3, 1), run(1, 3)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("pinned", [False, True])
def test_sources_are_held_over_the_call(pinned):
    """Three steps of one call with J in a field's own array, on the device or pinned on the host,
    equal three steps with J in an array of its own: sources are those of the call's start."""
    import torch
    ensure_lib()
    shape, d, dt = (96, 96), (1.0, 0.9), 0.4
    F = [synth.random_fields(shape, 1, s)[0] for s in (95, 96, 97)]

    def run(alias):
        t = [torch.from_numpy(a).float() for a in F]
        t = [a.pin_memory() if pinned else a.cuda() for a in t]
        own = t[0].clone()
        J0 = t[0] if alias else own.pin_memory() if pinned else own
        loc = capi.Local((96, 96), d, dt, px=2, py=2, guard=8, layout="te", prec="fp32", src="J")
        loc.step([t[0], t[1], None], [None, None, t[2]], [J0, torch.zeros_like(t[1], device="cuda"), None], nsteps=3)
        loc.sync()
        loc.destroy()
        return [a.cpu().numpy() for a in t]

    for a, b in zip(run(True), run(False)):
        assert np.array_equal(a, b)
