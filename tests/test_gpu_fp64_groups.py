"""FP64 passes at the edges of their split: lines of one thread to many, single lines per
block in component groups that are not whole warps (2, 3 or 6 groups by component count),
blocks of several lines, the longest lines.  One step against the FP64 oracle at the FP64
bound (1e-12), and the built-in shape against one group and one line per CTA, bitwise (the
split changes no operation)."""
import numpy as np
import pytest

from gpu_helpers import ensure_lib, mask_layout, psatd_gpu, rel_l2_fields
from oracle import psatd as orc
from paper_1608_05739_gb300 import capi, synth

pytestmark = pytest.mark.gpu

CASES = [
    ((8, 16), "te", "J"), ((16, 32), "2d6", "rho"), ((32, 64), "tm", "none"), ((128, 128), "2d6", "none"),
    ((64, 256), "te", "rho"), ((128, 1024), "te", "J"), ((8, 8, 16), "3d6", "J"), ((16, 64, 32), "3d6", "rho"),
    ((16, 4096), "tm", "J"), ((2048, 32), "te", "none"),
    ((64, 256), "2d6", "rho"),  # 129 blocks: the six components whole
    ((128, 64, 128), "3d6", "none"),  # radix-8 stages in the last axis
    ((64, 128, 256), "3d6", "none"), ((16, 256, 512), "3d6", "none"),  # rows of 128 and 256 points by 16 elements
]


@pytest.mark.parametrize("shape,layout,src", CASES)
def test_fp64_split(shape, layout, src):
    ensure_lib()
    d, dt = (1.0, 0.9, 1.1)[:len(shape)], 0.4
    E = mask_layout(synth.random_fields(shape, 3, 81), layout, "E")
    B = mask_layout(synth.random_fields(shape, 3, 82), layout, "B")
    J = mask_layout(synth.random_fields(shape, 3, 83), layout, "J")
    r0, r1 = (synth.random_fields(shape, 1, s)[0] for s in (84, 85))
    Eo, Bo = orc.psatd_step(E, B, J if src != "none" else None, r0 if src == "rho" else None,
                            r1 if src == "rho" else None, d=d, dt=dt, form=src)
    plan = capi.Plan(tuple(reversed(shape)), d, dt, layout=layout, prec="fp64", src=src)
    Eg, Bg = psatd_gpu(shape, d, dt, E, B, J, r0, r1, layout=layout, prec="fp64", src=src, plan=plan)
    assert rel_l2_fields(Eg, Bg, mask_layout(Eo, layout, "E"), mask_layout(Bo, layout, "B")) < 1e-12
    plan.set_launch([0, -1 if len(shape) == 2 else 0, -1 if len(shape) == 2 else 0, 0, 1, -1])
    plan.set_push_groups(1)
    E1, B1 = psatd_gpu(shape, d, dt, E, B, J, r0, r1, layout=layout, prec="fp64", src=src, plan=plan)
    assert np.array_equal(E1, Eg) and np.array_equal(B1, Bg)
    plan.destroy()


def test_six_components_as_two_sets_equal_the_whole():
    """65 lines of a 128 x 128 plan run as the TE and TM sets, three patches' 195 lines with the six
    components in a block: the same operations, the same bits."""
    import torch
    ensure_lib()
    shape, d, dt, n = (128, 128), (1.0, 0.9), 0.4, 3
    E, B, J = (synth.random_fields(shape, 3, s) for s in (91, 92, 93))
    r0, r1 = (synth.random_fields(shape, 1, s)[0] for s in (94, 95))
    one = psatd_gpu(shape, d, dt, E, B, J, r0, r1, layout="2d6", prec="fp64", src="rho")
    rep = lambda a: torch.from_numpy(np.concatenate([a.ravel()] * n)).cuda()
    Et, Bt, Jt = ([rep(a) for a in f] for f in (E, B, J))
    batch = capi.Batch([(128, 128)] * n, d, dt, layout="2d6", prec="fp64", src="rho")
    batch.step(Et, Bt, Jt, rep(r0), rep(r1))
    torch.cuda.synchronize()
    for got, want in zip(Et + Bt, list(one[0]) + list(one[1])):
        for p in got.cpu().numpy().reshape(n, *shape):
            assert np.array_equal(p, want)
    batch.destroy()
