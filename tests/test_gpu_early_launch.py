"""Passes launched early (while their predecessor in the stream drains): steps of two
plans of different sizes taken in turn on one stream, beside FDTD steps on the same
arrays and torch operations between them, must give the bits of the same sequence with a
synchronisation after every call; and steps captured into a CUDA graph by the caller must
replay to the bits of direct calls."""
import pytest

from gpu_helpers import ensure_lib
from paper_1608_05739_gb300 import capi

pytestmark = pytest.mark.gpu


def _arrays(n, seed):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn(tuple(reversed(n)), device="cuda", generator=g) for _ in range(5)]


def _step(p, a, **kw):
    p.step([a[0], a[1], None], [None, None, a[2]], [a[3], a[4], None], **kw)


def test_interleaved_calls_match_synchronised_ones():
    import torch
    ensure_lib()
    sizes = [(64, 64), (512, 256), (96, 48)]
    out = []
    for wait in (False, True):
        plans = [capi.Plan(n, (1.0, 1.0), 0.5, layout="te", prec="fp32", src="J") for n in sizes]
        arr = [_arrays(n, i) for i, n in enumerate(sizes)]
        for _ in range(20):
            for n, p, a in zip(sizes, plans, arr):
                _step(p, a)
                if wait:
                    torch.cuda.synchronize()
                a[3].mul_(0.99)
                capi.fdtd_step(n, (1.0, 1.0), 0.3, [a[0], a[1], None], [None, None, a[2]], [a[3], a[4], None],
                               scheme="yee", layout="te", nsteps=2)
                if wait:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        out.append(arr)
        for p in plans:
            p.destroy()
    for x, y in zip(*out):
        assert all(torch.equal(u, v) for u, v in zip(x, y))


@pytest.mark.parametrize("n", [(64, 64), (512, 512), (2048, 1024)])
def test_captured_steps_match_direct_ones(n):
    import torch
    ensure_lib()
    st = torch.cuda.Stream()
    p = capi.Plan(n, (1.0, 1.0), 0.5, layout="te", prec="fp32", src="J", stream=st)
    a = _arrays(n, 7)
    b = [x.clone() for x in a]
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        for _ in range(7):
            _step(p, a)
        _step(p, b)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        _step(p, b, nsteps=2)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(a, b))
    p.destroy()
