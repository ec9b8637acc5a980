"""Public calls captured into a CUDA graph by the caller give the bits of the same calls made eagerly.

Captured launches may start early, as eager ones may (see launch_chain): chains of stencils, smoothing steps, even-odd
operators, transfers and FP64 cycles, replayed several times back to back.
"""
import pytest

from gpu_util import require_gpu, torch
from paper_0811_4331_gb300 import inputs

pytestmark = pytest.mark.gpu


def _fill(t, seed):
    v = torch.view_as_real(t) if t.is_complex() else t
    v.copy_(torch.randn(v.shape, device="cuda", generator=torch.Generator("cuda").manual_seed(seed)).to(v.dtype))
    return t


def _bits(ts):
    return [(torch.view_as_real(t) if t.is_complex() else t).clone() for t in ts]


def _check(calls, outputs):
    for _ in range(2):
        calls()
    torch.cuda.synchronize()
    want = _bits(outputs)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        calls()
    for t in outputs:
        t.zero_()
    for _ in range(5):
        g.replay()
    torch.cuda.synchronize()
    for a, b in zip(want, _bits(outputs)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
def test_fine_operators(prec):
    wm = require_gpu()
    dims = (8, 6, 8, 12)
    kw = {} if prec == 0 else dict(mixed=1, fine_prec=prec)
    h = wm.mg_setup(inputs.random_gauge(dims, 3), dims, 0.1, wm.mg_default_params(n_levels=1, **kw))
    a, b, c, x, r = (wm.internal_empty(h, 0, prec) for _ in range(5))
    e, o, s = (wm.internal_empty(h, 0, prec, half=True) for _ in range(3))
    _fill(a, 1)

    def calls():
        x.zero_()
        wm.dslash_apply(h, prec, a, b)
        wm.dslash_apply(h, prec, b, c)
        wm.mr_apply(h, 0, prec, c, x, r, 3)
        wm.eo_split(h, prec, r, e, o)
        wm.schur_apply(h, prec, e, s)
        wm.eo_merge(h, prec, s, o, b)

    _check(calls, [b, c, x, r, s])


@pytest.mark.parametrize("prec,nrhs", [(0, 1), (1, 3), (2, 1), (2, 20), (3, 9)])
def test_transfers_and_coarse_operators(prec, nrhs):
    wm = require_gpu()
    dims = (8, 8, 8, 16)
    kw = {} if prec == 0 else dict(mixed=1, fine_prec=prec, coarse_mma=1)
    p = wm.mg_default_params(n_levels=3, block=[(4, 4, 4, 4), (2, 2, 2, 2)], nv=[12, 4], setup_sweeps=[3, 2], **kw)
    h = wm.mg_setup(inputs.random_gauge(dims, 3), dims, 0.1, p)
    pc = 0 if prec == 0 else 1
    f, g = (wm.internal_empty(h, 0, prec, nrhs) for _ in range(2))
    c, d = (wm.internal_empty(h, 1, pc, nrhs) for _ in range(2))
    _fill(f, 2)
    outputs = [g, c, d]
    if prec == 0:
        e = wm.internal_empty(h, 0, prec)
        outputs.append(e)

    def calls():
        wm.restrict_apply(h, 0, prec, f, c, nrhs)
        wm.coarse_apply(h, 1, pc, c, d, nrhs)
        wm.prolong_apply(h, 0, prec, d, g, nrhs)
        if prec == 0:
            wm.vcycle_apply(h, g[:1], e)

    _check(calls, outputs)
