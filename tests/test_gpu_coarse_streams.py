"""coarse_apply on one handle from several streams and inside captured graphs.

The tensor-core form rounds four and more right-hand sides to BF16 rows in a buffer first.  Calls on different
streams have their own, so overlapping calls give the bits of the same calls one after the other; so has each capture,
and its graph replays correctly after larger calls and beside others.  Streams and captures beyond the handle's
buffers gather the vectors instead.
"""
import numpy as np
import pytest

from gpu_util import require_gpu, torch
from paper_0811_4331_gb300 import inputs

pytestmark = pytest.mark.gpu


def _setup(wm, dims=(8, 8, 8, 16), nv=24):
    p = wm.mg_default_params(n_levels=3, block=[(2, 2, 2, 2), (2, 2, 2, 2)], nv=[nv, 2], setup_sweeps=[2, 1], mixed=1,
                             coarse_mma=1)
    return wm.mg_setup(inputs.random_gauge_fast(dims, 6), dims, -0.1, p)


def _field(wm, h, nrhs, seed):
    t = wm.internal_empty(h, 1, wm.MG_F32, nrhs)
    t.copy_(torch.randn(t.shape, dtype=t.dtype, device="cuda", generator=torch.Generator("cuda").manual_seed(seed)))
    return t


def _same(a, b):
    return torch.equal(torch.view_as_real(a), torch.view_as_real(b))


@pytest.mark.parametrize("streams", [2, 11])
def test_overlapping_calls_equal_serial_ones(streams):
    wm = require_gpu()
    h = _setup(wm)
    counts = [24, 8, 12, 5][: min(streams, 4)] * 3
    ins = [_field(wm, h, counts[i], i) for i in range(streams)]
    want = []
    for x in ins:
        o = torch.empty_like(x)
        wm.coarse_apply(h, 1, wm.MG_F32, x, o, x.shape[0])
        want.append(o)
    torch.cuda.synchronize()
    qs = [torch.cuda.Stream() for _ in range(streams)]
    for rep in range(20):
        outs = [torch.zeros_like(x) for x in ins]
        torch.cuda.synchronize()
        for _ in range(3):
            for q, x, o in zip(qs, ins, outs):
                wm.coarse_apply(h, 1, wm.MG_F32, x, o, x.shape[0], stream=q)
        torch.cuda.synchronize()
        assert all(_same(o, w) for o, w in zip(outs, want)), rep
    held = wm.mg_handle_bytes(h)
    assert wm.mg_release_work(h) > 0 and wm.mg_handle_bytes(h) < held


def test_captured_call_replays_after_larger_calls_and_beside_others():
    wm = require_gpu()
    h = _setup(wm)
    x, big = _field(wm, h, 6, 1), _field(wm, h, 64, 2)
    want, wbig, out, obig, oall = (torch.empty_like(t) for t in (x, big, x, big, big))
    wm.coarse_apply(h, 1, wm.MG_F32, x, want, 6)
    wm.coarse_apply(h, 1, wm.MG_F32, big, wbig, 64)
    wm.mg_release_work(h)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        wm.coarse_apply(h, 1, wm.MG_F32, x, out, 6)
        wm.coarse_apply(h, 1, wm.MG_F32, big, oall, 64)  # more than the capture's first buffer holds
        wm.coarse_apply(h, 1, wm.MG_F32, x, out, 6)
    q = torch.cuda.Stream()
    for rep in range(20):
        out.zero_()
        obig.zero_()
        torch.cuda.synchronize()
        wm.coarse_apply(h, 1, wm.MG_F32, big, obig, 64, stream=q)
        g.replay()
        wm.coarse_apply(h, 1, wm.MG_F32, big, obig, 64, stream=q)
        torch.cuda.synchronize()
        assert _same(out, want) and _same(obig, wbig) and _same(oall, wbig), rep
    wm.mg_release_work(h)
    out.zero_()
    wm.coarse_apply(h, 1, wm.MG_F32, big, obig, 64)
    g.replay()
    torch.cuda.synchronize()
    assert _same(out, want)


def test_more_captures_than_buffers():
    wm = require_gpu()
    h = _setup(wm)
    x = _field(wm, h, 12, 1)
    want = torch.empty_like(x)
    wm.coarse_apply(h, 1, wm.MG_F32, x, want, 12)
    outs, graphs = [torch.zeros_like(x) for _ in range(20)], []
    torch.cuda.synchronize()
    for o in outs:
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[-1]):
            wm.coarse_apply(h, 1, wm.MG_F32, x, o, 12)
    for g in graphs:
        g.replay()
    torch.cuda.synchronize()
    assert all(_same(o, want) for o in outs)


def test_capture_of_sizes_never_run_before():
    wm = require_gpu()
    h = _setup(wm, dims=(4, 4, 4, 8), nv=13)
    x = _field(wm, h, 9, 3)
    out, want = torch.empty_like(x), torch.empty_like(x)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        wm.coarse_apply(h, 1, wm.MG_F32, x, out, 9)
    g.replay()
    wm.coarse_apply(h, 1, wm.MG_F32, x, want, 9)
    torch.cuda.synchronize()
    assert _same(out, want) and bool(np.isfinite(torch.view_as_real(out).cpu().numpy()).all())
