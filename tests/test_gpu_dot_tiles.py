"""Fused dots and the fused setup step with several tiles of 128 sites per CTA, the numbers themselves.

Dots of the level-0 stencil: <out|in> and ||out||^2 of every right-hand side against FP64 sums over the stored
fields, with one and two right-hand sides per thread, partial last tiles, and CTAs that end between two tiles.  A
thread adds 36 products in FP32 and a tile 128 threads in a tree of seven levels, so the error is below 43 x 2^-24
of the sum of the absolute values, 4e-6 with the FP64 sum over tiles; a lost tile changes at least 1 in 1,000.
Both forms add in the same order: the same bits.

Setup step: more tiles than places (k > 1), against the FP64 relaxation's prolongator (FP32 arithmetic over 12
sweeps on a well-conditioned field, 1e-4 as in test_gpu_dslash_tiles.py).
"""
import ctypes

import numpy as np
import pytest

from gpu_util import rel_err, require_gpu, torch
from paper_0811_4331_gb300 import inputs

pytestmark = pytest.mark.gpu
TYPES = {1: torch.float32, 2: torch.float16, 3: torch.bfloat16}


@pytest.mark.parametrize("L,nrhs", [((16, 8, 8, 16), 64), ((12, 10, 6, 14), 48), ((18, 14, 10, 21), 6), ((16, 16, 16, 32), 12)])
@pytest.mark.parametrize("prec", [1, 2, 3])
def test_dots_of_every_right_hand_side(L, nrhs, prec):
    require_gpu()
    import launch_harness as lh
    lib = lh.load()
    V = int(np.prod(L))
    U = torch.from_numpy(inputs.random_gauge_fast(L, 3)).cuda().reshape(4, V, 3, 3).contiguous()
    links = torch.empty(4 * V * 6 * 2, dtype=TYPES[prec], device="cuda")
    assert lib.t_pack_links(prec, lh.ptr(U), lh.ptr(links), V) == 0
    gen = torch.Generator("cuda").manual_seed(V)
    x = torch.randn(nrhs, 12 * V, 2, device="cuda", generator=gen).to(TYPES[prec])
    outs, results = [], []
    for variant in range(lib.t_wilson_variants(prec, nrhs, V)):
        out, result = torch.empty_like(x), torch.zeros(nrhs, 4, dtype=torch.float64, device="cuda")
        partials = torch.full((nrhs * ((V + 31) // 32) * 3,), float("nan"), dtype=torch.float64, device="cuda")
        tickets = torch.zeros(nrhs, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert lib.t_wilson_dots(prec, lh.ptr(x), lh.ptr(out), lh.ptr(links), lh.ints(*L), ctypes.c_double(4.1),
                                 ctypes.c_double(-0.5), nrhs, lh.ptr(partials), lh.ptr(tickets), lh.ptr(result), variant) == 0
        torch.cuda.synchronize()
        assert int(tickets.abs().sum()) == 0
        outs.append(out)
        results.append(result[:, :3])
    assert len(outs) == 2 and torch.equal(outs[0], outs[1]) and torch.equal(results[0], results[1])
    for r in range(nrhs):
        o, i = (torch.view_as_complex(t[r].double()) for t in (outs[0], x))
        want = (o.conj() * i).sum()
        size = float((o.abs() * i.abs()).sum())
        assert abs(complex(results[0][r, 0], results[0][r, 1]) - complex(want)) < 4e-6 * size, r
        n2 = float((o.abs() ** 2).sum())
        assert abs(float(results[0][r, 2]) - n2) < 4e-6 * n2, r


@pytest.mark.parametrize("dims,block,nv", [((8, 8, 8, 16), (4, 4, 4, 4), 20), ((6, 6, 6, 14), (3, 3, 3, 7), 32),
                                           ((12, 8, 8, 12), (4, 4, 4, 4), 24)])
def test_setup_step_over_several_tiles(dims, block, nv):
    wm = require_gpu()
    U = inputs.random_gauge(dims, 5)
    P = []
    for mixed in (0, 1):
        p = wm.mg_default_params(n_levels=2, block=[block], nv=[nv], setup_sweeps=[12], mixed=mixed, seed=3, defer_coarsest=1)
        h = wm.mg_setup(U, dims, 0.2, p)
        P.append(wm.mg_get_prolongator(h, 0))
    assert rel_err(P[1], P[0]) < 1e-4
