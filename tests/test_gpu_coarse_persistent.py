"""The streaming coarse stencil where a CTA takes several items: more sites (times groups of right-hand sides) than the
launch has CTAs, so the ring's slot and parity, and the copies already under way, are carried from one item into the
next.

The sums of one right-hand side have the same order in the form that gathers its vectors itself, which runs for a
right-hand side alone: the same bits.  That form against the FP64 stencil: both operands rounded to BF16 (2^-8
relative each, on sums of 9 n random-sign terms), 2e-2.
"""
import numpy as np
import pytest

from gpu_util import rel_err, require_gpu, torch
from oracle import dirac
from paper_0811_4331_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nv,counts", [((16, 16, 16, 8), 24, (4, 9, 24, 64)), ((16, 16, 16, 16), 9, (5, 24)),
                                            ((18, 14, 10, 12), 20, (12, 33))])
def test_items_of_one_cta_match_right_hand_sides_alone(dims, nv, counts):
    wm = require_gpu()
    lc = [d // 2 for d in dims]
    p = wm.mg_default_params(n_levels=3, block=[(2, 2, 2, 2), tuple(2 if e % 2 == 0 else 1 for e in lc)], nv=[nv, 2],
                             setup_sweeps=[2, 1], mixed=1, coarse_mma=1, defer_coarsest=1)
    h = wm.mg_setup(inputs.random_gauge_fast(dims, 6), dims, -0.1, p)
    ld, nc, _ = wm.mg_level_info(h, 1)
    lat = (ld[3], ld[2], ld[1], ld[0])
    most = max(counts)
    gen = torch.Generator("cuda").manual_seed(nv)
    yi = wm.internal_empty(h, 1, wm.MG_F32, most)
    yi.copy_(torch.randn(yi.shape, dtype=yi.dtype, device="cuda", generator=gen))
    alone = torch.empty_like(yi)
    for r in range(most):
        wm.coarse_apply(h, 1, wm.MG_F32, yi[r:r + 1].contiguous(), alone[r:r + 1], 1)
    old = wm.mg_tune(0)
    try:
        for mode in (0, 3, 4):  # one group of right-hand sides per site, and the tuner's last and first split
            wm.mg_tune(mode)
            for nrhs in counts:
                out = torch.zeros_like(yi[:nrhs])
                wm.coarse_apply(h, 1, wm.MG_F32, yi[:nrhs].contiguous(), out, nrhs)
                assert torch.equal(torch.view_as_real(out), torch.view_as_real(alone[:nrhs])), (mode, nrhs)
    finally:
        wm.mg_tune(old)
    if nv < 16:
        A = wm.mg_get_coarse_op(h, 1).reshape((9,) + lat + (nc, nc))
        ext = [torch.empty((1,) + lat + (nc,), dtype=torch.complex128, device="cuda") for _ in range(2)]
        for src, e in zip((yi, alone), ext):
            wm.mg_field_from_internal(h, 1, wm.MG_F32, src[:1].contiguous(), e, 1)
        y, got = (e.cpu().numpy()[0] for e in ext)
        assert rel_err(got, dirac.stencil_apply(A, y)) < 2e-2
        assert np.isfinite(got).all()
