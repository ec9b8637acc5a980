"""The tensor-core coarse stencil on operators of five and more row tiles with up to 64 right-hand sides.

In the default launch shape (tuning off) and in the tuner's first and last shape the call takes them all: what a
shape cannot hold in shared memory it splits.  Every shape gives the bits of a right-hand side alone.
"""
import numpy as np
import pytest

from gpu_util import rel_err, require_gpu, torch
from oracle import dirac
from paper_0811_4331_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nv0", [((4, 4, 4, 2), 36), ((4, 4, 4, 2), 44), ((4, 4, 4, 2), 56), ((4, 4, 2, 2), 64)])
def test_every_right_hand_side_count_in_default_shapes(dims, nv0):
    wm = require_gpu()
    U = inputs.random_gauge(dims, 6)
    lc = [d // 2 for d in dims]
    p = wm.mg_default_params(n_levels=3, block=[(2, 2, 2, 2), tuple(2 if x % 2 == 0 else 1 for x in lc)],
                             nv=[nv0, 2], setup_sweeps=[2, 2], mixed=1, coarse_mma=1)
    old = wm.mg_tune(0)
    try:
        h = wm.mg_setup(U, dims, -0.1, p)
        ld, nc, _ = wm.mg_level_info(h, 1)
        lat = (ld[3], ld[2], ld[1], ld[0])
        rng = np.random.default_rng(nv0)
        most = 64
        y = rng.standard_normal((most,) + lat + (nc,)) + 1j * rng.standard_normal((most,) + lat + (nc,))
        yi = wm.internal_empty(h, 1, wm.MG_F32, most)
        wm.mg_field_to_internal(h, 1, wm.MG_F32, torch.from_numpy(y).cuda(), yi, most)
        alone = wm.internal_empty(h, 1, wm.MG_F32, most)
        for r in range(most):
            wm.coarse_apply(h, 1, wm.MG_F32, yi[r:r + 1].contiguous(), alone[r:r + 1], 1)
        for mode in (0, 4, 3):
            wm.mg_tune(mode)
            for nrhs in (40, 57, 64):
                out = wm.internal_empty(h, 1, wm.MG_F32, nrhs)
                wm.coarse_apply(h, 1, wm.MG_F32, yi[:nrhs].contiguous(), out, nrhs)
                assert torch.equal(torch.view_as_real(out), torch.view_as_real(alone[:nrhs])), (mode, nrhs)
    finally:
        wm.mg_tune(old)
    A = wm.mg_get_coarse_op(h, 1).reshape((9,) + lat + (nc, nc))
    ext = torch.empty(y.shape, dtype=torch.complex128, device="cuda")
    wm.mg_field_from_internal(h, 1, wm.MG_F32, alone, ext, most)
    # both operands rounded to BF16 (2^-8 relative each, on sums of 9 n random-sign terms)
    assert rel_err(ext[most - 1].cpu().numpy(), dirac.stencil_apply(A, y[most - 1])) < 2e-2
