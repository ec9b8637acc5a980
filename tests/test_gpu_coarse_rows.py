"""The tensor-core coarse stencil at the edges of its tiles: one to five row tiles (with and without padded
rows), site counts that are no multiple of 32, and the right-hand side counts at which it changes from
gathering the vectors to staging their BF16 rows.

Against the FP64 stencil the tolerance is the rounding of both operands to BF16 (2^-8 relative each, on sums of
9 n random-sign terms): 2e-2.  The rounding of the vectors and the order of every sum are the same in either
staging, so a right-hand side alone and among others gives the same bits.
"""
import numpy as np
import pytest

from gpu_util import rel_err, require_gpu, torch
from oracle import dirac
from paper_0811_4331_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nv0", [((4, 4, 4, 4), 4), ((6, 4, 8, 10), 16), ((4, 4, 6, 2), 21), ((8, 4, 4, 4), 32), ((4, 4, 4, 4), 52),
                                      ((4, 4, 4, 8), 36)])
def test_rows_and_gathers_match(dims, nv0):
    wm = require_gpu()
    U = inputs.random_gauge(dims, 6)
    lc = [d // 2 for d in dims]
    p = wm.mg_default_params(n_levels=3, block=[(2, 2, 2, 2), tuple(2 if x % 2 == 0 else x for x in lc)],
                             nv=[nv0, 2], setup_sweeps=[3, 2], mixed=1, coarse_mma=1)
    h = wm.mg_setup(U, dims, -0.1, p)
    ld, nc, _ = wm.mg_level_info(h, 1)
    lat = (ld[3], ld[2], ld[1], ld[0])
    A = wm.mg_get_coarse_op(h, 1).reshape((9,) + lat + (nc, nc))
    rng = np.random.default_rng(nv0)
    most = 64
    y = rng.standard_normal((most,) + lat + (nc,)) + 1j * rng.standard_normal((most,) + lat + (nc,))
    yi = wm.internal_empty(h, 1, wm.MG_F32, most)
    wm.mg_field_to_internal(h, 1, wm.MG_F32, torch.from_numpy(y).cuda(), yi, most)
    alone = wm.internal_empty(h, 1, wm.MG_F32, most)
    for r in range(most):
        wm.coarse_apply(h, 1, wm.MG_F32, yi[r:r + 1].contiguous(), alone[r:r + 1], 1)
    for nrhs in (3, 4, 9, 24, 64):
        out = wm.internal_empty(h, 1, wm.MG_F32, nrhs)
        wm.coarse_apply(h, 1, wm.MG_F32, yi[:nrhs].contiguous(), out, nrhs)
        assert torch.equal(torch.view_as_real(out), torch.view_as_real(alone[:nrhs])), nrhs
    ext = torch.empty(y.shape, dtype=torch.complex128, device="cuda")
    wm.mg_field_from_internal(h, 1, wm.MG_F32, alone, ext, most)
    ext = ext.cpu().numpy()
    for r in (0, 17, most - 1):
        assert rel_err(ext[r], dirac.stencil_apply(A, y[r])) < 2e-2, r
