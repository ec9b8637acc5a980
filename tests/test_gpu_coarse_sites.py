"""The CUDA-core coarse stencil at the edges of its tiles: site counts off the 16-byte groups (1, 2 or 4 sites),
rows past the component count, right-hand side counts between its groups, few and many outputs, every precision.

Tolerances against the FP64 stencil on the inputs as stored: FP64 1e-13; FP32 2e-6 (operator and sums in FP32);
FP16 4e-3 and BF16 3e-2, a few units of the storage rounding of the operator and the result.
"""
import numpy as np
import pytest

from gpu_util import rel_err, require_gpu, torch
from oracle import dirac
from paper_0811_4331_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = {0: 1e-13, 1: 2e-6, 2: 4e-3, 3: 3e-2}


@pytest.mark.parametrize("dims,nv", [((6, 6, 6, 2), 5), ((6, 4, 4, 10), 6), ((4, 4, 4, 4), 3), ((8, 8, 8, 8), 8),
                                     ((16, 16, 16, 16), 9)])
@pytest.mark.parametrize("prec", [0, 1, 2, 3])
def test_coarse_sites_match_oracle(dims, nv, prec):
    wm = require_gpu()
    U = inputs.random_gauge_fast(dims, 6)
    lc = [d // 2 for d in dims]
    block = [(2, 2, 2, 2), tuple(2 if x % 2 == 0 else x for x in lc)]
    kw = {} if prec == 0 else dict(mixed=1, fine_prec=prec, coarse_prec=prec)
    p = wm.mg_default_params(n_levels=3, block=block, nv=[nv, 2], setup_sweeps=[2, 2], defer_coarsest=1, **kw)
    h = wm.mg_setup(U, dims, -0.1, p)
    ld, nc, _ = wm.mg_level_info(h, 1)
    lat = (ld[3], ld[2], ld[1], ld[0])
    A = wm.mg_get_coarse_op(h, 1).reshape((9,) + lat + (nc, nc))
    rng = np.random.default_rng(nv)
    for nrhs in (1, 2, 3, 5):
        y = rng.standard_normal((nrhs,) + lat + (nc,)) + 1j * rng.standard_normal((nrhs,) + lat + (nc,))
        ext = torch.from_numpy(y).cuda()
        yi, oi = (wm.internal_empty(h, 1, prec, nrhs) for _ in range(2))
        wm.mg_field_to_internal(h, 1, prec, ext, yi, nrhs)
        wm.coarse_apply(h, 1, prec, yi, oi, nrhs)
        stored, out = torch.empty_like(ext), torch.empty_like(ext)
        wm.mg_field_from_internal(h, 1, prec, yi, stored, nrhs)
        wm.mg_field_from_internal(h, 1, prec, oi, out, nrhs)
        stored, out = stored.cpu().numpy(), out.cpu().numpy()
        for r in range(nrhs):
            assert rel_err(out[r], dirac.stencil_apply(A, stored[r])) < TOL[prec], (nrhs, r)
