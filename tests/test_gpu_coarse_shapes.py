"""The CUDA-core coarse stencil in every tile that its launch rule picks: FP64 tiles of 4 to 32 units counted through
all rows, FP32 and 16-bit tiles of one, two and four rows in whole and in shared CTAs, rows past the last one
(n = 46: four rows at a time), site counts off the 16-byte groups and a tile's right-hand sides past the last one.

Against the FP64 stencil on the inputs as stored, with the tolerances of test_gpu_coarse_sites.py (they bound the
storage rounding of operator and result and the FP32 sums, and do not grow with n: terms and sums are random-signed).
"""
import numpy as np
import pytest

from gpu_util import rel_err, require_gpu, torch
from oracle import dirac
from paper_0811_4331_gb300 import inputs
from test_gpu_coarse_sites import TOL

pytestmark = pytest.mark.gpu

CASES = [
    # lattice (2^4 aggregates), nv, right-hand sides
    ((2, 2, 2, 4), 32, (1, 3, 24, 64)),       # two sites: tiles across rows, the narrowest ones
    ((4, 4, 4, 4), 24, (3, 12)),              # 16 sites
    ((4, 6, 6, 4), 32, (1, 4, 12)),           # 36 sites: two rows and a part per CTA
    ((4, 6, 6, 6), 23, (1, 3, 12)),           # 54 sites, 46 rows
    ((8, 8, 8, 16), 23, (1, 2, 5, 8)),        # 512 sites: two and four rows per CTA
    ((10, 10, 6, 14), 16, (1, 3, 8)),         # 525 sites: single elements
]


@pytest.mark.parametrize("dims,nv,counts", CASES)
@pytest.mark.parametrize("prec", [0, 1, 2, 3])
def test_coarse_shapes_match_oracle(dims, nv, counts, prec):
    wm = require_gpu()
    U = inputs.random_gauge_fast(dims, 6)
    lc = [d // 2 for d in dims]
    block = [(2, 2, 2, 2), tuple(2 if x % 2 == 0 else 1 for x in lc)]
    kw = {} if prec == 0 else dict(mixed=1, fine_prec=prec, coarse_prec=prec)
    p = wm.mg_default_params(n_levels=3, block=block, nv=[nv, 2], setup_sweeps=[2, 2], defer_coarsest=1, **kw)
    h = wm.mg_setup(U, dims, -0.1, p)
    ld, nc, _ = wm.mg_level_info(h, 1)
    lat = (ld[3], ld[2], ld[1], ld[0])
    A = wm.mg_get_coarse_op(h, 1).reshape((9,) + lat + (nc, nc))
    rng = np.random.default_rng(nv)
    for nrhs in counts:
        y = rng.standard_normal((nrhs,) + lat + (nc,)) + 1j * rng.standard_normal((nrhs,) + lat + (nc,))
        ext = torch.from_numpy(y).cuda()
        yi, oi = (wm.internal_empty(h, 1, prec, nrhs) for _ in range(2))
        wm.mg_field_to_internal(h, 1, prec, ext, yi, nrhs)
        wm.coarse_apply(h, 1, prec, yi, oi, nrhs)
        stored, out = torch.empty_like(ext), torch.empty_like(ext)
        wm.mg_field_from_internal(h, 1, prec, yi, stored, nrhs)
        wm.mg_field_from_internal(h, 1, prec, oi, out, nrhs)
        stored, out = stored.cpu().numpy(), out.cpu().numpy()
        for r in sorted({0, nrhs // 2, nrhs - 1}):
            assert rel_err(out[r], dirac.stencil_apply(A, stored[r])) < TOL[prec], (nrhs, r)
