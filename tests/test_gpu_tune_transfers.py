"""The tuner times the launch shapes of the transfer kernels that run, every one of them once.

Transfers between 16-bit levels run on the plane kernels, whose shapes are groups of 1, 2, 3, 4, 6 or 8 tiles of
eight right-hand sides, as far as there are that many; level 0 with FP32 below it on the tile kernels.
"""
import numpy as np
import pytest

from gpu_util import require_gpu
from paper_0811_4331_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [9, 40, 64])
def test_shapes_of_the_kernels_that_run(nrhs):
    wm = require_gpu()
    dims = (4, 4, 4, 8)
    U = inputs.random_gauge(dims, 6)
    B = np.stack([inputs.gaussian_spinor(dims, 40 + r) for r in range(nrhs)])
    old = wm.mg_tune(2)
    wm.mg_tune(2)  # an empty table
    try:
        for coarse in (wm.MG_BF16, wm.MG_F32):
            p = wm.mg_default_params(n_levels=3, block=[(2, 2, 2, 4), (2, 2, 1, 1)], nv=[6, 2],
                                     setup_sweeps=[4, 2], mixed=1, fine_prec=wm.MG_BF16, coarse_prec=coarse, max_iter=4)
            h = wm.mg_setup(U, dims, 0.3, p)
            wm.mg_solve(h, B, np.zeros_like(B), 1e-2, raise_on_noconv=False)
            wm.mg_destroy(h)
        rep = {}
        for key, (_, us) in wm.mg_tune_report().items():
            f = key.split("|")  # kernel, fine and coarse storage, vectors, sites of an aggregate, aggregates, ...
            if f[0] in ("restrict_mma", "prolong_mma") and f[3:5] == ["6", "32"]:
                rep[f[0] + "|" + f[2]] = us
        tiles = (nrhs + 7) // 8
        planes = sum(t <= tiles for t in (1, 2, 3, 4, 6, 8))
        twice = 2 if nrhs > 16 else 1
        got = {k: len(us) for k, us in rep.items()}
        assert got == {"restrict_mma|%d" % wm.MG_BF16: planes, "prolong_mma|%d" % wm.MG_BF16: planes,
                       "restrict_mma|%d" % wm.MG_F32: 2 * twice, "prolong_mma|%d" % wm.MG_F32: 4 * twice}, got
        assert all(u > 0 for us in rep.values() for u in us), rep
    finally:
        wm.mg_tune(old)
