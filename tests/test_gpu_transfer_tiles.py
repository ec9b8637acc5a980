"""The pipelined level-0 transfers at the edges of their tiles (16 sites per stage, groups of four sites,
8 vectors and 16 right-hand sides per MMA tile), against P and the fields in FP64.

Tolerances: inputs and P enter rounded to the storage type (2^-11 relative for FP16, 2^-8 for BF16, each
operand once) and the result is rounded once more where it is 16 bits, so 8 units of that rounding bound the
2-norm of the error.
"""
import numpy as np
import pytest

from gpu_util import lattice, rel_err, require_gpu, torch
from oracle import multigrid as mg
from paper_0811_4331_gb300 import inputs
from test_gpu_transfer_mma import _oracle_P, _to_dev, _to_host

pytestmark = pytest.mark.gpu

CASES = [
    # dims, block, nv, right-hand sides, storage
    ((4, 2, 2, 2), (2, 2, 1, 1), 7, 2, 2),     # four sites: one group, part of one stage; columns past nv
    ((6, 6, 4, 2), (6, 3, 2, 1), 9, 17, 2),    # 36 sites: two full stages and one group; two splits of rows
    ((4, 4, 4, 4), (2, 2, 2, 2), 16, 16, 3),   # exactly one stage, one row tile
    ((8, 4, 4, 4), (4, 4, 4, 4), 24, 33, 2),   # 16 stages, three row tiles in two CTAs
    ((4, 4, 4, 8), (4, 4, 4, 4), 52, 15, 3),   # two groups of n-tiles
    ((4, 4, 4, 4), (2, 2, 4, 4), 64, 64, 2),   # the most vectors and right-hand sides
]


@pytest.mark.parametrize("dims,block,nv,nrhs,prec", CASES)
def test_tiles_match_fp64(dims, block, nv, nrhs, prec):
    wm = require_gpu()
    U = inputs.random_gauge(dims, 2)
    p = wm.mg_default_params(n_levels=2, block=[block], nv=[nv], setup_sweeps=[2], mixed=1, fine_prec=prec)
    h = wm.mg_setup(U, dims, 0.2, p)
    lat = lattice(dims)
    P = _oracle_P(wm.mg_get_prolongator(h, 0).reshape((nv,) + lat + (12,)), nv, 6)
    blk = mg.Blocking(lat, block, 12)
    rng = np.random.default_rng(nv)
    r = rng.standard_normal((nrhs,) + lat + (12,)) + 1j * rng.standard_normal((nrhs,) + lat + (12,))
    xc = rng.standard_normal((nrhs,) + blk.coarse + (2 * nv,)) + 1j * rng.standard_normal(
        (nrhs,) + blk.coarse + (2 * nv,))
    eps = 2.0 ** -11 if prec == 2 else 2.0 ** -8
    out = wm.internal_empty(h, 1, 1, nrhs)
    wm.restrict_apply(h, 0, prec, _to_dev(wm, h, 0, r, prec, nrhs), out, nrhs)
    got = _to_host(wm, h, 1, out, xc.shape, 1, nrhs)
    fo = wm.internal_empty(h, 0, prec, nrhs)
    wm.prolong_apply(h, 0, prec, _to_dev(wm, h, 1, xc, 1, nrhs), fo, nrhs)
    pro = _to_host(wm, h, 0, fo, r.shape, prec, nrhs)
    for i in range(nrhs):
        assert rel_err(got[i], mg.restrict(P, blk, r[i])) < 8 * eps, i
        assert rel_err(pro[i], mg.prolong(P, blk, xc[i])) < 8 * eps, i


def test_tile_shapes_give_the_same_bits():
    """20 right-hand sides: every split of the tile kernels (chiralities, parts, row tiles) in a whole solve."""
    wm = require_gpu()
    dims = (8, 4, 4, 8)
    U = inputs.random_gauge(dims, 6)
    B = np.stack([inputs.gaussian_spinor(dims, 40 + r) for r in range(20)])
    old = wm.mg_tune(0)
    got = []
    try:
        for mode in (0, 4, 3):
            wm.mg_tune(mode)
            p = wm.mg_default_params(n_levels=2, block=[(4, 2, 2, 4)], nv=[12], setup_sweeps=[6], mixed=1, seed=3)
            h = wm.mg_setup(U, dims, -0.2, p)
            x = np.zeros_like(B)
            wm.mg_solve(h, B, x, 1e-10)
            got.append(x)
    finally:
        wm.mg_tune(old)
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])
