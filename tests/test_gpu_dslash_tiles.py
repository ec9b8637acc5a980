"""The one-thread-per-site stencils where their launches change form: fused dots over several tiles per CTA
(many right-hand sides), FP32 fields on and off a 32-byte boundary, the fused setup step above and below the
small-lattice size.

FP32 fields 16 bytes off a 32-byte boundary run the 16-byte loads: the same operations in the same order, so
the same bits.  The multi-right-hand-side dots feed a solve, whose solution is checked against its own true FP64
residual; the relaxed null vectors are compared with the FP64 relaxation's prolongator (FP32 arithmetic over 12
sweeps on a well-conditioned field: 1e-4).
"""
import numpy as np
import pytest

from gpu_util import require_gpu, rel_err, torch
from oracle import dirac
from paper_0811_4331_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nrhs", [((16, 8, 8, 33), 1), ((12, 10, 6, 14), 4), ((16, 8, 8, 8), 7)])
def test_fp32_off_a_32_byte_boundary_gives_the_same_bits(dims, nrhs):
    wm = require_gpu()
    V = int(np.prod(dims))
    h = wm.mg_setup(inputs.random_gauge(dims, 3), dims, -0.2, wm.mg_default_params(n_levels=1, mixed=1, fine_prec=1))
    n = nrhs * 12 * V
    store = torch.zeros(n + 8, dtype=torch.complex64, device="cuda")
    vals = torch.randn(n, dtype=torch.complex64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    outs = []
    for off in (0, 2):  # complex64 elements: 0 or 16 bytes
        inp = store[off:off + n]
        inp.copy_(vals)
        out = torch.empty(n, dtype=torch.complex64, device="cuda")
        wm.dslash_apply(h, wm.MG_F32, inp, out, nrhs)
        outs.append(out)
    assert torch.equal(torch.view_as_real(outs[0]), torch.view_as_real(outs[1]))


@pytest.mark.parametrize("prec", [1, 2])
def test_dots_over_several_tiles_in_a_solve(prec):
    """16 x 8 x 8 x 16 with 64 right-hand sides: 8192 tiles of 128 sites, several per CTA in every type."""
    wm = require_gpu()
    dims, nrhs = (16, 8, 8, 16), 64
    U = inputs.random_gauge(dims, 4)
    p = wm.mg_default_params(n_levels=2, block=[(4, 4, 4, 4)], nv=[8], setup_sweeps=[8], mixed=1, fine_prec=prec)
    h = wm.mg_setup(U, dims, 0.2, p)
    B = np.stack([inputs.gaussian_spinor(dims, r) for r in range(nrhs)])
    x = np.zeros_like(B)
    wm.mg_solve(h, B, x, 1e-10)
    for r in (0, 31, nrhs - 1):
        assert np.linalg.norm(B[r] - dirac.wilson_dirac(U, x[r], 0.2)) <= 1e-10 * np.linalg.norm(B[r])


@pytest.mark.parametrize("dims,nv", [((8, 4, 4, 8), 8), ((8, 8, 4, 12), 12), ((12, 8, 8, 8), 7)])
def test_fused_relaxation_against_fp64(dims, nv):
    wm = require_gpu()
    U = inputs.random_gauge(dims, 5)
    P = []
    for mixed in (0, 1):
        p = wm.mg_default_params(n_levels=2, block=[(4, 4, 4, 4)], nv=[nv], setup_sweeps=[12], mixed=mixed, seed=3)
        h = wm.mg_setup(U, dims, 0.2, p)
        P.append(wm.mg_get_prolongator(h, 0))
    assert rel_err(P[1], P[0]) < 1e-4
