"""The streaming coarse stencil when the waits for its copies run out: every output is NaN, so that no right-hand side
comes back finite and wrong.

The limit of the waits is a launch argument; with none left, no wait is tried, no copy is issued and the kernel ends
at once (nothing hangs and no address depends on it).  With the usual limit the same launch gives the bits of the
form that gathers its vectors itself.
"""
import pytest

from gpu_util import require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R,variant", [(20, 24, -1), (48, 64, -1), (48, 24, 2), (90, 17, -1)])
def test_no_right_hand_side_survives_a_wait_that_ran_out(n, R, variant):
    require_gpu()
    import launch_harness as lh
    lib = lh.load()
    L = (4, 4, 4, 3)
    V = 192
    gen = torch.Generator("cuda").manual_seed(n)
    C = torch.randn(9, n, n, V, dtype=torch.complex128, device="cuda", generator=gen)
    x = torch.randn(R, n, V, dtype=torch.complex64, device="cuda", generator=gen)
    packed = torch.empty(lib.t_mma_pack_bytes(n, V), dtype=torch.uint8, device="cuda")
    scratch = torch.empty(lib.t_mma_scratch_bytes(n, V, R), dtype=torch.uint8, device="cuda")
    outs = []
    for s, spins in ((None, 1 << 18), (scratch, 1 << 18), (scratch, 0)):
        out = torch.zeros_like(x)
        torch.cuda.synchronize()
        assert lib.t_coarse_mma(lh.ptr(C), lh.ptr(packed), lh.ptr(x), lh.ptr(out), lh.ints(*L), n, R, variant, lh.ptr(s),
                                spins) == 0
        torch.cuda.synchronize()
        outs.append(torch.view_as_real(out))
    assert torch.equal(outs[0], outs[1])
    assert bool(torch.isnan(outs[2]).all())
