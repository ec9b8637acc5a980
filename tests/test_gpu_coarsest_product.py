"""The coarsest product in its forms, against FP64 matrix products: rows that do not start on 16 bytes, rows past the
last one, two and four rows per CTA, the vector in pieces (FP64 above 4096 rows), and the counts of right-hand sides
on both sides of the tiled product.

A sum of N products with random signs has a relative rounding error of about sqrt(N) units, an FP32 vector staged
from FP64 half a unit more: 1e-13 in FP64 and 3e-6 in FP32 hold to N = 5,000 with a margin of ten.
"""
import pytest

from gpu_util import require_gpu, torch

pytestmark = pytest.mark.gpu
TYPES = {0: torch.complex128, 1: torch.complex64}


@pytest.mark.parametrize("N", [3, 97, 512, 1026, 2048, 3073, 4100, 5000])
@pytest.mark.parametrize("pm,pv", [(0, 0), (1, 0), (1, 1)])
def test_products(N, pm, pv):
    require_gpu()
    import launch_harness as lh
    lib = lh.load()
    gen = torch.Generator("cuda").manual_seed(N)
    A = torch.randn(N, N, dtype=TYPES[pm], device="cuda", generator=gen)
    x = torch.randn(33, N, dtype=TYPES[pv], device="cuda", generator=gen)
    scratch = torch.zeros(lib.t_matvec_scratch_bytes(N), dtype=torch.uint8, device="cuda")
    want = x.to(torch.complex128) @ A.to(torch.complex128).T
    for nrhs in (1, 2, 3, 5, 12, 13, 16, 17, 33):
        y = torch.ones(nrhs, N, dtype=TYPES[pv], device="cuda")
        for acc in (0, 1):
            torch.cuda.synchronize()
            assert lib.t_matvec(pm, pv, pv, N, lh.ptr(A), lh.ptr(x), lh.ptr(y), nrhs, acc, lh.ptr(scratch)) == 0
            torch.cuda.synchronize()
        diff = torch.linalg.vector_norm(y.to(torch.complex128) - 2 * want[:nrhs], dim=1)
        rel = diff / torch.linalg.vector_norm(2 * want[:nrhs], dim=1)
        assert float(rel.max()) < (1e-13 if pm == 0 else 3e-6), (nrhs, float(rel.max()))
