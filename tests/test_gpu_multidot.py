"""Overlaps of the Gram-Schmidt passes, single and in pairs of elements: odd lengths, chunks past the vectors in use,
one block and more than one per SM, against FP64.

Partial sums of an FP32 thread hold at most 2 x 42 products here and are added in FP32 over the 256 threads of a
block, in FP64 over blocks: below 120 x 2^-24 of the sum of the absolute values.
"""
import ctypes

import pytest

from gpu_util import require_gpu, torch

pytestmark = pytest.mark.gpu
TYPES = {0: torch.complex128, 1: torch.complex64}


@pytest.mark.parametrize("n,nrhs,k", [(1, 1, 1), (257, 2, 3), (4098, 1, 8), (98304, 3, 9), (400001, 1, 8), (400002, 5, 17),
                                      (1572864, 1, 5), (1572864, 1, 40), (1572862, 7, 8)])
@pytest.mark.parametrize("prec", [0, 1])
def test_overlaps(n, nrhs, k, prec):
    require_gpu()
    import launch_harness as lh
    lib = lh.load()
    gen = torch.Generator("cuda").manual_seed(n)
    k8, kmax = (k + 7) // 8 * 8, 48
    W = torch.randn(k8, nrhs, n, dtype=TYPES[prec], device="cuda", generator=gen)
    w = torch.randn(nrhs, n, dtype=TYPES[prec], device="cuda", generator=gen)
    partials = torch.full((1216 * 16 * (8 * nrhs + 1),), float("nan"), dtype=torch.float64, device="cuda")
    tickets = torch.zeros(4096, dtype=torch.int32, device="cuda")
    result = torch.zeros(nrhs, kmax, 2, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.t_multidot(prec, ctypes.c_size_t(n), nrhs, k, kmax, lh.ptr(W), lh.ptr(w), lh.ptr(partials), lh.ptr(tickets),
                          lh.ptr(result)) == 0
    torch.cuda.synchronize()
    assert int(tickets.abs().sum()) == 0
    for j in range(k):
        v = W[j].to(torch.complex128)
        want = (v.conj() * w).sum(1)
        size = (v.abs() * w.abs()).sum(1)
        got = torch.view_as_complex(result[:, j].contiguous())
        assert bool(((got - want).abs() < (1e-13 if prec == 0 else 7.2e-6) * size).all()), j
