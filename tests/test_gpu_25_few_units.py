"""Narrow tiles for products with few units, and long rows shared by a block's warps: the same
bits as with the wide tile, and as with the operands stored along the other dimension (the
column kernels), for lengths around the row kernels' limits and with special lines."""
import pytest
import torch

import paper_2603_10634_gb300 as ozk
from paper_2603_10634_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [5, 12, 16])
@pytest.mark.parametrize("m,n,k", [(1, 200, 40), (256, 256, 1000), (300, 700, 500), (513, 513, 2000), (128, 2048, 300),
                                   (768, 768, 260)])
def test_tile_of_few_units(cuda, m, n, k, N):
    A, B = workloads.problem(m, n, k, 1.0, seed=m + k)
    A, B = A.to(cuda), B.to(cuda)
    C = ozk.dgemm(A, B, num_moduli=N)
    for t in (128, 256):
        with ozk.tile_width(t):
            assert torch.equal(ozk.dgemm(A, B, num_moduli=N), C)
    assert ozk.device_status() == "OZK2_OK"


@pytest.mark.parametrize("m,n", [(1, 3), (5, 64), (70, 9)])
@pytest.mark.parametrize("k", [8192, 8193, 8255, 10500, 33000])
def test_long_rows(cuda, m, n, k):
    A, B = (x.to(cuda) for x in workloads.problem(m, n, k, 2.0, seed=k))
    if m > 4:
        A[0] = 0.0
        A[1, k - 1] = float("nan")
        A[2] *= 2.0**-1030  # subnormal entries
        A[3, :k - 1] = 0.0
    Bt = B.T.contiguous().T
    C = ozk.dgemm(A, Bt)
    D = ozk.dgemm(A.T.contiguous().T, B)
    assert torch.equal(C.view(torch.int64), D.view(torch.int64))
    assert ozk.device_status() == ("OZK2_ERR_NONFINITE" if m > 4 else "OZK2_OK")
