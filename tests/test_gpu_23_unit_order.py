"""Order of the residue products' units: the CTAs without a Karatsuba unit in their last,
incomplete round take three single ones first.  Shapes with fewer units than CTAs, with and
without an incomplete round, with too few single units to catch up, singly and in pairs;
integer matrices whose products are exact in FP64."""
import pytest
import torch

import paper_2603_10634_gb300 as ozk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [12, 14, 16, 20])
@pytest.mark.parametrize("m,n,k", [(40, 70, 64), (256, 256, 300), (300, 700, 500), (1100, 1100, 600), (2048, 2432, 256),
                                   (9728, 256, 128), (1023, 777, 1501), (2050, 2300, 1100), (4864, 1024, 2048)])
def test_every_unit_is_computed(cuda, m, n, k, N):
    g = torch.Generator(device=cuda).manual_seed(m + n)
    A = torch.randint(-1000, 1001, (m, k), generator=g, device=cuda).double()
    B = torch.randint(-1000, 1001, (k, n), generator=g, device=cuda).double()
    C = ozk.dgemm(A, B, num_moduli=N)
    assert ozk.device_status() == "OZK2_OK"
    assert torch.equal(C, A @ B)
