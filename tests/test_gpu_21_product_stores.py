"""Stores of the residue products: four rows' pieces of 16 columns change lanes before they
are stored, so every row and column remainder of those pieces is checked, over one and several
exactness blocks (the later ones add to what is stored), with integer products exact in FP64."""
import pytest
import torch

import paper_2603_10634_gb300 as ozk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 3, 4, 31, 127, 130, 257])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 63, 65, 129, 321])
@pytest.mark.parametrize("k", [96, 33000])
def test_remainders_of_the_stored_pieces(cuda, m, n, k):
    g = torch.Generator(device=cuda).manual_seed(m * n)
    A = torch.randint(-1000, 1001, (m, k), generator=g, device=cuda).double()
    B = torch.randint(-1000, 1001, (k, n), generator=g, device=cuda).double()
    want = A @ B
    assert torch.equal(ozk.dgemm(A, B), want)
    assert torch.equal(ozk.dgemm_batched([A, A], [B, B])[1], want)
    assert ozk.device_status() == "OZK2_OK"
