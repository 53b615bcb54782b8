"""Residue products in CTA pairs (256 x 256 tiles over two CTAs, paced on long reductions):
integer matrices whose products are exact in FP64, at the edges of the tiles, the k-steps
and the exactness blocks; and a pair whose first wait runs out."""
import pytest
import torch

import paper_2603_10634_gb300 as ozk
from paper_2603_10634_gb300 import _lib

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def wide_tiles(cuda):
    """Pairs run 256-wide tiles; the smaller shapes here would take the narrow ones."""
    with ozk.tile_width(256):
        yield


def _integers(rows, cols, seed, device):
    g = torch.Generator(device=device).manual_seed(seed)
    return torch.randint(-1000, 1001, (rows, cols), generator=g, device=device).double()


@pytest.mark.parametrize("N", [12, 14])
@pytest.mark.parametrize("m,n,k", [(256, 256, 8192), (385, 257, 8191), (511, 1000, 4097), (640, 300, 16384),
                                   (641, 511, 16385), (1100, 1030, 1100), (2048, 2048, 129),
                                   (385, 600, 70000), (2050, 2049, 17000)])  # the last two are paced
def test_integer_products_are_exact(cuda, N, m, n, k):
    A, B = _integers(m, k, m + n, cuda), _integers(k, n, k, cuda)
    C = ozk.dgemm(A, B, num_moduli=N)
    assert ozk.device_status() == "OZK2_OK"
    assert torch.equal(C, A @ B)
    assert torch.equal(ozk.dgemm(A, B, num_moduli=N, out=torch.empty_like(C)), C)  # the pacing words are zero again


def test_stalled_pair_returns_a_timeout(cuda):
    lib = _lib.load()
    A, B = _integers(512, 8192, 1, cuda), _integers(8192, 512, 2, cuda)
    ref = ozk.dgemm(A, B, mode="fast")
    prev = lib.ozk2_set_wait_limit(2_000_000)
    try:
        lib.ozk2_debug_inject_fault(3)  # the first wait of the next FP8 product launch runs out
        ozk.dgemm(A, B, mode="fast")
        assert ozk.device_status() == "OZK2_ERR_TIMEOUT"
    finally:
        lib.ozk2_set_wait_limit(prev)
    assert torch.equal(ozk.dgemm(A, B, mode="fast"), ref)
    assert ozk.device_status() == "OZK2_OK"
