"""The residue conversion copies the next rows or columns while it converts the present ones,
and takes both operands in one launch: shapes of one and of many items a warp (rows) and tiles
a block (columns), with remainders of both, in aligned and unaligned rows, and with either
operand much the larger; integer matrices whose products are exact in FP64."""
import pytest
import torch

import paper_2603_10634_gb300 as ozk

pytestmark = pytest.mark.gpu


def _stored(rows, cols, transposed, pad, seed, device):
    g = torch.Generator(device=device).manual_seed(seed)
    shape = (cols, rows + pad) if transposed else (rows, cols + pad)
    X = torch.randint(-1000, 1001, shape, generator=g, device=device).double()
    return X[:, :rows].T if transposed else X[:, :cols]


@pytest.mark.parametrize("ta,tb", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("m,n,k", [(1, 1, 40), (2, 17, 129), (4000, 3, 1001), (5, 4100, 1003), (1030, 1025, 2050),
                                   (2061, 700, 33)])
def test_shapes_of_the_copies(cuda, m, n, k, ta, tb, pad):
    A, B = _stored(m, k, ta, pad, m, cuda), _stored(k, n, tb, pad, n, cuda)
    C = ozk.dgemm(A, B)
    assert ozk.device_status() == "OZK2_OK"
    assert torch.equal(C, A.contiguous() @ B.contiguous())
    if not (ta or tb):  # the batch takes row-major operands
        assert torch.equal(ozk.dgemm_batched([A, A], [B, B])[1], C)
