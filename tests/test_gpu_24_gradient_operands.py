"""The gradients' fixed operands, converted with an exponent per position: shapes around the
items' and tiles' edges, rows that do and do not start on 16 bytes, and one gradient alone.
Bit-exact against the oracle fed with the GPU's exponents."""
import numpy as np
import pytest
import torch

import paper_2603_10634_gb300 as ozk
from oracle import ozaki2 as oz
from paper_2603_10634_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("m,n,k,N", [(1, 9, 17, 12), (31, 129, 16, 12), (128, 33, 15, 14), (130, 64, 33, 12)])
def test_fixed_operands(cuda, m, n, k, N, pad):
    A, B = workloads.problem(m, n, k, 1.0, seed=m + n)
    dC = workloads.normal_matrix(m, n, seed=k)
    Ad = torch.nn.functional.pad(A, (0, pad)).to(cuda)[:, :k]
    Bd = torch.nn.functional.pad(B, (0, pad)).to(cuda)[:, :n]
    ws = torch.empty(ozk.workspace_size(m, n, k, N), dtype=torch.uint8, device=cuda)
    ozk.dgemm(Ad, Bd, num_moduli=N, workspace=ws)
    sc = ozk.scales(Ad, Bd, num_moduli=N)
    dA, dB = ozk.dgemm_backward(Ad, Bd, dC.to(cuda), ws, N)
    g, h = (x.cpu().numpy() for x in ozk.backward_exponents(m, n, k, N))
    r = oz.reuse_gradients(A.numpy(), B.numpy(), dC.numpy(), N, e=sc["e"].cpu().numpy(), f=sc["f"].cpu().numpy(), g=g, h=h)
    assert np.array_equal(dA.cpu().numpy().view(np.uint64), r["dA"].view(np.uint64))
    assert np.array_equal(dB.cpu().numpy().view(np.uint64), r["dB"].view(np.uint64))
    assert torch.equal(ozk.dgemm_backward(Ad, Bd, dC.to(cuda), ws, N, need_dB=False)[0], dA)
    assert torch.equal(ozk.dgemm_backward(Ad, Bd, dC.to(cuda), ws, N, need_dA=False)[1], dB)
    assert ozk.device_status() == "OZK2_OK"
