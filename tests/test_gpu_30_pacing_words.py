"""The pacing words of long paired reductions are zero again after every launch, so that each
launch of a call (output row blocks of a host call, both gradients) starts its count anew."""
import pytest
import torch

import paper_2603_10634_gb300 as ozk
from paper_2603_10634_gb300 import workloads

pytestmark = pytest.mark.gpu

PACE = slice(128, 136)  # the two words, 32 words into the flag region at the start of a workspace


def _zero(ws):
    return not bool(ws[PACE].any())


def test_products(cuda):
    m, n, k, N = 2048, 2048, 20000, 12
    A, B = workloads.problem(m, n, k, 1.0, seed=1, device=cuda)
    ws = torch.empty(ozk.workspace_size(m, n, k, N), dtype=torch.uint8, device=cuda)
    for _ in range(10):
        ozk.dgemm(A, B, num_moduli=N, workspace=ws)
        assert _zero(ws)
    assert ozk.device_status(workspace=ws) == "OZK2_OK"


def test_host_row_blocks_and_gradients(cuda):
    m, n, k, N = 4096, 4096, 9000, 12
    A, B = workloads.problem(m, n, k, 1.0, seed=2)
    ws = torch.empty(ozk.workspace_size_host(m, n, k, N), dtype=torch.uint8, device=cuda)
    C = ozk.dgemm_host(A.pin_memory(), B.pin_memory(), num_moduli=N, workspace=ws)
    assert _zero(ws)
    A, B = A.to(cuda), B.to(cuda)
    ref, state = ozk.dgemm_forward(A, B, N)
    assert torch.equal(C, ref.cpu())
    dC = workloads.normal_matrix(m, n, 3, cuda)
    ws = torch.empty(ozk.workspace_size_backward(m, n, k, N), dtype=torch.uint8, device=cuda)
    ozk.dgemm_backward_from(A, B, dC, state, N, workspace=ws)
    assert _zero(ws)
