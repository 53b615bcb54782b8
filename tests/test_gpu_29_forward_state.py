"""The state a forward product leaves for its gradients: its exponents alone, in little
memory, with the gradients that the forward's workspace gives, bit for bit."""
import ctypes

import pytest
import torch

import paper_2603_10634_gb300 as ozk
from paper_2603_10634_gb300 import _lib, workloads


def test_state_sizes_and_checks():
    from paper_2603_10634_gb300 import build

    build.build()
    lib = _lib.load()
    assert lib.ozk2_forward_state_size(64, 65) == 256 + 512
    assert lib.ozk2_forward_state_size(-1, 1) == 0 and lib.ozk2_forward_state_size(1, 2**21) == 0
    null, bogus = ctypes.c_void_p(0), ctypes.c_void_p(0x1000)
    fwd, bwd = lib.ozk2_dgemm_forward, lib.ozk2_dgemm_backward_from
    assert fwd(4, 4, 8, bogus, 4, bogus, 4, bogus, 4, 12, bogus, 4096, null, 0, null) == 1  # lda < k
    assert fwd(0, 4, 4, null, 4, null, 4, null, 4, 12, null, 0, null, 0, null) == 0  # empty: no state
    assert bwd(4, 4, 4, bogus, 4, bogus, 3, bogus, 4, bogus, 4, bogus, 4, 12, bogus, 4096, null, 0, null) == 1
    assert bwd(0, 4, 0, null, 1, null, 4, null, 4, null, 1, null, 4, 12, null, 0, null, 0, null) == 0


@pytest.mark.gpu
def test_a_layer_keeps_little_memory(cuda):
    m, n, k, layers = 512, 384, 2048, 3
    A, B = workloads.problem(m, n, k, 0.5, seed=1, device=cuda)
    A, B = A.requires_grad_(), B.requires_grad_()
    torch.cuda.synchronize()

    def requested():  # bytes asked for, without the caching allocator's rounding of blocks
        return torch.cuda.memory_stats()["requested_bytes.all.current"]

    before = requested()
    outs = [ozk.matmul(A, B) for _ in range(layers)]
    kept = requested() - before
    assert kept == layers * (8 * m * n + ozk.forward_state_size(m, n))  # C and the exponents
    grads = torch.autograd.grad(outs, (A, B), [torch.ones_like(outs[0])] * layers)
    assert all(torch.isfinite(g).all() for g in grads)


@pytest.mark.gpu
@pytest.mark.parametrize("m,n,k,N", [(1, 1, 1, 12), (65, 130, 33, 12), (300, 7, 500, 14), (128, 257, 4097, 20)])
@pytest.mark.parametrize("own", [False, True])
def test_gradients_from_the_state(cuda, m, n, k, N, own):
    A, B = workloads.problem(m, n, k, 1.0, seed=m + n, device=cuda)
    dC = workloads.normal_matrix(m, n, 4, cuda)
    ws = torch.empty(ozk.workspace_size(m, n, k, N), dtype=torch.uint8, device=cuda)
    C = ozk.dgemm(A, B, num_moduli=N, workspace=ws)
    dA, dB = ozk.dgemm_backward(A, B, dC, ws, N)
    space = None if own else torch.full_like(ws, 0x7F)
    C2, state = ozk.dgemm_forward(A, B, N, workspace=space)
    if space is not None:
        space.fill_(0x7F)  # nothing of the workspace is read again
    ozk.dgemm(B, A, num_moduli=N) if m == n else ozk.dgemm(A.T, A, num_moduli=N)
    gA, gB = ozk.dgemm_backward_from(A, B, dC, state, N)
    assert torch.equal(C, C2) and torch.equal(dA, gA) and torch.equal(dB, gB)
    assert torch.equal(ozk.dgemm_backward_from(A, B, dC, state, N, need_dA=False)[1], dB)
    assert torch.equal(ozk.matmul(A, B, N), C)


@pytest.mark.gpu
def test_unusable_states_are_refused(cuda):
    m, n, k = 65, 40, 33
    A, B = workloads.problem(m, n, k, 1.0, seed=1, device=cuda)
    state = ozk.dgemm_forward(A, B)[1]
    dC = torch.ones((m, n), dtype=torch.float64, device=cuda)
    wide = torch.zeros(state.numel() + 256, dtype=torch.uint8, device=cuda)
    for bad in (state[:-256], wide[16:]):
        with pytest.raises(ozk.Ozk2Error):
            ozk.dgemm_backward_from(A, B, dC, bad)
    with pytest.raises(TypeError):
        ozk.dgemm_backward_from(A, B, dC, state.cpu())
