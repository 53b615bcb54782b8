"""Chained launches (a kernel's prologue overlaps the previous kernel): calls back to back
on one stream, concurrently on two streams with their own workspaces, and replayed from a
CUDA graph give the bits of a call that runs alone."""
import pytest
import torch

import paper_2603_10634_gb300 as ozk
from paper_2603_10634_gb300 import workloads

pytestmark = pytest.mark.gpu

SHAPES = [(96, 80, 200), (256, 256, 256), (700, 130, 900), (1024, 1024, 512)]


def _alone(A, B, mode):
    torch.cuda.synchronize()
    C = ozk.dgemm(A, B, mode=mode)
    torch.cuda.synchronize()
    return C


@pytest.mark.parametrize("mode", ["accurate", "fast"])
def test_back_to_back_calls_of_changing_sizes(cuda, mode):
    probs = [workloads.problem(m, n, k, 1.0, seed=i, device=cuda) for i, (m, n, k) in enumerate(SHAPES)]
    want = [_alone(A, B, mode) for A, B in probs]
    for _ in range(20):  # one shared workspace: every call overwrites what the one before read
        got = [ozk.dgemm(A, B, mode=mode) for A, B in probs]
        assert all(torch.equal(g, w) for g, w in zip(got, want))


def test_two_streams_with_their_own_workspaces(cuda):
    probs = [workloads.problem(m, n, k, 1.0, seed=i, device=cuda) for i, (m, n, k) in enumerate(SHAPES)]
    want = [_alone(A, B, "accurate") for A, B in probs]
    need = max(ozk.workspace_size(m, n, k) for m, n, k in SHAPES)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    spaces = [torch.empty(need, dtype=torch.uint8, device=cuda) for _ in streams]
    outs = []
    torch.cuda.synchronize()
    for rep in range(10):
        for i, (A, B) in enumerate(probs):
            s = (rep + i) % 2
            with torch.cuda.stream(streams[s]):
                outs.append((i, ozk.dgemm(A, B, workspace=spaces[s])))
    torch.cuda.synchronize()
    assert all(torch.equal(C, want[i]) for i, C in outs)


@pytest.mark.parametrize("mode,ta", [("accurate", False), ("fast", True)])
def test_graph_replay(cuda, mode, ta):
    m, n, k = 512, 384, 4096  # large enough for CTA pairs
    A, B = workloads.problem(m, n, k, 1.0, seed=3, device=cuda)
    if ta:
        A = A.T.contiguous().T
    C = torch.empty((m, n), dtype=torch.float64, device=cuda)
    ws = torch.empty(ozk.workspace_size(m, n, k, 12, mode), dtype=torch.uint8, device=cuda)
    ozk.dgemm(A, B, out=C, workspace=ws, mode=mode)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ozk.dgemm(A, B, out=C, workspace=ws, mode=mode)
        ozk.dgemm(A, B, out=C, workspace=ws, mode=mode)
    for seed in (5, 6):
        A2, B2 = workloads.problem(m, n, k, 1.0, seed=seed, device=cuda)
        A.copy_(A2)
        B.copy_(B2)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(C, _alone(A, B, mode))
