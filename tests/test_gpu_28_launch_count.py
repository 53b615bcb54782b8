"""ozk2_last_launch_count against the kernel nodes of the call captured into a CUDA graph,
over the row lengths where the scaling takes one launch or two."""
import ctypes

import pytest
import torch

import paper_2603_10634_gb300 as ozk
from paper_2603_10634_gb300 import workloads

pytestmark = pytest.mark.gpu


def _kernel_nodes(graph):
    cu = ctypes.CDLL("libcuda.so.1")
    h, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(h, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(h, nodes, ctypes.byref(n)) == 0
    kernels = 0
    for node in nodes:
        kind = ctypes.c_int(-1)
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kernels += kind.value == 0  # CU_GRAPH_NODE_TYPE_KERNEL
    return kernels


def _launches(fn):
    fn()  # first-use set-up outside the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        fn()
    return ozk.last_launch_count(), _kernel_nodes(graph)


@pytest.mark.parametrize("mode", ["accurate", "fast"])
@pytest.mark.parametrize("k", [64, 4096, 4097, 8192, 8193])
def test_product(cuda, k, mode):
    A, B = (x.to(cuda) for x in workloads.problem(40, 50, k, 0.5, seed=k))
    ws = torch.empty(ozk.workspace_size(40, 50, k, 12, mode=mode), dtype=torch.uint8, device=cuda)
    At, Bt = A.T.contiguous().T, B.T.contiguous().T
    for a, b in [(A, B), (A, Bt), (At, B), (At, Bt)]:
        counted, made = _launches(lambda: ozk.dgemm(a, b, num_moduli=12, mode=mode, workspace=ws))
        assert counted == made


@pytest.mark.parametrize("m,n", [(40, 50), (5000, 40), (40, 5000)])
def test_gradients(cuda, m, n):
    k, N = 60, 12
    A, B = (x.to(cuda) for x in workloads.problem(m, n, k, 0.5, seed=m))
    dC = workloads.normal_matrix(m, n, 3, cuda)
    fws = torch.empty(ozk.workspace_size(m, n, k, N), dtype=torch.uint8, device=cuda)
    ws = torch.empty(ozk.workspace_size_backward(m, n, k, N), dtype=torch.uint8, device=cuda)
    ozk.dgemm(A, B, num_moduli=N, workspace=fws)
    for need in ((True, True), (True, False), (False, True)):
        counted, made = _launches(lambda: ozk.dgemm_backward(A, B, dC, fws, N, *need, workspace=ws))
        assert counted == made
