"""Fast mode's sums of squares in a workspace that holds other values: every R and S must be
the call's own, in all operand forms, for device, blocked and host-buffer calls, with few
rows and with many more rows than columns."""
import numpy as np
import pytest
import torch

import paper_2603_10634_gb300 as ozk
from oracle import ozaki2 as oz
from paper_2603_10634_gb300 import workloads

pytestmark = pytest.mark.gpu


def _forms(A, B, cuda):
    """(A, B) on the device, each row-major and as a transposed view."""
    rows = lambda X: X.to(cuda)  # noqa: E731
    cols = lambda X: X.T.contiguous().to(cuda).T  # noqa: E731
    return [(a(A), b(B)) for a in (rows, cols) for b in (rows, cols)]


def _bits(x):
    return np.asarray(x.cpu().numpy()).view(np.uint64)


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (8, 40, 70), (700, 30, 40), (1920, 64, 33), (70, 900, 20)])
def test_sums_do_not_depend_on_the_workspace(cuda, m, n, k):
    N = 12
    A, B = workloads.problem(m, n, k, 1.0, seed=m + k)
    orc = oz.scaling_exponents(A.numpy(), B.numpy(), N, mode="fast")
    zr, zc = ~np.any(A.numpy() != 0, axis=1), ~np.any(B.numpy() != 0, axis=0)
    big = workloads.problem(512, 512, 2100, 1.0, seed=5)
    ws = torch.empty(ozk.workspace_size(m, n, k, N, mode="fast"), dtype=torch.uint8, device=cuda)
    for a, b in _forms(A, B, cuda):
        ozk.dgemm(big[0].to(cuda), big[1].to(cuda), num_moduli=N)  # other values in the library's workspace
        sc = {key: v.cpu().numpy() for key, v in ozk.scales(a, b, num_moduli=N, mode="fast").items()}
        for got, want in ((sc["R"], orc["R"]), (sc["S"], orc["S"])):
            g, o = got.astype(np.float64), want.astype(np.float64)
            assert np.all(g >= o) and np.all(g <= o * (1 + (k + 2) * 2.0**-23) + 2.0**-120)
        pp, d = orc["pprime"], orc["delta"]
        assert list(sc["e"]) == [oz.final_exponent(sc["eprime"][i], sc["R"][i], pp, d, zr[i]) for i in range(m)]
        assert list(sc["f"]) == [oz.final_exponent(sc["fprime"][j], sc["S"][j], pp, d, zc[j]) for j in range(n)]
        want = oz.ozk2_dgemm(A.numpy(), B.numpy(), N, e=sc["e"], f=sc["f"], mode="fast")["C"].view(np.uint64)
        for fill in (0x00, 0x7F, 0xFF):  # 0, 3.39e38 and NaN where R and S will lie
            ws.fill_(fill)
            C = ozk.dgemm(a, b, num_moduli=N, mode="fast", workspace=ws)
            assert np.array_equal(_bits(C), want)
            assert ozk.device_status(workspace=ws) == "OZK2_OK"
        ozk.dgemm(big[0].to(cuda), big[1].to(cuda), num_moduli=N)
        C = ozk.dgemm_host(a.cpu(), b.cpu(), num_moduli=N, mode="fast")
        assert np.array_equal(_bits(C), want)


def test_blocked_sums_do_not_depend_on_the_workspace(cuda):
    m, n, k, N, block = 300, 140, 90, 13, (128, 64)
    A, B = workloads.problem(m, n, k, 1.0, seed=3)
    A[:128] *= 2.0**40
    ws = torch.empty(ozk.workspace_size(m, n, k, N, mode="fast", block=block), dtype=torch.uint8, device=cuda)
    for a, b in _forms(A, B, cuda):
        ws.fill_(0x7F)
        C = ozk.dgemm(a, b, num_moduli=N, mode="fast", block=block, workspace=ws)
        for i in range(0, m, block[0]):
            for j in range(0, n, block[1]):
                own = ozk.dgemm(a[i:i + block[0]], b[:, j:j + block[1]], num_moduli=N, mode="fast")
                assert np.array_equal(_bits(C[i:i + block[0], j:j + block[1]].contiguous()), _bits(own)), (i, j)
