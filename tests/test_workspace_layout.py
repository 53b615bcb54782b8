"""The workspace sizes of the documented layout, exactly, and the residue rows it holds, of a
multiple of 16 columns where they fit and of 8 where not.  Results in a workspace of exactly
that size equal those of the same product with zero columns added up to a multiple of 16,
bit for bit, and nothing past its end is written."""
import ctypes
import random

import pytest
import torch

from oracle import ozaki2 as oz


def _up(x, t):
    return (x + t - 1) // t * t


def _size(m, n, k, N, fast=False):
    kp, M = _up(k, 32), oz.num_digit_planes(N)
    parts = [256, 4 * m, 4 * n, 4 * m, 4 * n, 4 * m, 4 * n, m, n]
    parts += [4 * m * (kp // 32), 4 * n * (kp // 32)] if fast else [m * kp, n * kp]
    parts += [M * m * kp, M * n * kp, 2 * N * m * _up(n, 8)]
    return sum(_up(p, 256) for p in parts)


def test_sizes_of_the_layout():
    from paper_2603_10634_gb300 import _lib, build

    build.build()
    lib = _lib.load()
    rng = random.Random(7)
    shapes = [(1, 1, 1), (128, 8, 32), (100, 24, 999), (8192, 100, 4096), (16384, 16384, 16384)]
    shapes += [tuple(int(2 ** rng.uniform(0, 17)) for _ in range(3)) for _ in range(300)]
    for N in range(1, 21):
        for m, n, k in shapes:
            for mode in (0, 1):
                assert lib.ozk2_workspace_size_ex(m, n, k, N, mode, 0, 0) == _size(m, n, k, N, mode == 1), (m, n, k, N)
    # a product near the limit of ozk2_dgemm_noalloc (2^28 bytes)
    assert 0.98 * 2**28 < lib.ozk2_workspace_size(222000, 8, 32, 12) <= 2**28


CASES = [(130, 1, 40, 12), (257, 8, 300, 6), (64, 24, 16500, 12), (300, 100, 1000, 20), (1000, 40, 33000, 13),
         (1100, 1000, 3000, 12), (4100, 2056, 2500, 12), (2000, 2049, 16500, 14), (33, 7, 64, 1), (40, 250, 500, 9),
         (65, 40, 30, 8), (200, 8, 20, 12), (300, 24, 33, 20)]
FAST = [(257, 8, 300, 6), (300, 40, 100, 3), (700, 600, 20000, 5), (40000, 600, 480, 6), (90, 24, 30, 12)]


def _guarded(size, cuda):
    ws = torch.full((size + 4096,), 0x5A, dtype=torch.uint8, device=cuda)
    return ws, lambda: bool((ws[size:] == 0x5A).all())


@pytest.mark.gpu
@pytest.mark.parametrize("m,n,k,N,mode", [c + ("accurate",) for c in CASES] + [c + ("fast",) for c in FAST])
def test_ragged_rows(cuda, m, n, k, N, mode):
    import paper_2603_10634_gb300 as ozk
    from paper_2603_10634_gb300 import workloads

    A, B = workloads.problem(m, n, k, 1.0, seed=n, device=cuda)
    wide = torch.nn.functional.pad(B, (0, _up(n, 16) - n))
    for tile in (0, 128, 256):
        with ozk.tile_width(tile):
            want = ozk.dgemm(A, wide, num_moduli=N, mode=mode)[:, :n].contiguous()
            size = ozk.workspace_size(m, n, k, N, mode)
            ws, kept = _guarded(size, cuda)
            C = ozk.dgemm(A, B, num_moduli=N, mode=mode, workspace=ws[:size])
            assert torch.equal(C, want) and kept() and ozk.device_status(workspace=ws) == "OZK2_OK"
            with pytest.raises(ozk.Ozk2Error):
                ozk.dgemm(A, B, num_moduli=N, mode=mode, workspace=ws[:size - 256])
            plan = ozk.BatchPlan([A, wide.T.contiguous()], [B, A.T.contiguous()], num_moduli=N, mode=mode)
            assert torch.equal(plan.execute()[0], want)
    assert torch.equal(ozk.dgemm_host(A.cpu(), B.cpu(), num_moduli=N, mode=mode), want.cpu())


@pytest.mark.gpu
@pytest.mark.parametrize("m,n,k,N", [(300, 24, 100, 12), (129, 40, 1000, 13), (600, 1000, 520, 12)])
def test_ragged_gradients(cuda, m, n, k, N):
    import paper_2603_10634_gb300 as ozk
    from paper_2603_10634_gb300 import workloads

    A, B = workloads.problem(m, n, k, 1.0, seed=n, device=cuda)
    dC = workloads.normal_matrix(m, n, 5, cuda)

    def gradients(A, B, dC):
        m, k, n = *A.shape, B.shape[1]
        fws = torch.empty(ozk.workspace_size(m, n, k, N), dtype=torch.uint8, device=cuda)
        ozk.dgemm(A, B, num_moduli=N, workspace=fws)
        size = ozk.workspace_size_backward(m, n, k, N)
        ws, kept = _guarded(size, cuda)
        out = ozk.dgemm_backward(A, B, dC, fws, N, workspace=ws[:size])
        assert kept() and ozk.device_status(workspace=ws) == "OZK2_OK"
        return out

    pad = torch.nn.functional.pad
    kx, nx = _up(k, 16) - k, _up(n, 16) - n
    dA, dB = gradients(A, B, dC)
    wA, wB = gradients(pad(A, (0, kx)), pad(B, (0, nx, 0, kx)), pad(dC, (0, nx)))
    assert torch.equal(dA, wA[:, :k]) and torch.equal(dB, wB[:k, :n])


@pytest.mark.gpu
def test_noalloc_near_its_limit(cuda):
    import paper_2603_10634_gb300 as ozk
    from paper_2603_10634_gb300 import _lib, workloads

    m, n, k, N = 222000, 8, 32, 12
    A, B = workloads.problem(m, n, k, 1.0, seed=2, device=cuda)
    C = torch.empty((m, n), dtype=torch.float64, device=cuda)
    s = _lib.load().ozk2_dgemm_noalloc(m, n, k, ctypes.c_void_p(A.data_ptr()), k, ctypes.c_void_p(B.data_ptr()), n,
                                       ctypes.c_void_p(C.data_ptr()), n, N, ctypes.c_void_p(0))
    assert s == 0
    torch.cuda.synchronize()
    assert torch.equal(C, ozk.dgemm(A, B, num_moduli=N))
