"""The integers of the product path, one modulus of its residue system (csrc/rns.h) at a time,
read from the workspace of a call:

* digit planes: every byte an E4M3 integer of magnitude at most 32, u + beta v (Karatsuba
  moduli, with w = u + v) or the digit itself (single moduli) congruent to a' mod p;
* residues: congruent to the exact product A'B' mod p, at most p / 2 + 1 in magnitude;
* CRT: each C the correctly rounded value of the integer that the residues determine."""
import numpy as np
import pytest
import torch

import paper_2603_10634_gb300 as ozk
from oracle import ozaki2 as oz
from paper_2603_10634_gb300 import workloads
from test_residue_system import BETAS, KARS, NKAR, NSINGLE, SINGLES

pytestmark = pytest.mark.gpu


def _view(ws, at, count, dtype):
    size = torch.empty(0, dtype=dtype).element_size()
    return ws[at:at + count * size].view(dtype)


def _run(A, B, N, mode, cuda, ta=False, tb=False):
    """C and, from its workspace, e, f, digit planes (planes x lines x k) and residues."""
    m, k, n = *A.shape, B.shape[1]
    ws = torch.empty(ozk.workspace_size(m, n, k, N, mode), dtype=torch.uint8, device=cuda)
    a, b = (x.T.contiguous().to(cuda).T if t else x.to(cuda) for x, t in ((A, ta), (B, tb)))
    C = ozk.dgemm(a, b, num_moduli=N, mode=mode, workspace=ws)
    at = ozk.workspace_layout(m, n, k, N, mode)
    planes, row, cols = ozk.product_count(N), at["plane_row"], at["res_columns"]

    def digits(start, lines):
        x = _view(ws, start, planes * lines * row, torch.float8_e4m3fn).view(planes, lines, row).float()
        assert not bool(x[:, :, k:].any())
        return x[:, :, :k].double()

    res16 = _view(ws, at["res16"], NKAR[N] * m * cols, torch.int16).view(NKAR[N], m, cols)[:, :, :n]
    res8 = _view(ws, at["res8"], NSINGLE[N] * m * cols, torch.int8).view(NSINGLE[N], m, cols)[:, :, :n]
    e, f = (_view(ws, at[key], lines, torch.int32).cpu().numpy() for key, lines in (("e", m), ("f", n)))
    return C, e, f, digits(at["planesA"], m), digits(at["planesB"], n), [*res16.double(), *res8.double()]


def _congruent(x, want, p):
    return bool((torch.remainder(x - want, p) == 0).all())


def _check(A, B, N, mode, cuda, ta=False, tb=False, known=None):
    """known: the residues of A' and B' by modulus, if they have been computed."""
    known = {} if known is None else known
    C, e, f, dA, dB, res = _run(A, B, N, mode, cuda, ta, tb)
    for d in (dA, dB):
        assert float(d.abs().max()) <= 32 and torch.equal(d, d.round())
    moduli = KARS[:NKAR[N]] + SINGLES[:NSINGLE[N]]
    plane = 0
    for l, p in enumerate(moduli):
        if p not in known:
            known[p] = [torch.from_numpy(oz.scaled_residues_rows(X, ex, p)).double().to(cuda)
                        for X, ex in ((A.numpy(), e), (B.numpy().T, f))]
        ra, rb = known[p]
        for d, r in ((dA, ra), (dB, rb)):
            if l < NKAR[N]:
                u, v, w = d[plane:plane + 3]
                assert torch.equal(u + v, w) and _congruent(u + BETAS[l] * v, r, p), (l, p)
            else:
                assert _congruent(d[plane], r, p), (l, p)
        plane += 3 if l < NKAR[N] else 1
        # exact in double: |r| <= p / 2, so every sum stays below k 642^2 < 2^53
        assert _congruent(res[l], ra @ rb.T, p), (l, p)
        assert float(res[l].abs().max()) <= p // 2 + 1, (l, p)
    assert plane == ozk.product_count(N) == dA.shape[0]
    return C, e, f, res, moduli


@pytest.mark.parametrize("N", range(1, 21))
@pytest.mark.parametrize("mode", ["accurate", "fast"])
def test_every_modulus_and_the_crt(cuda, N, mode):
    m, n, k = 33, 20, 141
    A, B = workloads.problem(m, n, k, 1.0, seed=N)
    A[3, 5:] *= 2.0**-30
    A[4] = 0.0
    A[5] *= 2.0**-1040
    B[:, 2] *= 2.0**300
    B[7, 3] = 2.0**40
    C, e, f, res, moduli = _check(A, B, N, mode, cuda)
    P2 = 1
    for p in moduli:
        P2 *= p
    x = np.zeros((m, n), dtype=object)
    for r, p in zip(res, moduli):
        c = np.array([[int(v) for v in row] for row in r.cpu().numpy()], dtype=object)
        x += c * ((P2 // p) * pow(P2 // p, -1, p))
    x = np.vectorize(lambda v: (v + P2 // 2) % P2 - P2 // 2, otypes=[object])(x)
    want = np.array([[oz.round_scaled_to_double(int(x[i, j]), int(e[i]) + int(f[j])) for j in range(n)] for i in range(m)])
    assert np.array_equal(C.cpu().numpy().view(np.uint64), want.view(np.uint64))


# edges of tiles, of 8- and 16-column pieces and of the exactness blocks; wide, narrow and paired tiles
@pytest.mark.parametrize("m,n,k,N,mode", [(130, 257, 129, 12, "accurate"), (129, 72, 16384, 13, "accurate"),
                                          (64, 130, 16385, 20, "fast"), (40, 24, 33000, 12, "accurate"),
                                          (520, 768, 2100, 12, "accurate"), (280, 264, 16500, 14, "accurate"),
                                          (20, 26, 65600, 7, "fast"), (1, 1, 70000, 16, "accurate")])
def test_shapes(cuda, m, n, k, N, mode):
    A, B = workloads.problem(m, n, k, 2.0, seed=m + n)
    known = {}
    for tile in (0, 128, 256):
        with ozk.tile_width(tile):
            _check(A, B, N, mode, cuda, m % 3 == 1, n % 4 == 2, known)
