"""The residue system of the product path (csrc/rns.h) in exact arithmetic: its moduli,
digits, exactness blocks and CRT integer ranges.  The constants are read from the header;
the GPU parity tests check the kernels built from them."""
import os
import re

import numpy as np
import pytest
import torch

from oracle import ozaki2 as oz

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = open(os.path.join(ROOT, "paper_2603_10634_gb300", "csrc", "rns.h")).read()


def _list(name):
    return [int(x) for x in re.search(name + r"\[[^\]]*\]\s*=\s*\{([^}]*)\}", SRC).group(1).split(",")]


SINGLES, KARS, BETAS = _list("kSingleP"), _list("kKarP"), _list("kKarBeta")
NSINGLE, NKAR = _list("kRnsSingles"), _list("kRnsKars")
DIGITS = [d for a in range(33) if a <= 16 or a % 2 == 0 for d in {a, -a}]


def _product(xs):
    p = 1
    for x in xs:
        p *= int(x)
    return p


def test_moduli_are_coprime_and_cover_the_budget():
    every = SINGLES + KARS
    assert all(np.gcd(a, b) == 1 for i, a in enumerate(every) for b in every[:i])
    for N in range(1, 21):
        P = _product(oz.hybrid_moduli(N))
        P2 = _product(SINGLES[:NSINGLE[N]] + KARS[:NKAR[N]])
        assert 10 * P2 >= 11 * P, N
        # fewer products and planes than the hybrid list
        assert NSINGLE[N] + 3 * NKAR[N] < 3 * N and NSINGLE[N] + 3 * NKAR[N] <= oz.num_digit_planes(N), N


def test_every_residue_has_exact_digits():
    for d in DIGITS:  # exact in E4M3
        assert float(torch.tensor(float(d)).to(torch.float8_e4m3fn)) == d
    for p in SINGLES:
        assert {d % p for d in DIGITS} == set(range(p)), p
    for p, beta in zip(KARS, BETAS):
        ok = {(u + beta * v) % p for u in DIGITS for v in DIGITS if u + v in DIGITS}
        assert len(ok) == p, p
        # r r' = (1 - beta) uu' + (beta^2 - beta) vv' + beta (u + v)(u' + v')
        u, v, x, y = 5, -7, 12, 4
        assert ((u + beta * v) * (x + beta * y) - (1 - beta) * u * x - (beta * beta - beta) * v * y -
                beta * (u + v) * (x + y)) % p == 0


@pytest.mark.gpu
@pytest.mark.parametrize("N", [1, 2, 7, 8, 12, 13, 14, 15, 20])
@pytest.mark.parametrize("m,n,k", [(130, 258, 16384), (33, 17, 16385), (128, 256, 41856), (5, 300, 65665)])
def test_constant_lines_have_exact_products(cuda, N, m, n, k):
    """Every entry of row i of A is a_i and of column j of B is b_j, so all digits of a line
    are equal and the FP32 partial sums reach their largest magnitudes (k V^2 up to 2^24 at
    the edges of the exactness blocks).  C_ij = k a_i b_j is an integer below 2^53; it must
    be exact wherever N's scaling keeps the integers a_i, b_j whole (e_i, f_j >= 0)."""
    import paper_2603_10634_gb300 as ozk

    top = 2 ** min(17, max(1, 4 * N - 10))
    g = torch.Generator().manual_seed(N + k)
    a = torch.randint(-top, top + 1, (m, 1), generator=g).double()
    b = torch.randint(-top, top + 1, (1, n), generator=g).double()
    A, B = a.expand(m, k).contiguous().to(cuda), b.expand(k, n).contiguous().to(cuda)
    sc = ozk.scales(A, B, num_moduli=N)
    C = ozk.dgemm(A, B, num_moduli=N).cpu()
    whole = (sc["e"].cpu()[:, None] >= 0) & (sc["f"].cpu()[None, :] >= 0)
    assert torch.equal(C[whole], (k * a * b)[whole])
    if N >= 12:
        assert bool(whole.all())


@pytest.mark.gpu
@pytest.mark.parametrize("N", [2, 9, 12, 17, 20])
def test_unusual_elements_match_the_oracle(cuda, N):
    """Zeros of both signs, subnormals, entries far below and far above their line's
    neighbours (shifted out, or a' >= 2^53), in rows and in columns, bit for bit."""
    import paper_2603_10634_gb300 as ozk

    g = np.random.default_rng(N)
    m, n, k = 21, 18, 45
    special = np.array([0.0, -0.0, 5e-324, -3e-310, 2.0**-1022, 1.0, -2.0**-1000, 2.0**400, -1.5 * 2.0**60, 2.0**-60])
    A = np.where(g.random((m, k)) < 0.3, special[g.integers(0, len(special), (m, k))], g.standard_normal((m, k)))
    B = np.where(g.random((k, n)) < 0.3, special[g.integers(0, len(special), (k, n))], g.standard_normal((k, n)))
    A[0], B[:, 0] = 5e-324 * g.integers(0, 9, k), 2.0**-1030 * g.integers(-9, 9, k)  # subnormal lines
    A[1], B[:, 1] = 0.0, -0.0
    A[2] *= 2.0**-300
    Ad, Bd = torch.from_numpy(A).to(cuda), torch.from_numpy(B).to(cuda)
    sc = ozk.scales(Ad, Bd, num_moduli=N)
    C = ozk.dgemm(Ad, Bd, num_moduli=N).cpu().numpy()
    status = ozk.device_status()
    e, f = sc["e"].cpu().numpy(), sc["f"].cpu().numpy()
    want = oz.ozk2_dgemm(A, B, N, e=e, f=f)["C"]

    # an element whose significand would be scaled by 2^64 or more is out of the library's
    # range (possible for subnormal lines at large N): flagged, its line not compared
    def in_range(X, ex):
        lsb = np.maximum(np.frexp(X)[1] - 53, -1074)
        return ~((X != 0) & (lsb + ex[:, None] >= 64)).any(axis=1)

    ok = np.outer(in_range(A, e), in_range(B.T, f))
    assert status == ("OZK2_OK" if ok.all() else "OZK2_ERR_RANGE")
    assert np.array_equal(C.view(np.uint64)[ok], want.view(np.uint64)[ok])
    assert N > 12 or ok.all()
