"""Infinite and NaN entries beside the largest finite ones: they count as 0 in the bound
operands, so the other lines keep the exponents and results they have without them."""
import numpy as np
import pytest
import torch

import paper_2603_10634_gb300 as ozk
from paper_2603_10634_gb300 import workloads

pytestmark = pytest.mark.gpu

LARGE = [1.5 * 2.0**1023, 2.0**1023, np.finfo(np.float64).max, 2.0**1022, 1.0]


def _inputs(lines, k, seed):
    """Lines with a nonfinite entry beside one of LARGE, and the same with 0 in its place."""
    X = workloads.phi_matrix(lines, k, 1.0, seed).numpy()
    clean = X.copy()
    for i, big in enumerate(LARGE):
        for X_ in (X, clean):
            X_[i, 0] = -big if i & 1 else big
        X[i, k - 1] = [np.inf, -np.inf, np.inf, np.inf, -np.inf][i]
        clean[i, k - 1] = 0.0
    X[1, k // 2], clean[1, k // 2] = np.nan, 0.0
    return torch.from_numpy(X), torch.from_numpy(clean)


@pytest.mark.parametrize("mode", ["accurate", "fast"])
@pytest.mark.parametrize("k", [3, 512, 1000, 2000, 4096, 5000, 9000])
def test_nonfinite_entries_count_as_zero(cuda, k, mode):
    (A, A0), (Bt, B0t) = _inputs(9, k, k), _inputs(40, k, k + 1)
    rows = lambda X: X.to(cuda)  # noqa: E731
    cols = lambda X: X.T.contiguous().to(cuda).T  # noqa: E731
    for fa in (rows, cols):
        for fb in (rows, cols):
            got = ozk.scales(fa(A), fb(Bt).T, num_moduli=12, mode=mode)
            assert ozk.device_status() == "OZK2_ERR_NONFINITE"
            want = ozk.scales(fa(A0), fb(B0t).T, num_moduli=12, mode=mode)
            for key in want:
                if want[key] is not None:
                    assert torch.equal(got[key], want[key]), key


def test_finite_lines_of_a_batch(cuda):
    (A, A0), (Bt, B0t) = _inputs(9, 300, 1), _inputs(40, 300, 2)
    plans = [ozk.BatchPlan([a.to(cuda)], [b.T.contiguous().to(cuda)], num_moduli=12) for a, b in ((A, Bt), (A0, B0t))]
    got, want = (p.execute()[0].cpu() for p in plans)
    rows, cols = slice(len(LARGE), None), slice(len(LARGE), None)
    assert torch.equal(got[rows, cols], want[rows, cols]) and torch.isfinite(got[rows, cols]).all()
    assert torch.isnan(got[: len(LARGE)]).all() and torch.isnan(got[:, : len(LARGE)]).all()
