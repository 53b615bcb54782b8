"""The scaling kernels over their ranges: rows held in registers by 1 to 8 warps (the row
lengths where that changes, and the longer rows read twice), aligned and unaligned rows,
the column kernels' partial maxima, and lines without a normal maximum, in both operand
forms, against the oracle."""
import numpy as np
import pytest
import torch

import paper_2603_10634_gb300 as ozk
from oracle import ozaki2 as oz
from paper_2603_10634_gb300 import workloads

pytestmark = pytest.mark.gpu


def _inputs(lines, k, seed):
    X = workloads.phi_matrix(lines, k, 1.5, seed).numpy()
    X[1 % lines] = 0.0
    X[2 % lines] *= 2.0**-1060  # mostly subnormal and zero entries
    X[3 % lines, k // 2] = np.inf
    X[4 % lines, -1] = np.nan
    X[5 % lines] = 2.0**-9 * np.arange(k)  # exact E4M3 values and subnormals of E4M3 below the maximum
    return X


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("k", [1, 63, 64, 65, 511, 512, 513, 1025, 2049, 4095, 4097, 8192, 8193])
def test_scaling_matches_the_oracle(cuda, k, offset):
    m, n = 9, 34
    A, Bt = _inputs(m, k, k), _inputs(n, k, k + 1)

    def oracle(X):
        X = np.where(np.isfinite(X), X, 0.0)
        ep = oz.prelim_exponent_rows(X)
        return np.where(np.any(X != 0, axis=1), ep, 0), oz.bound_operand(X, ep)

    (ea, bar_a), (eb, bar_b) = oracle(A), oracle(Bt)

    def padded(X):  # rows that start `offset` doubles past a 16-byte boundary
        full = torch.zeros((X.shape[0], X.shape[1] + 2 * offset), dtype=torch.float64)
        full[:, offset:offset + X.shape[1]] = torch.from_numpy(X)
        return full.to(cuda)[:, offset:offset + X.shape[1]]

    rows_a, rows_b = padded(A), padded(Bt)
    cols_a, cols_b = padded(np.ascontiguousarray(A.T)).T, padded(np.ascontiguousarray(Bt.T))
    for a, b in [(rows_a, cols_b), (cols_a, rows_b.T), (rows_a, rows_b.T), (cols_a, cols_b)]:
        sc = {key: v.cpu().numpy() for key, v in ozk.scales(a, b, num_moduli=12).items()}
        assert ozk.device_status() == "OZK2_ERR_NONFINITE"
        assert np.array_equal(sc["eprime"], ea) and np.array_equal(sc["fprime"], eb)
        assert np.array_equal(sc["Abar"][:, :k], bar_a) and not sc["Abar"][:, k:].any()
        assert np.array_equal(sc["BbarT"][:, :k], bar_b) and not sc["BbarT"][:, k:].any()
