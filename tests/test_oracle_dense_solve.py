"""The oracle's coarsest solve (dense LU with partial pivoting) is a solve:
one V-cycle of a one-level hierarchy gives A^-1 b, also where rows change
places (an exchange after a multiplier of an earlier column was formed moves
that multiplier with its row)."""
import numpy as np
import pytest

import oracle as O


@pytest.mark.parametrize("n", [1, 2, 3, 17, 128])
@pytest.mark.parametrize("seed", [0, 1])
def test_dense_coarse_solve_with_row_exchanges(n, seed):
    rng = np.random.default_rng(1000 * n + seed)
    A = rng.standard_normal((n, n)) + 0.1 * np.eye(n)
    b = rng.standard_normal(n)
    m = O.OracleAMG(np.arange(n + 1, dtype=np.int32) * n, np.tile(np.arange(n, dtype=np.int32), n),
                    A.reshape(-1), coarse_max=max(n, 1))
    assert len(m.levels()) == 1
    x = m.vcycle(b)
    # backward error of LU with partial pivoting: n eps growth, growth below 2^7 here
    assert np.abs(A @ x - b).max() <= 128 * n * 2.3e-16 * (np.abs(A).sum(1).max() *
                                                           np.abs(x).max() + np.abs(b).max())
