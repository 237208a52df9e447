"""LU solves of the FP64 recovery against the oracle: sizes around a warp, a
panel (32), the one-block kernel's limit and a column strip (128)."""
import numpy as np
import pytest

import lpgen
import oracle

from test_gpu_fp32 import _assert_matches_fp64, _run, tsx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 31, 32, 33, 64, 100, 160, 167, 168, 190, 193, 224, 225, 288, 289, 420])
def test_recovery_of_a_basis_of_k_structurals(tsx, k):   # noqa: F811
    A, b, c = lpgen.diag_dominant_lp(k, k, 40 + k)
    ref = oracle.solve(A, b, c)
    st, sol, _, _, _, stats = _run(tsx, A, b, c)
    assert st == tsx.LP_OPTIMAL == ref.status
    assert stats["k"] == int((ref.basis < k).sum()) and stats["cleanup_pivots"] == 0
    _assert_matches_fp64(A, b, c, sol, ref, tol=1e-11)


def test_rows_that_need_pivoting(tsx):   # noqa: F811
    # a permuted diagonal: the largest entry of every column lies off the diagonal
    A, b, c = lpgen.diag_dominant_lp(230, 230, 5)
    perm = np.random.default_rng(2).permutation(230)
    ref = oracle.solve(A[perm], b, c)
    st, sol, _, _, _, stats = _run(tsx, A[perm], b, c)
    assert st == tsx.LP_OPTIMAL == ref.status and stats["cleanup_pivots"] == 0
    _assert_matches_fp64(A[perm], b, c, sol, ref, tol=1e-11)


# more rows than one warp of a cluster block holds (k > 512), the largest entry of
# a column in any of them
@pytest.mark.parametrize("k", [513, 545, 1030])
def test_pivots_in_every_warp(tsx, k):   # noqa: F811
    A, b, c = lpgen.diag_dominant_lp(k, k, 7)
    A = A[np.random.default_rng(k).permutation(k)]
    st, sol, _, _, _, stats = _run(tsx, A, b, c)
    assert st == tsx.LP_OPTIMAL and stats["k"] == k and stats["cleanup_pivots"] == 0
    # cond(A) = 1.13; a stable solve errs by at most about k eps cond(A), both do
    x, y = np.linalg.solve(A, b), np.linalg.solve(A.T, c)
    assert np.abs(sol.x - x).max() <= 4 * k * 2.2e-16 * np.abs(x).max()
    assert np.abs(sol.y - y).max() <= 4 * k * 2.2e-16 * np.abs(y).max()


@pytest.mark.parametrize("k", [60, 166, 600])
def test_equal_candidates(tsx, k):   # noqa: F811
    # 2 x 2 blocks [[2, 2], [2, 1]] with their rows and columns spread out: every
    # column has two largest entries, in other warps and blocks.  x and y are whole
    # numbers, so the factors and the solves are exact.
    rng = np.random.default_rng(k)
    A = np.kron(np.eye(k // 2), [[2.0, 2.0], [2.0, 1.0]])[rng.permutation(k)][:, rng.permutation(k)]
    x, y = rng.integers(1, 9, k).astype(float), rng.integers(1, 9, k).astype(float)
    st, sol, _, _, _, stats = _run(tsx, A, A @ x, A.T @ y)
    assert st == tsx.LP_OPTIMAL and stats["k"] == k and stats["cleanup_pivots"] == 0
    np.testing.assert_array_equal(sol.x, x)
    np.testing.assert_array_equal(sol.y, y)
