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
