"""The cluster kernel's 512-thread build, its quotients from a reciprocal, and
the line between the cluster and the grid-wide kernel, against the oracle
(tolerance 0)."""
import numpy as np
import pytest

import lpgen

from test_gpu_parity import _assert_same, _gpu_run, _oracle_run, tsx  # noqa: F401

pytestmark = pytest.mark.gpu


# 16 rows of 249 and 250 entries a block: the line of the wider build; above 600
# rows or columns: the grid from 15000 entries a block on (600 x 600, 22838 of
# them, stays on the cluster)
@pytest.mark.parametrize("m,n,cluster", [(256, 248, True), (256, 249, True), (600, 600, True), (601, 394, False),
                                         (601, 380, True), (384, 601, True), (400, 601, False), (700, 500, False),
                                         (2000, 64, True)])
def test_route_and_bits(tsx, m, n, cluster):   # noqa: F811
    A, b, c = lpgen.dense_lp(m, n, 3)
    run = _gpu_run(tsx, A, b, c)
    _assert_same(run, _oracle_run(A, b, c))
    assert run[5]["path"] == (tsx.LP_PATH_CLUSTER if cluster else tsx.LP_PATH_PERSISTENT)


@pytest.mark.parametrize("seed", range(6))
def test_quotients_of_zeros_and_extremes(tsx, seed):   # noqa: F811
    # pivot rows with zeros and with entries far outside the reciprocal's range
    rng = np.random.default_rng(seed)
    A, b, c = lpgen.dense_lp(70, 50, seed)
    A[rng.random(A.shape) < 0.5] = 0.0
    A *= 2.0 ** rng.integers(-520, 500, (70, 1))
    b *= A.max(axis=1) + 1e-300
    A[:, rng.integers(50, size=5)] *= 2.0 ** -40
    for kw in ({}, {"eps_p": 0.0}):
        _assert_same(_gpu_run(tsx, A, b, c, path=tsx.LP_PATH_CLUSTER, **kw), _oracle_run(A, b, c, **kw))
