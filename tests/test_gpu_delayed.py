"""Delayed updates (the condensed tableau's persistent path): up to 16 (FP32:
32) pivots share one pass over the tableau.

Every entry takes the undelayed update's fused multiply-adds in the same order,
so the tableau, the pivots and the results equal the oracle's, and where entries
overflow the undelayed condensed path's, entry for entry (tolerance 0).
"""
import numpy as np
import pytest

import lpgen
import oracle

from test_gpu_parity import _assert_same, _gpu_run, _oracle_run, tsx  # noqa: F401

pytestmark = pytest.mark.gpu


# columns around a strip (128 doubles, 256 floats) and a 32-byte group, rows
# around a tile (8); pivots around a round (16, 32); and one block, whose own
# rows and columns do not fit its shared memory
SHAPES = [(8, 127), (9, 128), (7, 129), (255, 257), (63, 1021)]


@pytest.mark.parametrize("m,n", SHAPES)
@pytest.mark.parametrize("k", [1, 15, 16, 17, 33, -1])
def test_rounds_and_remainders(tsx, m, n, k):   # noqa: F811
    A, b, c = lpgen.diag_dominant_lp(m, n, 3 + m)   # about min(m, n) pivots or more
    ref = _oracle_run(A, b, c, max_iters=k)
    _assert_same(_gpu_run(tsx, A, b, c, path=1, max_iters=k), ref)


@pytest.mark.parametrize("m,n", [(9, 255), (40, 257), (257, 300)])
def test_float_rounds(tsx, m, n):   # noqa: F811
    A, b, c = lpgen.diag_dominant_lp(m, n, 5 + m)
    st32, it32, qref, pref, Tref, _ = oracle.solve32(A, b, c)
    _, _, T, q, p, stats = _gpu_run(tsx, A, b, c, path=1, precision=tsx.LP_PREC_FP32)
    assert stats["pivot_status"] == st32 and stats["iters"] == it32
    np.testing.assert_array_equal(q, qref)
    np.testing.assert_array_equal(p, pref)
    np.testing.assert_array_equal(T, Tref.astype(np.float64))


@pytest.mark.parametrize("blocks", [1, 3])
@pytest.mark.parametrize("threads", [128, 256, 512])
def test_parts_that_do_not_fit_shared_memory(tsx, blocks, threads):   # noqa: F811
    A, b, c = lpgen.dense_lp(1900, 700, 3)
    ref = _oracle_run(A, b, c, max_iters=40)
    _assert_same(_gpu_run(tsx, A, b, c, path=1, max_iters=40, blocks=blocks, threads=threads), ref)


@pytest.mark.parametrize("kw", [{"k_cyc": 3}, {"rule": 1}])
def test_rules_with_pending_updates(tsx, kw):   # noqa: F811
    A0, b0, c0 = lpgen.dense_lp(60, 45, 11)
    A = np.vstack([A0, A0[:20], np.ones((3, 45))])
    b = np.concatenate([b0, b0[:20], np.full(3, 50.0)])
    _assert_same(_gpu_run(tsx, A, b, c0, path=1, **kw), _oracle_run(A, b, c0, **kw))


# LPs whose scaled pivot row overflows after some pivots, with pivots after it
# (a row of tiny entries and b = 0: the pivot element is ~1e-300); the last
# pivot count stops right at the overflow
@pytest.mark.parametrize("seed,first", [(10, 5), (147, 3), (183, 5), (336, 5)])
def test_overflow_ends_a_round(tsx, seed, first):   # noqa: F811
    rng = np.random.default_rng(seed)
    A, b, c = lpgen.dense_lp(20, 15, seed)
    A = A - 3.0
    i = int(rng.integers(20))
    b[i] = 0.0
    A[i] *= 10.0 ** -rng.integers(290, 308)
    A[i][rng.integers(15)] = 5
    for k in (first, -1):
        one = _gpu_run(tsx, A, b, c, path=1, eps_p=0.0, max_iters=k)
        ref = _gpu_run(tsx, A, b, c, path=2, eps_p=0.0, max_iters=k)
        assert not np.isfinite(ref[2]).all()
        assert one[0] == ref[0] and one[1].iters == ref[1].iters
        for x, y in zip((one[1].x, one[1].y, one[1].basis, *one[2:5]), (ref[1].x, ref[1].y, ref[1].basis, *ref[2:5])):
            np.testing.assert_array_equal(x, y)
        assert one[1].obj == ref[1].obj or (np.isnan(one[1].obj) and np.isnan(ref[1].obj))


# LPs large enough for passes that run behind the pivots (rounds of 8 pivots in
# FP64): against the oracle, and in FP32 and with overflowing entries against
# the passes in turn (threads given) and the undelayed path
@pytest.mark.parametrize("m,n", [(1100, 1000), (2000, 640), (640, 2000)])
@pytest.mark.parametrize("kw", [{"max_iters": 1}, {"max_iters": 8}, {"max_iters": 9}, {"max_iters": 40}, {},
                                {"rule": 1, "max_iters": 30}])
def test_overlapped_passes(tsx, m, n, kw):   # noqa: F811
    A, b, c = lpgen.dense_lp(m, n, 9)
    _assert_same(_gpu_run(tsx, A, b, c, path=1, **kw), _oracle_run(A, b, c, **kw))


def test_overlapped_passes_revisit_rows_and_columns(tsx):   # noqa: F811
    # many ties and degenerate pivots: rows and column slots come back within a round
    rng = np.random.default_rng(4)
    A = rng.integers(1, 4, (1050, 1000)).astype(float)
    b = rng.integers(0, 3, 1050).astype(float)
    c = rng.integers(1, 4, 1000).astype(float)
    for kw in ({"max_iters": 60}, {"k_cyc": 3, "max_iters": 120}):
        _assert_same(_gpu_run(tsx, A, b, c, path=1, **kw), _oracle_run(A, b, c, **kw))


def test_overlapped_passes_in_float(tsx):   # noqa: F811
    A, b, c = lpgen.dense_lp(300, 75000, 2)
    one = _gpu_run(tsx, A, b, c, precision=tsx.LP_PREC_FP32, path=1)
    ref = _gpu_run(tsx, A, b, c, precision=tsx.LP_PREC_FP32, path=1, threads=256)
    assert one[5]["iters"] == ref[5]["iters"] > 33
    for x, y in zip((one[1].x, one[1].y, *one[2:5]), (ref[1].x, ref[1].y, *ref[2:5])):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("seed,first", [(10, 5), (147, 3), (183, 5), (336, 5)])
def test_overlapped_passes_overflow(tsx, seed, first):   # noqa: F811
    rng = np.random.default_rng(seed)
    A0, b0, c0 = lpgen.dense_lp(20, 15, seed)
    A0 = A0 - 3.0
    i = int(rng.integers(20))
    b0[i] = 0.0
    A0[i] *= 10.0 ** -rng.integers(290, 308)
    A0[i][rng.integers(15)] = 5
    A = np.full((1010, 1000), 1e-3)   # around it: rows that never leave, columns that never enter
    A[:20, 15:] = 0.0
    A[:20, :15] = A0
    b = np.concatenate([b0, np.full(990, 1e6)])
    c = np.concatenate([c0, np.full(985, -1.0)])
    for k in (first, -1):
        one = _gpu_run(tsx, A, b, c, path=1, eps_p=0.0, max_iters=k)
        ref = _gpu_run(tsx, A, b, c, path=2, eps_p=0.0, max_iters=k)
        assert not np.isfinite(ref[2]).all()
        assert one[0] == ref[0] and one[1].iters == ref[1].iters
        for x, y in zip((one[1].x, one[1].y, one[1].basis, *one[2:5]), (ref[1].x, ref[1].y, ref[1].basis, *ref[2:5])):
            np.testing.assert_array_equal(x, y)


def test_overlapped_passes_time_out(tsx):   # noqa: F811
    A, b, c = lpgen.dense_lp(1100, 1000, 1)
    with tsx.Problem(A, b, c) as pr:
        assert tsx.lp_solve(pr.h, tsx.options(path=1, barrier_timeout_ns=0)) == tsx.LP_ERR_TIMEOUT
        assert pr.solve(tsx.options(path=1, max_iters=20)) == tsx.LP_ITER_LIMIT
        np.testing.assert_array_equal(pr.tableau(), _oracle_run(A, b, c, max_iters=20).T)


# limits around the length of a wait: a solve either times out or is right
@pytest.mark.parametrize("m,n", [(300, 260), (1100, 1000)])
def test_waits_that_run_out_late(tsx, m, n):   # noqa: F811
    A, b, c = lpgen.dense_lp(m, n, 6)
    ref = _oracle_run(A, b, c, max_iters=3)
    with tsx.Problem(A, b, c) as pr:
        for ns in list(range(600, 12000, 600)) * 10 + [10 ** 9]:
            st = pr.solve(tsx.options(path=1, max_iters=3, barrier_timeout_ns=ns))
            assert st == tsx.LP_ERR_TIMEOUT and ns < 10 ** 9 or st == tsx.LP_ITER_LIMIT
            if st == tsx.LP_ITER_LIMIT:
                sol = pr.solution()
                assert sol.iters == 3 and sol.obj == ref.obj
                np.testing.assert_array_equal(sol.x, ref.x)
                np.testing.assert_array_equal(sol.y, ref.y)


def test_many_with_a_large_lp(tsx):   # noqa: F811
    # an FP64 LP above 4e6 entries that would outlast its list is solved on the
    # whole grid
    shapes = [(300, 200), (2100, 1950), (700, 300)]
    problems = [lpgen.dense_lp(m, n, 20 + k) for k, (m, n) in enumerate(shapes)]
    refs = [oracle.solve(*p) for p in problems]
    for blocks, large in ((0, tsx.LP_PATH_PERSISTENT), (16, tsx.LP_PATH_TEAM)):
        prs = [tsx.Problem(*p) for p in problems]
        try:
            assert tsx.solve_many(prs, tsx.options(blocks=blocks)) == [r.status for r in refs]
            for pr, ref, path in zip(prs, refs, (tsx.LP_PATH_TEAM, large, tsx.LP_PATH_TEAM)):
                sol = pr.solution()
                assert sol.iters == ref.iters and sol.obj == ref.obj and pr.stats()["path"] == path
                np.testing.assert_array_equal(sol.x, ref.x)
                np.testing.assert_array_equal(sol.y, ref.y)
        finally:
            for pr in prs:
                pr.close()


@pytest.mark.parametrize("count,on_grid", [(14, False), (13, True)])
def test_many_large_lps_by_their_share(tsx, count, on_grid):   # noqa: F811
    # equal LPs above 4e6 entries: each is 1 / count of the list, and goes to the
    # grid where that is above 0.35 of what a wide team (64 of 304 blocks) gets
    # through meanwhile, 0.0737 of it
    A, b, c = lpgen.dense_lp(2050, 1960, 40)
    prs = [tsx.Problem(A, b, c) for _ in range(count)]
    try:
        assert prs[0].solve() == tsx.LP_OPTIMAL
        alone = prs[0].solution()
        assert tsx.solve_many(prs) == [tsx.LP_OPTIMAL] * count
        for pr in prs:
            assert pr.stats()["path"] == (tsx.LP_PATH_PERSISTENT if on_grid else tsx.LP_PATH_TEAM)
            sol = pr.solution()
            assert sol.iters == alone.iters and sol.obj == alone.obj
            np.testing.assert_array_equal(sol.x, alone.x)
            np.testing.assert_array_equal(sol.y, alone.y)
    finally:
        for pr in prs:
            pr.close()
