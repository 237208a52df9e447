"""The library's host side on a fake CUDA runtime (no GPU; see fakecuda)."""
import shutil

import pytest

import fakecuda

pytestmark = pytest.mark.skipif(not (shutil.which("nvcc") or shutil.which("/usr/local/cuda/bin/nvcc")),
                                reason="needs nvcc")


# 300 x 300: k_pivot_delayed, 1000 x 1000: k_pivot_overlap
@pytest.mark.parametrize("m,kernel", [(300, "k_pivot_delayed"), (1000, "k_pivot_overlap")])
def test_a_block_that_gave_up_is_a_timeout(m, kernel):
    # a block whose last wait ran out has left its right-hand sides and objective
    # entries unstored, whatever status block 0 has written meanwhile
    fakecuda.run(f"""
    for status in (tsx.LP_OPTIMAL, tsx.LP_UNBOUNDED, tsx.LP_ITER_LIMIT):
        fake.fake_reset()
        fake.fake_plan(status, 1, 0)
        st, stats = solve({m}, {m}, path=1)
        assert "{kernel}" in kernels()
        assert st == tsx.LP_ERR_TIMEOUT == stats["pivot_status"], (status, st)
        assert "wait" in tsx.lp_last_error()
    fake.fake_plan(0, 1, 0)
    assert solve({m}, {m}, path=1, precision=tsx.LP_PREC_FP32)[0] == tsx.LP_ERR_TIMEOUT
    fake.fake_plan(0, 0, 0)
    assert solve({m}, {m}, path=1)[0] == tsx.LP_OPTIMAL
    """)


def test_a_second_device_runs_the_same_kernels():
    # kernel attributes (shared memory, cluster size) belong to a device
    fakecuda.run("""
    def calls(device):
        fake.fake_reset()
        fake.fake_plan(0, 0, 100)
        st = [solve(300, 300, device, precision=tsx.LP_PREC_FP32)[0]]       # one-block LU, 86 KB
        fake.fake_plan(0, 0, 400)
        st.append(solve(500, 500, device, precision=tsx.LP_PREC_FP32)[0])   # panels: clusters of 16
        fake.fake_plan(0, 0, 0)
        for m, kw in ((256, {}), (600, {}), (300, {"path": 1}), (1000, {}), (300, {"threads": 128, "path": 1}),
                      (300, {"layout": tsx.LP_LAYOUT_FULL})):
            st.append(solve(m, m, device, **kw)[0])
        for precision in (tsx.LP_PREC_FP64, tsx.LP_PREC_FP32):
            prs = [tsx.Problem(*lp(300, 300)) for _ in range(3)]
            st += tsx.solve_many(prs, tsx.options(precision=precision))
            for pr in prs: pr.close()
        with tsx.Batch([lp(120, 120)] * 3) as b:
            b.solve(tsx.batch_options(threads=128))
        assert set(st) == {tsx.LP_OPTIMAL}, (device, st, tsx.lp_last_error())
        assert all(x[1] == device for x in log()), log()
        return sorted((x[0],) + x[2:] for x in log())   # (recoveries run on several threads)
    first = calls(0)
    names = [x[0] for x in first]
    for k in ("k_rec_lu_small", "k_lu_panel", "k_lu_solve", "k_cluster_solve", "k_pivot_delayed", "k_pivot_overlap",
              "k_pivot_persistent", "k_team_solve", "k_batch_solve"):
        assert k in names, (k, names)
    for device in (1, 2, 70):   # 70: beyond the table of devices
        assert calls(device) == first
    assert calls(0) == first
    """)


def test_a_refused_launch_takes_the_next_kernel():
    fakecuda.run("""
    fake.fake_refuse(b"k_pivot_overlap")
    st, stats = solve(1000, 1000)
    assert kernels()[-2:] == ["refused k_pivot_overlap", "k_pivot_delayed"], kernels()
    assert st == tsx.LP_OPTIMAL and stats["path"] == tsx.LP_PATH_PERSISTENT and stats["block"] == 256
    assert stats["update_bytes"] > 0
    fake.fake_reset()
    fake.fake_refuse(b"k_pivot_")   # none of them: one launch per phase
    st, stats = solve(1000, 1000)
    assert kernels()[4:7] == ["refused k_pivot_overlap", "refused k_pivot_delayed", "k_ml_init"], kernels()
    assert st == tsx.LP_OPTIMAL and stats["path"] == tsx.LP_PATH_MULTILAUNCH and stats["block"] == 256
    with tsx.Problem(*lp(1000, 1000)) as pr:
        assert tsx.lp_solve(pr.h, tsx.options(path=tsx.LP_PATH_PERSISTENT)) == tsx.LP_ERR_CUDA
        fake.fake_reset()
        assert pr.solve(tsx.options(path=tsx.LP_PATH_PERSISTENT)) == tsx.LP_OPTIMAL
        assert kernels()[-1] == "k_pivot_overlap" and pr.stats()["block"] == 512
    """)


# what a request holds on the device against the server's account of it: long rows
# (the delayed updates' buffers outweigh the vectors) and a tableau with a second
# copy (passes behind the pivots), solved by the lane, by waves and one at a time
@pytest.mark.parametrize("m,n,precision", [(16, 20000, 0), (16, 20000, 1), (20000, 16, 0), (1100, 1000, 0),
                                           (300, 75000, 1)])
@pytest.mark.parametrize("how", [{}, {"continuous": 0}, {"team_blocks": -1, "path": 0}, {"team_blocks": -1}])
def test_a_request_holds_no_more_than_the_server_counts(m, n, precision, how):
    fakecuda.run(f"""
    import time
    for k in (0, 16):
        with tsx.Server(workers=1, batch_small=0, precision={precision}, **{how}) as sv:
            fake.fake_reset()
            fake.fake_plan(0, 0, k)
            before = fake.fake_live()
            t = sv.submit(*lp({m}, {n}))
            assert sv.wait(t, 60.0) == tsx.LP_OPTIMAL, sv.last_error()
            held, counted = fake.fake_peak() - before, sv.stats()["peak_bytes"]
            assert 0 < held <= counted, (held, counted, kernels())
    """)


def test_a_budget_without_room_for_a_second_copy():
    # still solved, in one copy of the tableau and within the budget
    fakecuda.run("""
    one, two = 20 << 20, 40 << 20
    for budget, kernel in ((one, "k_pivot_delayed"), (two, "k_pivot_overlap")):
        with tsx.Server(workers=1, batch_small=0, precision=tsx.LP_PREC_FP64, team_blocks=-1, path=0,
                        budget_bytes=budget) as sv:
            fake.fake_reset()
            before = fake.fake_live()
            t = sv.submit(*lp(1100, 1000))
            assert sv.wait(t, 60.0) == tsx.LP_OPTIMAL, sv.last_error()
            assert kernel in kernels(), kernels()
            assert fake.fake_peak() - before <= sv.stats()["peak_bytes"] <= budget
    """)


def test_a_certain_cleanup_starts_from_the_inverse():
    # after a capped or unbounded float phase the checks fail for certain, and the
    # cleanup pivots need the explicit inverse: no LU before it
    fakecuda.run("""
    for status, inverse in ((tsx.LP_ITER_LIMIT, True), (tsx.LP_UNBOUNDED, True), (tsx.LP_OPTIMAL, False)):
        for k, m in ((100, 300), (400, 500)):
            fake.fake_reset()
            fake.fake_plan(status, 0, k)
            assert solve(m, m, precision=tsx.LP_PREC_FP32)[0] == tsx.LP_OPTIMAL
            prs = [tsx.Problem(*lp(m, m)) for _ in range(2)]
            assert tsx.solve_many(prs, tsx.options(precision=tsx.LP_PREC_FP32)) == [tsx.LP_OPTIMAL] * 2
            for pr in prs: pr.close()
            names = kernels()
            assert ("k_rec_gj_inplace" in names) == inverse, (status, k, names)
            assert any("_lu_" in x for x in names) != inverse, (status, k, names)
    """)


# 700 x 500: a cluster block would hold more than 15000 entries, and the grid is
# faster where it may use all of its blocks
@pytest.mark.parametrize("blocks,cluster", [(0, False), (1, True), (16, True), (76, True), (151, True), (152, False)])
def test_a_capped_grid_does_not_take_a_clusters_place(blocks, cluster):
    fakecuda.run(f"""
    st, stats = solve(700, 500, blocks={blocks})
    assert st == tsx.LP_OPTIMAL
    assert stats["path"] == (tsx.LP_PATH_CLUSTER if {cluster} else tsx.LP_PATH_PERSISTENT), stats
    """)


# blocks of a delayed solve (152 SMs): as few as cost a solve alone next to
# nothing, so that solves of several threads run side by side
@pytest.mark.parametrize("m,n,precision,most,least", [
    (300, 300, 0, 30, 24), (400, 400, 0, 50, 38), (512, 512, 0, 76, 64), (700, 500, 0, 76, 64), (700, 700, 0, 152, 152),
    (1000, 1000, 0, 152, 152), (48, 48, 0, 13, 1), (256, 256, 1, 30, 24), (1069, 42, 0, 30, 24), (4062, 42, 0, 76, 64), (700, 700, 1, 30, 16), (1000, 1000, 1, 50, 32),
    (1500, 1400, 1, 76, 64), (2000, 2000, 1, 152, 152), (3000, 100, 1, 50, 25), (33, 16384, 1, 152, 100)])
def test_small_solves_leave_room_for_others(m, n, precision, most, least):
    fakecuda.run(f"""
    st, stats = solve({m}, {n}, precision={precision}, path=1)
    assert st == tsx.LP_OPTIMAL and {least} <= stats["grid"] <= {most}, stats["grid"]
    st, stats = solve({m}, {n}, precision={precision}, path=1, blocks=5)
    assert stats["grid"] == 5
    """)


def test_wide_teams_start_with_their_own_lps():
    # the heavy list's counter starts behind the wide teams' first LPs
    fakecuda.run("""
    for count, blocks in ((5, 1), (5, 2), (3, 0), (1, 0), (400, 1)):
        prs = [tsx.Problem(*lp(100, 90 + 10 * (k < 3))) for k in range(count)]
        assert tsx.solve_many(prs, tsx.options(blocks=blocks)) == [tsx.LP_OPTIMAL] * count
        for pr in prs: pr.close()
        nxt = list((ctypes.c_uint * 2).in_dll(fake, "fake_team_next"))
        wide = ctypes.c_int.in_dll(fake, "fake_team_wide").value
        assert nxt == [0, wide] and (wide > 0 or count == 400), (count, blocks, nxt, wide)
    """)


def test_an_idle_lane_makes_room_for_a_batch_that_waits_for_it():
    # the lane's launch would stay for 3 s; a micro-batch whose blocks do not fit
    # beside it is done long before, and later requests start a new launch
    fakecuda.run("""
    import time
    lane_ms = ctypes.c_int.in_dll(fake, "fake_lane_ms")
    lane_ms.value = 3000
    with tsx.Server(workers=1, precision=tsx.LP_PREC_FP64) as sv:
        def ask(m, n):
            t = sv.submit(*lp(m, n))
            t0 = time.perf_counter()
            assert sv.wait(t, 60.0) == tsx.LP_OPTIMAL, sv.last_error()
            sv.result(t)
            return time.perf_counter() - t0
        for launches in (1, 2, 3):
            ask(300, 260)                       # the lane's
            assert ask(64, 48) < 0.5            # a micro-batch beside it: the launch stays
            assert ask(300, 260) < 0.5 and sv.stats()["lane_launches"] == launches
            fake.fake_batch_waits(1)
            assert ask(64, 48) < 0.5, launches
            fake.fake_batch_waits(0)
        lane_ms.value = 0
        assert sv.stats()["batches"] == 6
    """)


def test_a_short_list_gives_every_lp_a_team():
    fakecuda.run("""
    def teams(shapes, **kw):
        prs = [tsx.Problem(*lp(m, n)) for m, n in shapes]
        assert tsx.solve_many(prs, tsx.options(**kw)) == [tsx.LP_OPTIMAL] * len(shapes)
        for pr in prs: pr.close()
        return [x for x in (ctypes.c_int * 512).in_dll(fake, "fake_team_size") if x]
    assert teams([(1000, 1000)] * 8) == [38] * 8                       # 304 blocks
    assert teams([(1000, 1000)] * 8, blocks=16) != [38] * 8            # the caller's team size
    assert teams([(1000, 1000)] * 14) == [21] * 14
    assert 64 in teams([(1000, 1000)] * 15)                            # little of the GPU is left
    assert 64 in teams([(1000, 1000)] * 8, precision=tsx.LP_PREC_FP32)
    assert teams([(200, 200)] * 2) == [30, 30]                         # more would not shorten them
    mixed = teams([(300, 300), (1200, 1100), (600, 500)])              # largest first
    assert mixed == sorted(mixed, reverse=True) and 16 <= mixed[2] and sum(mixed) <= 304 and mixed[0] > 100
    assert sum(teams([(900 + 40 * k, 800) for k in range(11)])) <= 304
    assert max(teams([(1400, 1400)])) <= 160
    """)
