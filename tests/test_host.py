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
