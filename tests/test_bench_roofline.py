"""Host-side pieces of bench.py's roofline: what is left on the integer multiply
pipes when a column stage's BConv runs on the tensor cores, and the lanes that
a batch's operations share. CPU only."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_bconv_products_leave_the_integer_pipes():
    N = 1 << bench.LOG_N
    m = bench.kernel_models(40, 14)
    assert bench.converted_values("modup_cols", 40, 14) == 122 * N
    assert bench.converted_values("moddown_cols", 40, 14) == 80 * N
    assert bench.converted_values("rescale_cols", 40, 14) == 80 * N
    assert bench.converted_values("keymult", 40, 14) == 0
    w = bench.integer_pipe_work(m["modup_cols"], 122 * N)
    assert w["mac"] == 0 and w["bytes"] == m["modup_cols"]["bytes"]
    assert w["shoup"] == (40 + 122) * (N // 2) * 6 + 122 * N
    assert w["modmul"] == w["shoup"] + w["smr"]


@pytest.mark.parametrize("lanes,n,alpha,used", [(4, 40, 14, 2), (1, 40, 14, 1), (4, 2, 14, 4), (8, 4, 14, 5),
                                                (4, 40, 40, 2)])
def test_lanes_used(lanes, n, alpha, used):
    assert bench.lanes_used(lanes, n, alpha) == used
