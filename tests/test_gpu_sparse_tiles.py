"""The sparse streams where their work is cut: block counts just beside a warp's share of the bins (1024 blocks), a tile
(256), a lane's share (8), rows that start inside a tile, more tiles than one step of the scan takes.  Everything is
integer or bit work and compared exactly."""
import math

import numpy as np
import pytest

import oracle
from paper_2605_14929_b200 import binding as B
from paper_2605_14929_b200 import inputs as I

from .test_gpu_sparse import assert_opq, oracle_wr, run_opq, run_wr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K", [(1, 16), (1, 48), (255, 16), (257, 16), (41, 400), (1023, 16), (1025, 16), (3, 4096), (65, 1040)])
def test_streams_at_the_edges_of_tiles_and_shares(M, K):
    L = I.student_layer(7, 3, M, K, 32, 4.0)
    for q in (0.6, 1e-6):                              # a record or two per tile's block, and more than a tile keeps at hand
        m = B.opq_threshold(q, 16)
        assert_opq(run_opq(L.W, m), oracle.opq_extract(L.W, m))
        assert_opq(run_opq(L.W, m, capacity=M * K // 40), {**oracle.opq_extract(L.W, m), "records": oracle.opq_extract(L.W, m)["records"][:M * K // 40]})
    for fmt_name, rom in (("E5M6", ["NF4", "SH4"]), ("UE4M4", ["NF5", "SH5"])):
        fmt = I.scale_format(fmt_name)
        n_keep = math.ceil(0.03 * M * K)
        sw, out, got = run_wr(L, fmt, rom, n_keep, None)
        want = oracle_wr(L, fmt, out, sw, n_keep)
        assert got["count"] == want["count"] and got["scale_exp"] == want["scale_exp"]
        assert np.array_equal(got["row_start"], want["row_start"]) and np.array_equal(got["records"], want["records"])


def test_more_tiles_than_a_step_of_the_scan():
    """16400 tiles: the scan's second step starts from the first one's sum."""
    M, K = 8200, 8192
    L = I.laplace_outlier_layer(23, 3, M, K, 16)
    m = B.opq_threshold(0.92, 16)
    assert_opq(run_opq(L.W, m), oracle.opq_extract(L.W, m))
