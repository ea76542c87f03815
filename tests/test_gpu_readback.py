"""The ends of a call (csrc/rips_api.cu): results around the 2048 bars that one
block puts in order, with the bound on their number above and below that, and
sparse inputs whose edge count has too many bits for the sort keys while the
number of distinct lengths has not."""
import math

import numpy as np
import pytest

from paper_1908_02518_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _key(bars):
    none = np.iinfo(np.uint64).max
    return [(int(b["dim"]), float(b["birth"]), float(b["death"]), int(b["birth_simplex"]),
             int(none) if int(b["death_simplex"]) < 0 else int(b["death_simplex"])) for b in bars]


@pytest.mark.parametrize("n,dim_max,t", [(1, 0, math.inf), (2047, 0, math.inf), (2048, 0, math.inf),
                                         (2049, 0, math.inf), (33, 1, math.inf), (700, 1, 0.3), (1500, 1, 0.15),
                                         (2040, 1, 0.05)])
def test_order_and_bars(oracle_mod, n, dim_max, t):
    import torch
    import paper_1908_02518_gb300 as rg
    d = W.distance_matrix(W.cube_points(n, 11))
    got = _key(rg.barcodes(torch.from_numpy(d).cuda(), dim_max, t).bars)
    assert [g[:4] for g in got] == sorted(g[:4] for g in got)
    assert sorted(got) == sorted(_key(oracle_mod.barcodes(d, dim_max, t).bars))


@pytest.mark.parametrize("squares", [3, 700])
def test_many_edges_of_few_lengths(squares):
    """Squares among 20000 points, each with one longer side: C(20000, 4) takes 53
    bits, the 2800 edges 12 and their two lengths 1; each square is a class born
    at the longer side that never dies."""
    import paper_1908_02518_gb300 as rg
    n = 20000
    a = 4 * np.arange(squares, dtype=np.int32)
    i = np.concatenate([a, a + 1, a + 2, a + 3])
    j = np.concatenate([a + 1, a + 2, a + 3, a])
    length = np.repeat(np.array([1, 1, 1, 2], dtype=np.float32), squares)
    res = rg.barcodes_sparse(i, j, length, n, 2, math.inf)
    h0, h1 = res.dim(0, 0), res.dim(1, 0)
    assert len(res.bars) == len(h0) + len(h1)
    assert len(h0) == n and np.isinf(h0["death"]).sum() == n - 3 * squares
    assert len(h1) == squares and (h1["birth"] == 2).all() and np.isinf(h1["death"]).all()
