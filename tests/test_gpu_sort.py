"""Edge order (csrc/rips_sort.cu, edge keys in csrc/rips_prologue.cu) where its
paths change: one-block sort up to 8192 edges, key lists in index order beyond,
radix passes with and without a scan launch (64 tiles of 2048 keys), row scans
by one block and by three kernels.  Small whole-number lengths make most edges
ties, so any slip in the order of equal lengths shows in the simplices."""
import math

import numpy as np
import pytest

from paper_1908_02518_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _key(bars):
    none = np.iinfo(np.uint64).max
    return sorted((int(b["dim"]), float(b["birth"]), float(b["death"]), int(b["birth_simplex"]),
                   int(none) if int(b["death_simplex"]) < 0 else int(b["death_simplex"])) for b in bars)


@pytest.mark.parametrize("n,t", [(2, math.inf), (3, math.inf), (23, math.inf), (24, math.inf), (65, math.inf),
                                 (91, math.inf), (128, math.inf), (129, math.inf), (129, 2.0), (512, 3.0), (513, 3.0),
                                 (513, 500.0), (700, 0.5)])
def test_order_of_ties(oracle_mod, n, t):
    import torch
    import paper_1908_02518_gb300 as rg
    d = W.random_integer_matrix(n, 3 if n < 512 else 500, n)
    dim = 1 if n < 512 else 0
    got = rg.barcodes(torch.from_numpy(d).cuda(), dim, t)
    assert _key(got.bars) == _key(oracle_mod.barcodes(d, dim, t).bars)


@pytest.mark.parametrize("count,n", [(3, 75), (40, 31), (1200, 14)])
def test_order_in_batches(oracle_mod, count, n):
    import torch
    import paper_1908_02518_gb300 as rg
    mats = [W.random_integer_matrix(n - c % 5, 4, 100 + c) for c in range(count)]
    res = rg.barcodes_batched_dists([torch.from_numpy(m).cuda() for m in mats], 1, math.inf)
    for c in range(0, count, max(1, count // 25)):
        got = np.concatenate([res.dim(d, c) for d in (0, 1)])
        assert _key(got) == _key(oracle_mod.barcodes(mats[c], 1).bars), c
