"""Wide elimination (csrc/rips_wide.cuh) at the sizes where its paths change:
stored columns longer and shorter than the sorted ones, coefficients whose sums
wrap and invert, coboundaries by the generic code (d >= 4), ties (many rows of
one diameter in a window), neighbour lists of a sparse input, columns given to a
block at once, one block per SM, tables grown from a tiny arena, and every pivot
owned through the table.  Bars must equal the oracle's one by one."""
import math

import numpy as np
import pytest

from paper_1908_02518_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _circle(n):
    return W.distance_matrix(W.circle_points(np.random.Generator(np.random.PCG64(5)), n).astype(np.float32))


CASES = [
    ("circle33", lambda: _circle(33), 1, math.inf, 2),
    ("circle150", lambda: _circle(150), 1, math.inf, 2),  # a chain of hundreds, a stored column of thousands
    ("circle97_p65521", lambda: _circle(97), 1, math.inf, 65521),
    ("torus260_p7", lambda: W.distance_matrix(W.torus_points(260, 9)), 2, 1.3, 7),
    ("s3_40", lambda: W.distance_matrix(W.sphere_points(40, 11)), 3, math.inf, 3),
    ("s3_17_d4", lambda: W.distance_matrix(W.sphere_points(17, 12, 6)), 4, math.inf, 3),
    ("ties31", lambda: W.random_integer_matrix(31, 77, 3), 2, math.inf, 5),
    ("polygon64", lambda: W.regular_polygon_matrix(64), 1, math.inf, 2),
    ("simplex16", lambda: W.regular_simplex_matrix(16), 2, math.inf, 2),
]


def _key(bars):
    none = np.iinfo(np.uint64).max
    return sorted((int(b["dim"]), float(b["birth"]), float(b["death"]), int(b["birth_simplex"]),
                   int(none) if int(b["death_simplex"]) < 0 else int(b["death_simplex"])) for b in bars)


@pytest.fixture(autouse=True)
def _defaults():
    import paper_1908_02518_gb300 as rg
    from paper_1908_02518_gb300 import tuning
    yield
    rg.set_limits()
    rg.set_options()
    tuning.clear_tuning()


@pytest.mark.parametrize("name,make,dim_max,t,p", CASES, ids=[c[0] for c in CASES])
def test_wide_elimination_matches_oracle(oracle_mod, name, make, dim_max, t, p):
    import torch
    import paper_1908_02518_gb300 as rg
    from paper_1908_02518_gb300 import tuning
    d = make()
    x = torch.from_numpy(d).cuda()
    want = _key(oracle_mod.barcodes(d, dim_max, t, p).bars)
    assert _key(rg.barcodes(x, dim_max, t, p).bars) == want
    for params in ({"warp_chain_limit": 1, "warp_merge_max": 1}, {"reduce_blocks_per_sm": 1}):
        for dim in range(1, dim_max + 1):
            tuning.set_tuning(dim, 1, 1 << 20, params)
        assert _key(rg.barcodes(x, dim_max, t, p).bars) == want, params
    tuning.clear_tuning()
    rg.set_limits(arena_entries=4096)
    assert _key(rg.barcodes(x, dim_max, t, p).bars) == want, "tiny arena"
    rg.set_limits()
    rg.set_options(apparent=False)
    assert _key(rg.barcodes(x, dim_max, t, p).bars) == want, "no apparent pairs"
    rg.set_options()
    i, j = np.tril_indices(len(d), -1)
    thr = t if math.isfinite(t) else rg.barcodes(x, 0).threshold
    got = rg.barcodes_sparse(i, j, d[i, j], len(d), dim_max, thr, p)
    assert _key(got.bars) == want, "edge list"
