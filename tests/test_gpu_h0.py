"""H0 by contraction (csrc/rips_h0.cu) where its paths change: one edge batch and
several, block sizes, disconnected threshold graphs (the whole list is read),
ties, zero lengths, and a chain of growing gaps, which merges one component a
round and is finished by one thread.  Bars must equal the oracle's one by one."""
import math

import numpy as np
import pytest

from paper_1908_02518_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _line(n):
    """Points on a line with growing gaps, in order: vertex i + 1 lies nearer to i than to i + 2."""
    x = np.cumsum(np.linspace(1.0, 2.0, n)).astype(np.float32)
    return np.abs(x[:, None] - x[None, :]).astype(np.float32)


def _clusters(n):
    x = W.cube_points(n, 5)
    x[n // 2:] += 10.0
    return W.distance_matrix(x)


def _doubled(n):
    x = W.cube_points(n, 6)
    return W.distance_matrix(np.concatenate([x, x[: n // 3]]))  # zero distances


CASES = [("one", lambda: W.distance_matrix(W.cube_points(1, 3)), math.inf), ("two", lambda: _line(2), math.inf),
         ("line257", lambda: _line(257), math.inf), ("line1500", lambda: _line(1500), math.inf),
         ("clusters300", lambda: _clusters(300), math.inf), ("clusters300_apart", lambda: _clusters(300), 2.0),
         ("sparse256", lambda: W.distance_matrix(W.cube_points(256, 8)), 0.05),
         ("doubled240", lambda: _doubled(180), math.inf), ("ties97", lambda: W.random_integer_matrix(97, 4, 3), math.inf),
         ("torus1024", lambda: W.distance_matrix(W.torus_points(1024, 8)), math.inf)]


def _key(bars):
    none = np.iinfo(np.uint64).max
    return sorted((int(b["dim"]), float(b["birth"]), float(b["death"]), int(b["birth_simplex"]),
                   int(none) if int(b["death_simplex"]) < 0 else int(b["death_simplex"])) for b in bars)


@pytest.mark.parametrize("name,make,t", CASES, ids=[c[0] for c in CASES])
def test_h0_matches_oracle(oracle_mod, name, make, t):
    import torch
    import paper_1908_02518_gb300 as rg
    d = make()
    got = rg.barcodes(torch.from_numpy(d).cuda(), 0, t)
    want = oracle_mod.barcodes(d, 0, t)
    assert _key(got.bars) == _key(want.bars)
    assert got.stats[0][0]["essential"] == want.stats[0]["essential"]


def test_h0_of_a_batch(oracle_mod):
    import torch
    import paper_1908_02518_gb300 as rg
    mats = [c[1]() for c in CASES if c[0] not in ("line1500", "torus1024")]
    res = rg.barcodes_batched_dists([torch.from_numpy(m).cuda() for m in mats], 0, math.inf)
    for c, m in enumerate(mats):
        assert _key(res.dim(0, c)) == _key(oracle_mod.barcodes(m, 0).bars), c
