"""Teams of blocks (csrc/rips_reduce.cuh), where the blocks of a launch divide
themselves anew: a column that outlives the others and passes from a block to 64
of them and, after 4,096 additions, to the whole grid.  Which team a block is in
follows from lists that stay as they are while the teams run, so every run gives
the same bars."""
import math

import pytest

from paper_1908_02518_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LARGE = 4096  # additions after which a lone column's team grows from 64 blocks to all

# name, distances, dimension, threshold, p, additions of the longest chain at least
CASES = [("s3_112", lambda: W.distance_matrix(W.sphere_points(112, 1005, 4)), 3, math.inf, 3, LARGE),
         ("so3_700", lambda: W.distance_matrix(W.so3_points(700, 1005)), 1, math.inf, 2, 32)]


def _key(bars):
    return sorted((int(b["dim"]), float(b["birth"]), float(b["death"]), int(b["birth_simplex"]),
                   int(b["death_simplex"]) % 2**64) for b in bars)


@pytest.mark.parametrize("name,make,dim_max,t,p,chain", CASES, ids=[c[0] for c in CASES])
def test_columns_that_change_teams(oracle_mod, name, make, dim_max, t, p, chain):
    import torch
    import paper_1908_02518_gb300 as rg
    d = make()
    want = _key(oracle_mod.barcodes(d, dim_max, t, p).bars)
    x = torch.from_numpy(d).cuda()
    for _ in range(10):
        res = rg.barcodes(x, dim_max, t, p)
        assert max(s["longest_chain"] for s in res.stats[0]) >= chain
        assert _key(res.bars) == want


def test_columns_that_start_with_a_team(oracle_mod):
    """A few columns left, with thousands of stored rows (a circle's last ones):
    a team each from the start of the round, which all blocks have to agree on."""
    import torch
    import numpy as np
    import paper_1908_02518_gb300 as rg
    clouds = [W.circle_points(np.random.Generator(np.random.PCG64(s)), n).astype(np.float32)
              for s, n in ((5, 150), (6, 149), (7, 33), (8, 128))]
    off = np.cumsum([0] + [len(c) for c in clouds])
    x = torch.from_numpy(np.concatenate(clouds)).cuda()
    want = [_key(oracle_mod.barcodes(W.distance_matrix(c), 1).bars) for c in clouds]
    for _ in range(10):
        res = rg.barcodes_batched(x, off, 1)
        for c in range(len(clouds)):
            assert _key(res.bars[res.bars["cloud"] == c]) == want[c], c


def test_a_full_table_ends_all_blocks_together():
    """A claim that finds the pivot table full is seen by every block at the same
    point: none is left at a barrier until its wait runs out (30 s, and a timeout
    status)."""
    import time
    import torch
    import paper_1908_02518_gb300 as rg
    from paper_1908_02518_gb300 import _lib
    x = torch.from_numpy(W.distance_matrix(W.sphere_points(64, 1005, 4))).cuda()
    want = _key(rg.barcodes(x, 3, math.inf, 3).bars)
    try:
        for slots in (16, 32, 64):
            rg.set_limits(table_slots=slots)
            for _ in range(10):
                t0 = time.monotonic()
                with pytest.raises(_lib.RipsError) as e:
                    rg.barcodes(x, 3, math.inf, 3)
                assert e.value.status == -4  # RIPS_ERR_OOM
                assert time.monotonic() - t0 < 10
    finally:
        rg.set_limits()
    assert _key(rg.barcodes(x, 3, math.inf, 3).bars) == want


def test_a_wait_that_runs_out_is_a_timeout_with_a_full_arena_too():
    """A reduction whose waits run out is not started over in a larger arena, also
    when the arena was full at that time: as many launches as with room."""
    import torch
    import paper_1908_02518_gb300 as rg
    from paper_1908_02518_gb300 import _lib
    x = torch.from_numpy(W.distance_matrix(W.torus_points(300, 21))).cuda()
    want = _key(rg.barcodes(x, 2, 1.2).bars)
    launches = []
    try:
        for entries in (0, 64):
            rg.set_limits(barrier_wait_ns=1, chain_ns=1, arena_entries=entries)
            rg.launch_count(reset=True)
            with pytest.raises(_lib.RipsError) as e:
                rg.barcodes(x, 2, 1.2)
            assert e.value.status == -6  # RIPS_ERR_DEVICE_TIMEOUT
            launches.append(rg.launch_count())
    finally:
        rg.set_limits()
    assert launches[1] <= launches[0]
    assert _key(rg.barcodes(x, 2, 1.2).bars) == want


def _uniform(n):
    import numpy as np
    a = np.tril(np.random.Generator(np.random.PCG64(n)).random((n, n)).astype(np.float32), -1)
    return a + a.T


def _hamming(n, bits):
    import numpy as np
    x = np.random.Generator(np.random.PCG64(n)).integers(0, 2, (n, bits))
    return (x[:, None] != x[None]).sum(-1).astype(np.float32)


@pytest.mark.parametrize("name,make,dim_max", [("uniform140", lambda: _uniform(140), 1),
                                               ("uniform60", lambda: _uniform(60), 2),
                                               ("hamming200", lambda: _hamming(200, 40), 1)])
def test_lengths_without_geometry(oracle_mod, name, make, dim_max):
    """Random lengths: rows come back as fast as they are eliminated, windows are cut
    back time and again, and all blocks of a team have to cut them alike."""
    import torch
    import paper_1908_02518_gb300 as rg
    d = make()
    want = _key(oracle_mod.barcodes(d, dim_max).bars)
    x = torch.from_numpy(d).cuda()
    for _ in range(20):
        assert _key(rg.barcodes(x, dim_max).bars) == want
