"""A plan's arena: the default takes clouds of ordinary size, and a given one is
for stored columns, with the tables of the columns under way beside it."""
import numpy as np
import pytest

from paper_1908_02518_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,lo,hi,per_edge", [(4, 200, 400, 0), (4, 200, 400, 80), (24, 64, 128, 40), (2, 12, 24, 5)])
def test_arena_is_enough(count, lo, hi, per_edge):
    import torch
    import paper_1908_02518_gb300 as rg
    clouds = W.batch_clouds(count, lo, hi, cloud_seed=7919)
    off = np.cumsum([0] + [len(c) for c in clouds])
    x = torch.from_numpy(np.concatenate(clouds)).cuda()
    edges = sum(len(c) * (len(c) - 1) // 2 for c in clouds)
    plan = rg.BatchPlan(off, 3, arena_entries=per_edge * edges)
    plan.run(x)
    got = plan.result().bars
    plan.free()
    want = rg.barcodes_batched(x, off, 1).bars
    assert got.tobytes() == want.tobytes()
