"""What a plan holds: its arena follows the caller's entries (three times as many,
or 640 per edge more, with the tables of the columns under way), and a run of what
the entries are for stays within it, again and again."""
import numpy as np
import pytest

from paper_1908_02518_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ENTRY = 12        # bytes
PER_EDGE = 2048   # bytes an edge of all other buffers (keys, ranks, lists, pivot table, bars)
SLACK = 96 << 20


@pytest.mark.parametrize("count,lo,hi,per_edge", [(24, 64, 128, 0), (24, 64, 128, 40), (4, 200, 400, 300),
                                                  (48, 80, 160, 400)])
def test_memory_of_a_plan(count, lo, hi, per_edge):
    import torch
    import paper_1908_02518_gb300 as rg
    clouds = W.batch_clouds(count, lo, hi, cloud_seed=7919)
    off = np.cumsum([0] + [len(c) for c in clouds])
    edges = sum(len(c) * (len(c) - 1) // 2 for c in clouds)
    x = torch.from_numpy(np.concatenate(clouds)).cuda()
    want = rg.barcodes_batched(x, off, 1).bars
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    plan = rg.BatchPlan(off, 3, arena_entries=per_edge * edges)
    held = before - torch.cuda.mem_get_info()[0]
    arena = max(3 * per_edge, per_edge + 640) if per_edge else 1024
    assert held <= edges * (ENTRY * arena + PER_EDGE) + SLACK, held / edges
    for _ in range(5):
        plan.run(x)
        assert plan.result().bars.tobytes() == want.tobytes()
    plan.free()
