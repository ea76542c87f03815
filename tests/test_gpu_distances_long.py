"""Device distances are the float64 rule's bit for bit in many coordinates too,
where the round-offs of a running sum add up: equal differences (all of one sign),
images in one grey level each, features that are there or not, and one large
coordinate before many small ones; in every entry point that takes points."""
import math

import numpy as np
import pytest

from paper_1908_02518_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# two points with all coordinates equal, whose distance needs more than the first few of the sum's low bits
PAIRS = [(169, 0.9720024, 0.8214535), (196, 0.5034641, 0.0), (324, 0.94473314, 0.0)]


def _points(kind, n, k):
    rng = np.random.Generator(np.random.PCG64(1000 * n + k))
    if kind == "equal":
        x = np.repeat(rng.random((n, 1)), k, 1)
    elif kind == "grey":
        x = np.repeat((rng.integers(0, 256, (n, 1)) / 255).astype(np.float32), k, 1)
    elif kind == "features":
        x = np.floor(1.7 * rng.random((n, k))) * rng.random((n, 1))
    elif kind == "first":
        x = np.repeat(rng.random((n, 1)), k, 1)
        x[:, 0] *= 30
    else:
        x = rng.standard_normal((n, k))
    return x.astype(np.float32)


def _same(x):
    import torch
    import paper_1908_02518_gb300 as rg
    got = rg.distance_matrix(torch.from_numpy(x).cuda()).cpu().numpy()
    assert np.array_equal(got.view(np.uint32), W.distance_matrix(x).view(np.uint32))


@pytest.mark.parametrize("n,k", [(200, 17), (200, 48), (300, 169), (300, 196), (260, 400), (256, 784), (70, 4096)])
@pytest.mark.parametrize("kind", ["equal", "grey", "features", "first", "normal"])
def test_distances_are_the_rule(kind, n, k):
    _same(_points(kind, n, k))


@pytest.mark.parametrize("k,a,b", PAIRS)
def test_every_entry_point_uses_the_rule(k, a, b):
    import torch
    import paper_1908_02518_gb300 as rg
    x = np.repeat(np.array([[a], [b]], dtype=np.float32), k, 1)
    _same(x)
    d = float(W.distance_matrix(x)[1, 0])
    pts = torch.from_numpy(x).cuda()
    got = [rg.barcodes_batched(pts, [0, 2], 0).bars, rg.barcodes_sparse_points(pts, 100.0, 0).bars]
    for bars in got:
        assert sorted(bars["death"].tolist()) == [d, math.inf]
