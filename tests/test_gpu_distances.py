"""Device distances are the float64 rule's bit for bit: pairs settled in FP32
pairs and pairs left to float64 (middles between two FP32 numbers, powers of two,
very small and very large coordinates, coincident points), at the edges of tiles
and of the coordinate chunks, alone and in a batch of clouds."""
import numpy as np
import pytest

from paper_1908_02518_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _points(kind, n, k, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    x = rng.random((n, k))
    if kind == "integers":  # exact roots, ties and powers of two
        x = np.floor(8 * x)
    elif kind == "offset":  # differences of nearby numbers
        x = x + 1000.0
    elif kind == "tiny":
        x = x * 1e-20
    elif kind == "huge":
        x = x * 1e17
    elif kind == "doubled":
        x[n // 2:] = x[: n - n // 2]
    return x.astype(np.float32)


@pytest.mark.parametrize("n,k", [(1, 3), (2, 1), (31, 2), (32, 16), (33, 17), (65, 3), (257, 9), (100, 70)])
@pytest.mark.parametrize("kind", ["unit", "integers", "offset", "tiny", "huge", "doubled"])
def test_distances_are_the_rule(kind, n, k):
    import torch
    import paper_1908_02518_gb300 as rg
    x = _points(kind, n, k, 31 * n + k)
    with np.errstate(over="ignore"):
        want = W.distance_matrix(x)
    got = rg.distance_matrix(torch.from_numpy(x).cuda()).cpu().numpy()
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))


def test_many_pairs_near_the_middle():
    import torch
    import paper_1908_02518_gb300 as rg
    x = W.so3_points(1500, 77)  # 1.1 M pairs, some of them left to float64
    got = rg.distance_matrix(torch.from_numpy(x).cuda()).cpu().numpy()
    assert np.array_equal(got, W.distance_matrix(x))


def test_clouds_and_edge_lists_use_the_same_distances():
    import torch
    import paper_1908_02518_gb300 as rg
    clouds = [_points("unit", n, 3, n) for n in (5, 32, 33, 70)]
    off = np.cumsum([0] + [len(c) for c in clouds])
    res = rg.barcodes_batched(torch.from_numpy(np.concatenate(clouds)).cuda(), off, 1)
    for c, x in enumerate(clouds):
        one = rg.barcodes(W.distance_matrix(x), 1)
        assert np.array_equal(np.sort(res.bars[res.bars["cloud"] == c]["death"]), np.sort(one.bars["death"]))
    x = W.clifford_points(201, 4)
    a = rg.barcodes_sparse_points(torch.from_numpy(x).cuda(), 0.5, 1)
    b = rg.barcodes(W.distance_matrix(x), 1, 0.5)
    assert np.array_equal(a.bars, b.bars)
