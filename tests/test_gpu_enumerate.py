"""Enumeration (csrc/rips_dim.cu): the number of simplices of every dimension at
sizes around the warp's 32 candidates and its buffer of 128 simplices, from the
rank matrix and from neighbour lists alone, in the kernels for triangles and
tetrahedra and in the one for any dimension, with several clouds at once."""
import numpy as np
import pytest

from paper_1908_02518_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _counts(d, t, dim):
    """Simplices of dimension 1..dim with diameter <= t, each grown by vertices above its top one."""
    a = np.triu(d <= t, 1)
    level = [(v, a[v]) for v in range(len(d))]
    out = []
    for _ in range(dim):
        level = [(j, up & a[j]) for _, up in level for j in np.flatnonzero(up)]
        out.append(len(level))
    return out


@pytest.mark.parametrize("n,dim,t", [(2, 2, 9.0), (4, 3, 9.0), (33, 2, 9.0), (33, 3, 9.0), (20, 4, 9.0), (129, 2, 0.4),
                                     (70, 3, 0.5), (40, 4, 0.5), (131, 2, 0.02)])
def test_counts(n, dim, t):
    import torch
    import paper_1908_02518_gb300 as rg
    x = W.cube_points(n, 5)
    d = W.distance_matrix(x)
    for res in (rg.barcodes(torch.from_numpy(d).cuda(), dim, t),
                rg.barcodes_sparse_points(torch.from_numpy(x).cuda(), t, dim)):
        assert [res.stats[0][k]["simplices"] for k in range(1, dim + 1)] == _counts(d, res.thresholds[0], dim)


@pytest.mark.parametrize("dim", [2, 3])
def test_counts_of_several_clouds(dim):
    import torch
    import paper_1908_02518_gb300 as rg
    ds = [W.distance_matrix(W.cube_points(n, n)) for n in (3, 31, 32, 33, 5, 24)]
    res = rg.barcodes_batched_dists([torch.from_numpy(d).cuda() for d in ds], dim, 0.7)
    got = [[row[k]["simplices"] for k in range(1, dim + 1)] for row in res.stats]
    assert got == [_counts(d, t, dim) for d, t in zip(ds, res.thresholds)]
