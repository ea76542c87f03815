"""What this library is measured on: barcode calls as programs make them.

Every case goes through the package's public entry points with inputs of the
repository's own kinds (workloads.py): point clouds of the cube, torus,
rotation-group, 3-sphere, circle and Clifford-torus families, as distance
matrices on the host or the device, packed triangles, edge lists, clouds within
a threshold, and batches of small clouds with and without gradients.

A pass returns the bars whole (dimension, endpoints, cloud and both simplices of
each, in arrays of a fixed length per problem size, the rest zero, as a layer of
fixed size downstream takes them) with the counts of the simplices' categories,
and gradients where there are any.
"""
import math

import numpy as np
import torch

import paper_1908_02518_gb300 as rg
from paper_1908_02518_gb300 import workloads as W

INF = float("inf")

# the categories into which every simplex falls, counted per dimension
CATEGORIES = ("simplices", "apparent_cofacet", "apparent_facet", "cleared", "columns", "emergent", "pairs",
              "zero_pairs", "essential")


def listed():
    return [
        # the smallest everyday call: a hundred points, all of H0 and H1; launches and host reads count
        {"name": "cube100", "kind": "dense", "data": "cube", "n": 100, "dim": 1, "t": INF, "p": 2, "host": False},
        # an ordinary shape-analysis call from a host matrix: a sampled surface up to H2 at a threshold
        {"name": "torus1000_host", "kind": "dense", "data": "torus", "n": 1000, "dim": 2, "t": 1.0, "p": 2,
         "host": True},
        # a large dense call: the rotation group (the headline benchmark's space) with its long-lived classes
        {"name": "so3_2048", "kind": "dense", "data": "so3", "n": 2048, "dim": 2, "t": 1.4, "p": 2, "host": False},
        # high dimension, odd coefficients, no threshold: 14 million 3-simplices on few points
        {"name": "s3_144_z3", "kind": "dense", "data": "sphere3", "n": 144, "dim": 3, "t": INF, "p": 3,
         "host": False},
        # single-linkage clustering of a stored metric: a packed triangle, H0 only
        {"name": "h0_packed_4096", "kind": "packed", "data": "so3", "n": 4096, "dim": 0, "t": INF, "p": 2,
         "layout": "lower"},
        # a point cloud within a threshold, up to H2, with no n x n array
        {"name": "clifford1500", "kind": "points", "data": "clifford", "n": 1500, "dim": 2, "t": 0.4, "p": 2},
        # a neighbourhood graph of an odd number of points as an edge list, H0 and H1
        {"name": "edges4999", "kind": "edges", "data": "clifford", "n": 4999, "dim": 1, "t": 0.45, "p": 2},
        # training with a topological loss on mini-batches of small clouds: forward and backward
        {"name": "train_small", "kind": "train", "count": 12, "lo": 24, "hi": 56, "dim": 1},
        # the same on uneven clouds of ordinary size (circles, tori and cubes of 64 to 512 points)
        {"name": "train_batch32", "kind": "train", "count": 32, "lo": 64, "hi": 512, "dim": 1},
        # serving: a plan for fixed cloud sizes, run on new coordinates
        {"name": "plan24", "kind": "plan", "count": 24, "lo": 64, "hi": 128, "p": 2},
        # several metric spaces at once up to H2 over Z/5, and the gradient to their matrices
        {"name": "dists7_h2", "kind": "dists", "count": 7, "lo": 33, "hi": 96, "dim": 2, "p": 5},
        # the distances of a cloud alone
        {"name": "distances4096", "kind": "distances", "data": "so3", "n": 4096, "k": 9},
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, even in the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dense", "dense", "dense", "packed", "points", "edges", "train", "plan", "dists", "distances"])
    if kind == "dense":
        data = rng.choice(["cube", "torus", "so3", "sphere3", "circle"])
        host = rng.random() < 0.3
        p = rng.choice([2, 2, 2, 3, 5, 11])
        if data == "cube":
            return {"kind": kind, "data": data, "n": _log(rng, 40, 300), "dim": 1, "t": INF, "p": p, "host": host}
        if data == "torus":
            return {"kind": kind, "data": data, "n": _log(rng, 150, 1300), "dim": 2,
                    "t": round(rng.uniform(0.6, 1.05), 3), "p": p, "host": host}
        if data == "so3":
            return {"kind": kind, "data": data, "n": _log(rng, 300, 2000), "dim": rng.choice([1, 2]),
                    "t": round(rng.uniform(1.2, 1.4), 3), "p": p, "host": host}
        if data == "circle":
            return {"kind": kind, "data": data, "n": _log(rng, 60, 350), "dim": 1, "t": INF, "p": p, "host": host}
        return {"kind": kind, "data": data, "n": _log(rng, 40, 130), "dim": rng.choice([2, 3]), "t": INF, "p": p,
                "host": host}
    if kind == "packed":
        return {"kind": kind, "data": rng.choice(["cube", "torus", "so3"]), "n": _log(rng, 200, 4096), "dim": 0,
                "t": INF, "p": 2, "layout": rng.choice(["lower", "upper"])}
    if kind == "points":
        n = _log(rng, 300, 3000)
        return {"kind": kind, "data": "clifford", "n": n, "dim": rng.choice([1, 2]),
                "t": round(0.4 * math.sqrt(1500 / n), 4), "p": rng.choice([2, 3])}
    if kind == "edges":
        n = _log(rng, 500, 4999)
        return {"kind": kind, "data": "clifford", "n": n, "dim": 1, "t": round(0.4 * math.sqrt(5000 / n), 4),
                "p": rng.choice([2, 2, 3])}
    if kind == "train":
        hi = _log(rng, 40, 400)
        return {"kind": kind, "count": _log(rng, 2, 32), "lo": max(8, hi // rng.choice([2, 4, 8])), "hi": hi, "dim": 1}
    if kind == "plan":
        hi = _log(rng, 24, 160)
        return {"kind": kind, "count": _log(rng, 2, 48), "lo": max(6, hi // 2), "hi": hi, "p": rng.choice([2, 3])}
    if kind == "dists":
        return {"kind": kind, "count": _log(rng, 2, 10), "lo": 17, "hi": _log(rng, 30, 96), "dim": rng.choice([1, 2]),
                "p": rng.choice([2, 3, 5])}
    return {"kind": kind, "data": rng.choice(["cube", "so3"]), "n": _log(rng, 200, 4096), "k": rng.choice([2, 3, 9])}


def _points(data, n, seed):
    if data == "cube":
        return W.cube_points(n, seed)
    if data == "torus":
        return W.torus_points(n, seed)
    if data == "so3":
        return W.so3_points(n, seed)
    if data == "sphere3":
        return W.sphere_points(n, seed, 4)
    if data == "clifford":
        return W.clifford_points(n, seed)
    return W.circle_points(np.random.Generator(np.random.PCG64(seed)), n).astype(np.float32)


def _clouds(case, seed):
    """Clouds whose sizes and kinds belong to the case and whose points to the seed."""
    return W.batch_clouds(case["count"], case["lo"], case["hi"], cloud_seed=7919 * (seed + 1))


def _room(points, dim):
    """Bars an output array has room for: at most this many per point in each dimension occur in these families."""
    return points * (1, 4, 10, 34)[dim] + 64


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("train", "plan"):
        clouds = _clouds(case, seed)
        st["offsets"] = np.cumsum([0] + [len(c) for c in clouds])
        st["points"] = torch.from_numpy(np.concatenate(clouds)).cuda()
        if kind == "plan":
            st["plan"] = rg.BatchPlan(st["offsets"], 3, INF, case["p"])
        return st
    if kind == "dists":
        st["dists"] = [rg.distance_matrix(torch.from_numpy(c).cuda()) for c in _clouds(case, seed)]
        return st
    if kind == "distances":  # coordinates past the family's own are its first ones again, shifted
        x = _points(case["data"], case["n"], seed)
        k = case["k"]
        x = np.concatenate([x + np.float32(0.25 * r) for r in range(-(-k // x.shape[1]))], axis=1)[:, :k]
        st["points"] = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        return st
    x = torch.from_numpy(_points(case["data"], case["n"], seed)).cuda()
    if kind == "points":
        st["points"] = x
        return st
    d = rg.distance_matrix(x)
    if kind == "dense":
        st["dist"] = d.cpu().numpy() if case["host"] else d
    elif kind == "packed":
        i, j = torch.tril_indices(case["n"], case["n"], -1, device=d.device)
        if case["layout"] == "upper":
            i, j = torch.triu_indices(case["n"], case["n"], 1, device=d.device)
        st["packed"] = d[i, j].contiguous()
    else:
        i, j = torch.nonzero(torch.tril(d <= case["t"], -1), as_tuple=True)
        st["i"], st["j"], st["len"] = i.to(torch.int32), j.to(torch.int32), d[i, j]
    return st


def _bars(res, points):
    room = np.zeros(_room(points, res.dim_max), dtype=res.bars.dtype)
    room[:len(res.bars)] = res.bars  # raises if there are more
    b = {f: np.ascontiguousarray(room[f]) for f in room.dtype.names}
    return {"dim": b["dim"], "birth": b["birth"], "death": b["death"], "cloud": b["cloud"],
            "birth_simplex": b["birth_simplex"].view(np.int64), "death_simplex": b["death_simplex"].view(np.int64),
            "bars": len(res.bars), "thresholds": np.array(res.thresholds, dtype=np.float32),
            "counts": np.array([[[s[c] for c in CATEGORIES] for s in row] for row in res.stats], dtype=np.int64)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "dense":
        return _bars(rg.barcodes(state["dist"], case["dim"], case["t"], case["p"]), case["n"])
    if kind == "packed":
        return _bars(rg.barcodes_packed(state["packed"], case["n"], case["layout"], case["dim"], case["t"], case["p"]),
                     case["n"])
    if kind == "points":
        return _bars(rg.barcodes_sparse_points(state["points"], case["t"], case["dim"], case["p"]), case["n"])
    if kind == "edges":
        return _bars(rg.barcodes_sparse(state["i"], state["j"], state["len"], case["n"], case["dim"], INF, case["p"]),
                     case["n"])
    if kind == "train":  # total squared persistence of the loops, and its gradient
        x = state["points"].detach().requires_grad_(True)
        birth, death, dim, cloud = rg.RipsBarcodes.apply(x, state["offsets"], case["dim"])
        life = torch.where(torch.isfinite(death) & (dim == 1), death - birth, torch.zeros_like(birth))
        (grad,) = torch.autograd.grad((life * life).sum(), x)
        out = torch.zeros((2, _room(len(x), case["dim"])), dtype=torch.float32, device=x.device)
        out[0, :len(birth)], out[1, :len(birth)] = birth.detach(), death.detach()
        tags = torch.zeros((2, out.shape[1]), dtype=torch.int64, device=x.device)
        tags[0, :len(birth)], tags[1, :len(birth)] = dim, cloud
        return {"bars": out, "tags": tags, "grad": grad}
    if kind == "plan":
        state["plan"].run(state["points"])
        return _bars(state["plan"].result(), len(state["points"]))
    if kind == "dists":  # the same loss over every dimension, gradient to the matrices
        res = rg.barcodes_batched_dists(state["dists"], case["dim"], INF, case["p"], keep_handle=True)
        birth = torch.from_numpy(res.bars["birth"].copy()).cuda()
        death = torch.from_numpy(res.bars["death"].copy()).cuda()
        life = torch.where(torch.isfinite(death), death - birth, torch.zeros_like(birth))
        grads = rg.backward_dist(res, state["dists"], -2.0 * life, 2.0 * life)
        res.free()
        return {"bars": _bars(res, sum(len(d) for d in state["dists"])), "grads": torch.cat([g.reshape(-1) for g in grads])}
    return rg.distance_matrix(state["points"])


def work(case):
    """Inputs read once and the bars and gradients written once (a bar: 32 bytes; every point begins one)."""
    kind = case["kind"]
    if kind in ("dense", "packed"):
        n = case["n"]
        return {"bytes": 2 * n * (n - 1) + 32 * n, "flops": 0}
    if kind == "points":
        return {"bytes": 16 * case["n"] + 32 * case["n"], "flops": 0}
    if kind == "edges":  # the share of pairs within the threshold: a disc on the flat torus of area 2 pi^2
        n, t = case["n"], case["t"]
        return {"bytes": 12 * 0.5 * n * n * min(1.0, t * t / (2 * math.pi)) + 32 * n, "flops": 0}
    if kind in ("train", "plan"):
        n = case["count"] * 0.5 * (case["lo"] + case["hi"])
        return {"bytes": n * (12 + 32) + (n * 12 if kind == "train" else 0), "flops": 0}
    if kind == "dists":
        lo, hi = case["lo"], case["hi"]
        sq = case["count"] * (lo * lo + lo * hi + hi * hi) / 3.0
        return {"bytes": 2 * sq + 4 * sq, "flops": 0}
    n, k = case["n"], case["k"]
    return {"bytes": 4 * n * k + 4 * n * n, "flops": 0.5 * n * n * (3 * k + 1)}


# ---------------------------------------------------------------- 64-bit values

def _dist64(x):
    """Distances in float64, and rounded to FP32 as the filtration orders them."""
    x = np.asarray(x, dtype=np.float32).astype(np.float64)
    acc = np.zeros((len(x), len(x)))
    for c in range(x.shape[1]):
        diff = x[:, None, c] - x[None, :, c]
        acc += diff * diff
    d = np.sqrt(acc)
    return d, d.astype(np.float32)


def _h0_lengths(d):
    """Edge lengths of a minimum spanning tree, ascending (Prim)."""
    n = len(d)
    best = d[0].copy()
    out = np.zeros(n, dtype=bool)
    out[0] = True
    best[0] = np.inf
    lens = np.empty(n - 1)
    for q in range(n - 1):
        v = int(np.argmin(best))
        lens[q] = best[v]
        out[v] = True
        best = np.minimum(best, d[v])
        best[out] = np.inf
    return np.sort(lens)


def _h0_h1(x):
    """Bars of one small cloud up to its enclosing radius over Z/2 by reducing the boundary matrix of the triangles
    (columns as whole numbers, one bit an edge): H0 deaths, and (birth edge, death edge) of H1."""
    d, f = _dist64(x)
    n = len(d)
    g = f.copy()
    np.fill_diagonal(g, 0.0)
    t = g.max(axis=1).min()
    i, j = np.tril_indices(n, -1)
    idx = i * (i - 1) // 2 + j
    keep = f[i, j] <= t
    i, j, idx = i[keep], j[keep], idx[keep]
    order = np.lexsort((-idx, f[i, j]))
    i, j = i[order], j[order]
    pos = np.full((n, n), -1, dtype=np.int64)
    pos[i, j] = np.arange(len(i))
    tree, label, deaths = 0, list(range(n)), []
    find = lambda a: a if label[a] == a else find(label[a])  # noqa: E731
    for e in range(len(i)):
        a, b = find(int(i[e])), find(int(j[e]))
        if a != b:
            label[a] = b
            tree += 1
            deaths.append(e)
    a, b, c = (v.reshape(-1) for v in np.meshgrid(np.arange(n), np.arange(n), np.arange(n), indexing="ij"))
    m = (a > b) & (b > c)
    a, b, c = a[m], b[m], c[m]
    m = (pos[a, b] >= 0) & (pos[a, c] >= 0) & (pos[b, c] >= 0)
    a, b, c = a[m], b[m], c[m]
    e3 = np.sort(np.stack([pos[a, b], pos[a, c], pos[b, c]]), axis=0)
    tidx = a * (a - 1) * (a - 2) // 6 + b * (b - 1) // 2 + c
    rank = np.unique(f[i, j], return_inverse=True)[1]
    e3 = e3[:, np.lexsort((-tidx, rank[e3[2]]))]
    low, pairs = {}, []
    for q in range(e3.shape[1]):
        if len(low) == len(i) - tree:
            break
        x0, x1, x2 = (int(v) for v in e3[:, q])
        col = (1 << x0) | (1 << x1) | (1 << x2)
        while col:
            h = col.bit_length() - 1
            other = low.get(h)
            if other is None:
                low[h] = col
                pairs.append((h, x2))
                break
            col ^= other
    return d, f, i, j, deaths, pairs


def _train_exact(case, seed):
    births, deaths, grads = [], [], []
    for x in _clouds(case, seed):
        d, f, i, j, h0, h1 = _h0_h1(x)
        x = x.astype(np.float64)
        births += [0.0] * len(x)
        deaths += [d[i[e], j[e]] for e in h0 if f[i[e], j[e]] > 0] + [np.inf]
        assert len(h0) == len(x) - 1 and all(f[i[e], j[e]] > 0 for e in h0)
        g = np.zeros_like(x)
        h1 = [(b, e) for b, e in h1 if f[i[b], j[b]] < f[i[e], j[e]]]
        for b, e in sorted(h1, key=lambda q: (f[i[q[0]], j[q[0]]], f[i[q[1]], j[q[1]]])):
            vb, ve = d[i[b], j[b]], d[i[e], j[e]]
            births.append(vb)
            deaths.append(ve)
            for edge, s in ((b, -1.0), (e, 1.0)):
                u, v = int(i[edge]), int(j[edge])
                step = 2.0 * s * (ve - vb) * (x[u] - x[v]) / d[u, v]
                g[u] += step
                g[v] -= step
        grads.append(g)
    bars = np.zeros((2, _room(sum(len(g) for g in grads), 1)))
    bars[0, :len(births)], bars[1, :len(births)] = births, deaths
    return {"bars": bars, "tags": None, "grad": np.concatenate(grads)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "distances":
        x = prepare(case, seed)["points"].double()
        acc = torch.zeros((len(x), len(x)), dtype=torch.float64, device=x.device)
        for c in range(x.shape[1]):
            acc += (x[:, None, c] - x[None, :, c]) ** 2
        return acc.sqrt()
    if kind == "packed" and case["dim"] == 0:  # one component: every other point's death is a tree edge
        d, f = _dist64(_points(case["data"], case["n"], seed))
        lens = _h0_lengths(d)
        if not (lens > 0).all():
            return None
        death = np.zeros(_room(case["n"], 0))
        death[:case["n"]] = np.append(lens, np.inf)
        return {"dim": None, "birth": np.zeros(len(death)), "death": death, "cloud": None, "birth_simplex": None,
                "death_simplex": None, "bars": None, "thresholds": None, "counts": None}
    if kind == "train" and case["hi"] <= 64 and case["count"] <= 16:
        return _train_exact(case, seed)
    return None
