"""Digests of FP64 results on inputs that are exact on every host (integers over powers of two):
nearest triangles of points, and brackets with their counts.  `python tests/golden/fp64_bits.py`
writes tests/golden/fp64_bits.json with the library it finds; the file in the tree was made on a
GB300 with the sources of commit c4cf736, whose FP64 traversal and bounds have no FP32 in them.
"""
import hashlib
import json
import os
import sys

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
PATH = os.path.join(HERE, "fp64_bits.json")


def _terrain(n, seed, rough=200):
    """An n x n grid of two triangles a cell, heights in 1/1024, jittered in x and y."""
    rng = np.random.default_rng(seed)
    i, j = np.meshgrid(np.arange(n + 1), np.arange(n + 1), indexing="ij")
    V = np.stack([1024 * i, 1024 * j, 0 * i], -1).reshape(-1, 3) + rng.integers(-rough, rough + 1, ((n + 1) ** 2, 3))
    a = ((n + 1) * i[:-1, :-1] + j[:-1, :-1]).reshape(-1)
    F = np.concatenate([np.stack([a, a + n + 1, a + n + 2], 1), np.stack([a, a + n + 2, a + 1], 1)])
    return V / 1024.0, F.astype(np.int32)


def _mesh(kind, n, seed):
    if kind == "flat":  # every vertex and edge on a lattice: exact ties everywhere
        V, F = _terrain(n, seed, 0)
    else:
        V, F = _terrain(n, seed)
    if kind == "slivers":  # a row of needles, zero-area and repeated-vertex triangles
        rng = np.random.default_rng(seed + 1)
        W = rng.integers(0, 1024 * n, (300, 3)) / 1024.0
        W[1::3] = W[::3] + rng.integers(-4096, 4097, (100, 3)) / 1024.0
        W[2::3] = W[::3] + (W[1::3] - W[::3]) * (rng.integers(0, 5, (100, 1)) / 4.0) + rng.integers(-1, 2, (100, 3)) / 2.0**20
        F = np.concatenate([F, len(V) + np.arange(300).reshape(-1, 3), np.array([[0, 0, 1], [2, 2, 2]])]).astype(np.int32)
        V = np.concatenate([V, W])
    return V, F


def _points(V, F, n, seed):
    rng = np.random.default_rng(seed)
    lo, hi = np.floor(V.min(0)), np.ceil(V.max(0))
    T = V[F]
    half = T[rng.integers(len(F), size=n)]
    return np.concatenate([
        V[rng.integers(len(V), size=n)],  # on vertices
        (half[:, 0] + half[:, 1]) / 2,  # on edges
        lo + (hi - lo) * rng.integers(-512, 1537, (n, 3)) / 1024.0,  # in the volume and around it
        (half[:, 0] + half[:, 1] + 2 * half[:, 2]) / 4 + rng.integers(-64, 65, (n, 3)) / 4096.0,  # near the surface
    ])


NEAREST = [(k, n, s, t, v, leaf) for k, n in (("flat", 12), ("rough", 40), ("slivers", 24))
           for s, t in ((0, 0.0), (0, 2.0**20), (-83, 0.0), (100, 0.0))
           for v, leaf in (("f32", 1), ("f64", 1), ("f64", 16))]
BRACKETS = [(s, t, order, batched) for s, t in ((0, 0.0), (0, 2.0**14), (-83, 0.0))
            for order in ((1, 2, 3, 4), (3, 1)) for batched in (False, True)]
COUNTS = ("rounds", "splits", "queries", "leaf_tests", "long_queries", "retired", "discards")


def nearest(hd, kind, n, scale, shift, vtype, leaf):
    import torch

    V, F = _mesh(kind, n, 7)
    V = V * 2.0**scale + shift
    if vtype == "f32":
        V = V.astype(np.float32)
    P = _points(np.asarray(V, np.float64) if shift == 0 else V - shift, F, 400, 11)
    P = P + shift if shift else P
    bvh = hd.hd_build_B(V, F, hd.hd_options_default(leaf_size=leaf))
    out = hashlib.sha256()
    for x in hd.hd_nearest(bvh, torch.from_numpy(np.ascontiguousarray(P, np.float64)).cuda(), hd.HD_FP64)[:3]:
        out.update(x.cpu().numpy().tobytes())
    return out.hexdigest()


def bracket(hd, scale, shift, order, batched):
    VB, FB = _mesh("rough", 24, 7)
    VA, FA = _mesh("rough", 24, 8)
    VA, VB = VA * 2.0**scale + shift, (VB + [0, 0, 1 / 8]) * 2.0**scale + shift
    o = hd.hd_options_default(tol_mode=hd.HD_TOL_REL, bound_order=order, flags=hd.HD_FLAG_EXACT_QUERIES)
    bvh = hd.hd_build_B(VB, FB)
    r = hd.hd_hausdorff_batched([bvh], [(VA, FA)], 1e-4, o)[0] if batched else hd.hd_hausdorff(bvh, VA, FA, 1e-4, o)
    return [r["lower"].hex(), r["upper"].hex(), r["status"]] + [r["stats"][k] for k in COUNTS[:-1]] + list(r["stats"]["discards"].values())


def key(case):
    return " ".join(str(x) for x in case)


if __name__ == "__main__":
    sys.path.insert(0, os.getcwd())
    import paper_2406_10357_gb300 as hd

    with open(PATH if len(sys.argv) < 2 else sys.argv[1], "w") as f:
        json.dump(dict(nearest={key(c): nearest(hd, *c) for c in NEAREST}, bracket={key(c): bracket(hd, *c) for c in BRACKETS}),
                  f, indent=0, sort_keys=True)
        f.write("\n")
