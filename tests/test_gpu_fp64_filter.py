"""FP64 queries and bounds decided by FP32 filters, where a filter could decide wrongly: exact
ties (points on vertices and edges of B), zero-area triangles, scales whose squares leave the
float range, coordinates far from the origin (float forms of the points are then coarse), both
input types, leaf ranges, and counts at the edges of a warp.

Tolerance: both sides compute in double with round-to-nearest; a distance carries at most a
few hundred roundings relative to the largest coordinate C, so 1e-12 C.
"""
import numpy as np
import pytest

import meshgen as mg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.fixture(scope="module")
def hd():
    from paper_2406_10357_gb300 import build

    build.build()
    import paper_2406_10357_gb300 as hd

    return hd


@pytest.mark.parametrize("n", [1, 31, 33, 701])
@pytest.mark.parametrize("scale,shift", [(1.0, 0.0), (1.0, 1e6), (1e-25, 0.0), (1e30, 0.0)])
@pytest.mark.parametrize("vtype,leaf", [("f32", 1), ("f64", 1), ("f64", 16)])
def test_nearest_fp64_filtered(hd, orc, n, scale, shift, vtype, leaf):
    rng = np.random.default_rng(n)
    VB, FB = mg.superquadric(1.0, 1.0, 1.0, 26, 13, 0.3, mg.stream(7, 1))
    VB = VB * scale + shift
    if vtype == "f32":
        VB = VB.astype(np.float32)
    W = np.asarray(VB, np.float64)
    T = W[FB]
    kinds = [
        W[rng.integers(len(W), size=n)],  # on vertices
        T[rng.integers(len(FB), size=n), :2].mean(1),  # on edges
        shift + scale * rng.uniform(-1.6, 1.6, (n, 3)),  # in the volume
        T.mean(1)[rng.integers(len(FB), size=n)] + scale * rng.normal(0, 1e-3, (n, 3)),  # near the surface
        shift + (W[rng.integers(len(W), size=n)] - shift) * 1.5,  # outwards of vertices
    ]
    P = np.concatenate(kinds)
    bvh = hd.hd_build_B(torch.from_numpy(VB).cuda(), torch.from_numpy(FB).cuda(), hd.hd_options_default(leaf_size=leaf))
    d, idx, foot, _ = (x.cpu().numpy() for x in hd.hd_nearest(bvh, torch.from_numpy(P).cuda(), hd.HD_FP64))
    do, _, _ = orc.nearest(P, W, FB)
    C = max(np.abs(W).max(), np.abs(P).max())
    assert np.all((idx >= 0) & (idx < len(FB)))
    assert np.max(np.abs(d - do)) <= 1e-12 * C
    for i in range(0, len(P), max(1, len(P) // 40)):  # the triangle named holds the closest point
        dd, _ = orc.point_triangle(P[i], *T[idx[i]])
        assert abs(dd - do[i]) <= 1e-12 * C
    assert np.max(np.abs(np.linalg.norm((P - foot) / scale, axis=1) * scale - d)) <= 1e-12 * C
