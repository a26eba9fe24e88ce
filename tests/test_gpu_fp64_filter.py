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


def _perturbed_copy(nu, nv, sigma, scale, shift, dtype):
    """A torus and a copy of it moved along its normals: A's edges follow B's, so vertices of A's
    sub-triangles lie close to u3's bisecting planes."""
    P, F, N = mg.torus(1.0, 0.3, nu, nv)
    g = mg.stream(11, nu)
    VA, VB = P * scale + shift, (P + N * g.normal(len(P), sigma)[:, None]) * scale + shift
    return VA.astype(dtype), F, VB.astype(dtype), F.copy()


@pytest.mark.parametrize("nu,nv,sigma,tol", [(3, 3, 1e-1, 1e-4), (16, 9, 1e-2, 1e-5), (24, 11, 1e-3, 1e-5)])
@pytest.mark.parametrize("scale,shift", [(1.0, 0.0), (1.0, 1e4), (1e-25, 0.0), (1e25, 0.0)])
@pytest.mark.parametrize("order", [(1, 2, 3, 4), (3, 1), (4, 3)])
def test_bracket_fp64_filtered(hd, orc, nu, nv, sigma, tol, scale, shift, order):
    """The bracket of a pair whose bounds the filter decides meets the oracle's and a tighter
    one's, alone and in a batch; the two runs split the same sub-triangles.  Both sides hold h
    up to their rounding, 1e-12 of the largest coordinate."""
    VA, FA, VB, FB = _perturbed_copy(nu, nv, sigma, scale, shift, np.float64)
    o = hd.hd_options_default(tol_mode=hd.HD_TOL_REL, bound_order=order)
    bvh = hd.hd_build_B(VB, FB)
    r = hd.hd_hausdorff(bvh, VA, FA, tol, o)
    rb, _ = hd.hd_hausdorff_batched([bvh, bvh], [(VA, FA), (VA, FA)], tol, o)
    ro = orc.hausdorff(VA, FA, VB, FB, tol, 1)
    rt = orc.hausdorff(VA, FA, VB, FB, tol / 10, 1)
    eps, C = r["stats"]["eps_abs"], max(np.abs(VA).max(), np.abs(VB).max())
    for x in (r, rb):
        assert x["status"] == hd.HD_OK and x["upper"] - x["lower"] <= eps * (1 + 1e-12) + 1e-12 * C
        for y in (ro, rt):
            assert max(x["lower"], y["lower"]) <= min(x["upper"], y["upper"]) + 1e-12 * C
    assert r["stats"]["splits"] == rb["stats"]["splits"] and r["stats"]["rounds"] == rb["stats"]["rounds"]
