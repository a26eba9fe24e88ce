"""hd_stats.discards counts each discard for the bound that decided it.  In FP64 an FP32 filter
discards most items; the bound counted has to be the one the FP64 cascade finds first.

With a tolerance above every bound nothing is split, so the discards are those of A's faces at
the final l, and hd_upper_bounds, which runs the cascade in double throughout, names the deciding
bound of each: whole numbers, equal.  The batched MIXED run, which gathers the items that reach
u3, has to count as single runs do."""
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


def _needles(rng, n, offset):
    """B: a grid of unit squares, exact in float32.  A: acute needles over its edges, so that their
    vertices are nearest to two triangles; a float pair hides up to a tenth of their width at
    2^23.  u2 = R + d lies within 1% of 6e-3."""
    X, Y = np.meshgrid(np.arange(33), np.arange(33), indexing="ij")
    VB = (offset + np.stack([X, Y, 0 * X], -1).reshape(-1, 3)).astype(np.float32)
    i = (33 * X[:-1, :-1] + Y[:-1, :-1]).reshape(-1)
    FB = np.concatenate([np.stack([i, i + 33, i + 34], 1), np.stack([i, i + 34, i + 1], 1)]).astype(np.int32)
    c = np.stack([rng.integers(1, 31, n), rng.integers(1, 31, n) + 0.25, 1e-3 * rng.uniform(0.95, 1.05, n)], 1)
    w = 2e-7 * rng.uniform(0.5, 1.5, n)
    T = np.repeat((c + offset)[:, None], 3, 1)
    T[:, :, 0] += [5e-3, -5e-3, -5e-3]
    T[:, 1, 1] -= w / 2
    T[:, 2, 1] += w / 2
    return T.reshape(-1, 3), np.arange(3 * n, dtype=np.int32).reshape(n, 3), VB, FB, 6e-3


def _pair(kind, scale, shift):
    """A, B and the value l starts from (chosen so that each of the first bounds decides some faces)."""
    rng = np.random.default_rng(1)
    if kind == "needles":
        return _needles(rng, 4000, shift)
    if kind == "slivers":
        p = mg.workload(3, 0.02)
        return np.asarray(p.VA, float) * scale + shift, p.FA, np.asarray(p.VB, float) * scale + shift, p.FB, 0.15 * scale
    P, F, N = mg.torus(1.0, 0.3, 120, 61)
    VB, FB, _ = mg.torus(1.0, 0.3, 90, 40, 0.3, mg.stream(2, 2))
    VA = P + N * mg.stream(4, 1).normal(len(P), 3e-3)[:, None]
    return VA * scale + shift, F, VB * scale + shift, FB, 0.044 * scale


CASES = [("torus", 1.0, 0.0), ("torus", 1.0, 1e4), ("torus", 1.0, 1e6), ("torus", 1e-12, 0.0), ("torus", 1e-25, 0.0),
         ("torus", 1e15, 0.0), ("torus", 1e25, 0.0), ("slivers", 1.0, 0.0), ("slivers", 1.0, 1e3), ("needles", 1.0, 0.0),
         ("needles", 1.0, 2.0**23)]


@pytest.mark.parametrize("kind,scale,shift", CASES)
@pytest.mark.parametrize("order", [(1, 2, 3, 4), (2, 1, 3), (1, 2), (3, 1), (4, 3), (4, 2, 1, 3), (1, 4), (2,)])
def test_fp64_counts_the_bound_that_decides(hd, kind, scale, shift, order):
    VA, FA, VB, FB, l0 = _pair(kind, scale, shift)
    bvh = hd.hd_build_B(VB, FB)
    o = hd.hd_options_default(bound_order=order, flags=hd.HD_FLAG_EXACT_QUERIES)
    d, idx, q, _ = hd.hd_nearest(bvh, torch.from_numpy(VA).cuda(), hd.HD_FP64)
    f = torch.from_numpy(FA).long().cuda()
    args = (torch.from_numpy(VA).cuda()[f].reshape(-1, 9), d[f], idx[f], q[f].reshape(-1, 9))
    for l in (0.0, l0):
        r = hd.hd_hausdorff_from(bvh, VA, FA, 1e30 * scale, l, o)
        assert r["stats"]["splits"] == 0
        _, code = hd.hd_upper_bounds(bvh, *args, r["lower"], o)
        want = np.bincount(code.cpu().numpy(), minlength=6)[:5]
        got = list(r["stats"]["discards"].values())[:5]
        print(want, got)
        assert got == list(want)


@pytest.mark.parametrize("k", [2, 3])
def test_batched_mixed_counts_as_single_runs(hd, k):
    p = mg.workload(k, 0.05)
    bvh = hd.hd_build_B(p.VB, p.FB)
    o = hd.hd_options_default(tol_mode=hd.HD_TOL_REL, precision=hd.HD_MIXED, flags=hd.HD_FLAG_EXACT_QUERIES)
    r = hd.hd_hausdorff(bvh, p.VA, p.FA, 1e-5, o)["stats"]
    b = hd.hd_hausdorff_batched([bvh], [(p.VA, p.FA)], 1e-5, o)[0]["stats"]
    assert (b["discards"], b["splits"], b["retired"]) == (r["discards"], r["splits"], r["retired"])
