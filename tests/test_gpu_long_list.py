"""Rounds whose handed-off queries grow from few to many: the host leaves the reordering of the list
out where the round before handed off few, and the cooperative pass must then take this round's
list in its own order, not the copy an earlier round reordered."""
import numpy as np
import pytest

import meshgen as mg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

SORT_MIN = 2048  # handed-off queries from which a list is reordered


@pytest.fixture(scope="module")
def hd():
    from paper_2406_10357_gb300 import build

    build.build()
    import paper_2406_10357_gb300 as hd

    return hd


def _pair(n):
    """B: a unit sphere and a speck at every corner of A that lies off it.  A: triangles (2m - u, u,
    -2m - u) for orthogonal unit vectors m and u.  Their corners are on B; so are the midpoints of
    their edges, m, -m and -u, whose queries are short; the midpoint of m and -m in the round
    after is the centre, as far from every triangle of the sphere: each such query is handed off."""
    rng = np.random.default_rng(3)
    VS, FS = mg.superquadric(1.0, 1.0, 1.0, 80, 40, 0.0, mg.stream(7, 1))
    m = rng.normal(size=(n, 3))
    m /= np.linalg.norm(m, axis=1)[:, None]
    u = np.cross(m, rng.normal(size=(n, 3)))
    u /= np.linalg.norm(u, axis=1)[:, None]
    VA = np.stack([2 * m - u, u, -2 * m - u], 1)
    far = VA[:, [0, 2]].reshape(-1, 3)
    speck = (far[:, None] + 1e-4 * rng.normal(size=(len(far), 3, 3))).reshape(-1, 3)
    VB = np.concatenate([np.asarray(VS, float), speck])
    FB = np.concatenate([FS, len(VS) + np.arange(len(speck)).reshape(-1, 3)]).astype(np.int32)
    return (VA.reshape(-1, 3).astype(np.float32), np.arange(3 * n, dtype=np.int32).reshape(n, 3), VB.astype(np.float32), FB)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_few_handed_off_then_many(hd, precision):
    n = 3000
    VA, FA, VB, FB = _pair(n)
    prec = hd.HD_MIXED if precision == "mixed" else hd.HD_FP64
    bvh = hd.hd_build_B(VB, FB)

    def run(rounds, batched=False):
        o = hd.hd_options_default(tol_mode=hd.HD_TOL_REL, precision=prec, max_rounds=rounds, flags=hd.HD_FLAG_EXACT_QUERIES)
        if batched:
            return hd.hd_hausdorff_batched([bvh], [(VA, FA)], 1e-4, o)[0]
        return hd.hd_hausdorff(bvh, VA, FA, 1e-4, o)

    one, two = run(1), run(2)
    assert one["stats"]["splits"] == n and two["stats"]["splits"] == 5 * n
    few, many = one["stats"]["long_queries"], two["stats"]["long_queries"] - one["stats"]["long_queries"]
    print("handed off:", few, "then", many)
    assert few * 8 < SORT_MIN <= many  # eight: twice the growth of a round
    # the batched run does not reorder its lists
    b = run(2, batched=True)
    assert (two["lower"], two["upper"], two["status"]) == (b["lower"], b["upper"], b["status"])
    for k in ("queries", "long_queries", "retired", "discards"):
        assert two["stats"][k] == b["stats"][k], k
