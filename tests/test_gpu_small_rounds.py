"""The small-round kernel's hand-back: rounds over at most 512 sub-triangles (FP64: 64) that hand off
at most 64 queries run inside one cluster, larger ones on the whole GPU.  Runs that cross these
limits give what HD_FLAG_NO_SMALL_ROUNDS gives."""
import numpy as np
import pytest

import meshgen as mg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

FRONT = {"mixed": 512, "fp64": 64}
LONG = 64


@pytest.fixture(scope="module")
def hd():
    from paper_2406_10357_gb300 import build

    build.build()
    import paper_2406_10357_gb300 as hd

    return hd


def _both(hd, precision, VA, FA, VB, FB, tol):
    """(with small rounds, launches of their kernel, without them), every query exact."""
    prec = hd.HD_MIXED if precision == "mixed" else hd.HD_FP64
    bvh = hd.hd_build_B(VB, FB)
    opt = [hd.hd_options_default(tol_mode=hd.HD_TOL_REL, precision=prec, flags=hd.HD_FLAG_EXACT_QUERIES | f)
           for f in (0, hd.HD_FLAG_NO_SMALL_ROUNDS)]
    hd.hd_trace_enable(True)
    hd.hd_trace_read(True)
    a = hd.hd_hausdorff(bvh, VA, FA, tol, opt[0])
    small = hd.hd_trace_read(True)["small_rounds"]["launches"]
    hd.hd_trace_enable(False)
    return a, small, hd.hd_hausdorff(bvh, VA, FA, tol, opt[1])


def _same(a, b):
    assert (a["lower"], a["upper"], a["status"]) == (b["lower"], b["upper"], b["status"])
    for k in ("rounds", "splits", "queries", "long_queries", "retired", "peak_frontier", "discards", "promoted"):
        assert a["stats"][k] == b["stats"][k], k


@pytest.mark.parametrize("precision,nu,nv", [("mixed", 12, 8), ("mixed", 20, 12), ("fp64", 6, 5), ("fp64", 8, 4)])
def test_frontier_passes_the_limit_and_comes_back(hd, precision, nu, nv):
    """A coarse torus whose vertices lie on a fine one: every face sags by about as much, so the
    frontier starts below the limit, grows past it while l is low, and shrinks to a few items."""
    VB, FB, _ = mg.torus(1.0, 0.3, 90, 40)
    P, F, N = mg.torus(1.0, 0.3, nu, nv)
    VA = P + N * mg.stream(4, 1).normal(len(P), 1e-3)[:, None]
    a, small, b = _both(hd, precision, VA.astype(np.float32), F, VB.astype(np.float32), FB, 1e-6)
    s = a["stats"]
    print(precision, len(F), "faces, rounds", s["rounds"], "peak", s["peak_frontier"], "small", small)
    assert a["status"] == hd.HD_OK
    _same(a, b)
    assert len(F) <= FRONT[precision] < s["peak_frontier"] and small >= 2


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_small_round_with_many_long_queries(hd, precision):
    """Small rounds around the centre of a sphere, as far from all of it: every midpoint near it
    is handed off, more than a small round takes."""
    n = 60 if precision == "fp64" else 100
    rng = np.random.default_rng(5)
    VB, FB = mg.superquadric(1.0, 1.0, 1.0, 80, 40, 0.0, mg.stream(7, 1))
    VA = rng.normal(0, 0.02, (3 * n, 3)).astype(np.float32)
    a, small, b = _both(hd, precision, VA, np.arange(3 * n, dtype=np.int32).reshape(n, 3), np.asarray(VB, np.float32), FB, 3e-3)
    s = a["stats"]
    print(precision, "rounds", s["rounds"], "peak", s["peak_frontier"], "long", s["long_queries"], "small", small)
    assert a["status"] == hd.HD_OK and s["rounds"] >= 1 and s["long_queries"] - 3 * n > LONG
    _same(a, b)
