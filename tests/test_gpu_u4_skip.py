"""The paper-order kernels leave u4 out where it cannot lower U (u4_idle).  The order (2, 1, 3, 4)
runs the general kernels, which evaluate it for every item they keep; U is the minimum of the
same bounds either way, so the two runs must agree in every value and count."""
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


def _pair(kind):
    if kind == "copy":
        P, F, N = mg.torus(1.0, 0.3, 60, 31)
        return P.astype(np.float32), F, (P + N * mg.stream(4, 1).normal(len(P), 1e-3)[:, None]).astype(np.float32), F.copy(), 1e-5
    if kind == "far":  # an offset much larger than the edges, and one mesh shifted
        P, F, _ = mg.torus(1.0, 0.3, 60, 31)
        return P.astype(np.float32), F, (1.3 * P + 0.1).astype(np.float32), F.copy(), 1e-4
    p = mg.workload(*kind)
    return p.VA, p.FA, p.VB, p.FB, p.tol


@pytest.mark.parametrize("kind", ["copy", "far", (2, 0.05), (3, 0.02), (5, 0.01)])
@pytest.mark.parametrize("batched", [False, True])
def test_skipping_u4_changes_nothing(hd, kind, batched):
    VA, FA, VB, FB, tol = _pair(kind)
    bvh = hd.hd_build_B(VB, FB)
    got = []
    for order in ((1, 2, 3, 4), (2, 1, 3, 4)):
        o = hd.hd_options_default(tol_mode=hd.HD_TOL_REL, precision=hd.HD_MIXED, bound_order=order,
                                  flags=hd.HD_FLAG_EXACT_QUERIES)
        r = hd.hd_hausdorff_batched([bvh], [(VA, FA)], tol, o)[0] if batched else hd.hd_hausdorff(bvh, VA, FA, tol, o)
        assert r["status"] == hd.HD_OK
        got.append((r["lower"], r["upper"]) + tuple(r["stats"][k] for k in ("rounds", "splits", "retired", "promoted")))
    assert got[0] == got[1]
