"""hd_upper_bounds in FP64 runs point-triangle tests only for items that reach u3.  A cascade of u1
alone has none: it takes a small part of the time of u3 alone, whose four to fifteen tests per
item bound it.  Three tests per item would by themselves be a third of the latter's time."""
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


def test_bounds_without_u3_run_no_point_triangle_tests(hd):
    P, F, N = mg.torus(1.0, 0.3, 500, 300)
    VB, FB, _ = mg.torus(1.0, 0.3, 224, 112, 0.3, mg.stream(2, 2))
    V = torch.from_numpy(P + N * mg.stream(4, 1).normal(len(P), 1e-3)[:, None]).cuda()
    bvh = hd.hd_build_B(VB, FB)
    d, idx, q, _ = hd.hd_nearest(bvh, V, hd.HD_FP64)
    f = torch.from_numpy(F).long().cuda()
    args = (V[f].reshape(-1, 9).contiguous(), d[f].contiguous(), idx[f].contiguous(), q[f].reshape(-1, 9).contiguous())

    def us(order):
        o = hd.hd_options_default(bound_order=order)
        t = []
        for i in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(5):
                hd.hd_upper_bounds(bvh, *args, 0.0, o)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b) * 200)
        return float(np.median(t[3:]))

    u1, u3 = us((1,)), us((3,))
    print("u1 alone %.0f us, u3 alone %.0f us" % (u1, u3))
    assert u1 < 0.2 * u3
