"""hd_nearest answers each point on its own: the same bits whatever points come with it, in
whatever order.  Large sets in random order are regrouped by cell, sets in coherent order are
not, short ones are spread over more warps; all three must agree."""
import numpy as np
import pytest

import meshgen as mg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

N = (1 << 15) + 77  # above the size from which sets are regrouped


@pytest.fixture(scope="module")
def hd():
    from paper_2406_10357_gb300 import build

    build.build()
    import paper_2406_10357_gb300 as hd

    return hd


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("where", ["surface", "volume", "one_cell"])
def test_results_do_not_depend_on_the_order(hd, precision, dtype, where):
    prec = hd.HD_MIXED if precision == "mixed" else hd.HD_FP64
    rng = np.random.default_rng(5)
    VB, FB, _ = mg.torus(1.0, 0.3, 60, 30, 0.3, mg.stream(2, 2))
    if where == "surface":
        P = VB[FB].mean(1)[rng.integers(len(FB), size=N)] + rng.normal(0, 0.01, (N, 3))
    elif where == "volume":
        P = rng.uniform(-1.5, 1.5, (N, 3))
    else:
        P = np.array([1.3, 0.0, 0.0]) + rng.uniform(-1e-3, 1e-3, (N, 3))
    P = torch.from_numpy(P.astype(dtype)).cuda()
    bvh = hd.hd_build_B(VB, FB)

    def ask(x):
        return [y.cpu().numpy() for y in hd.hd_nearest(bvh, x, prec)]

    all_ = ask(P)
    by_x = torch.argsort(P[:, 0])  # neighbours mostly in the same cell
    for got, want in zip(ask(P[by_x]), all_):
        assert np.array_equal(got, want[by_x.cpu().numpy()])
    at = 0
    for n in (1, 2, 31, 33, 151, 153, 1217, 2433, 4865):
        for got, want in zip(ask(P[at:at + n]), all_):
            assert np.array_equal(got, want[at:at + n]), n
        at += n
