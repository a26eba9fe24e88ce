"""Batched runs on both sides of the number of pairs from which warps that hold items of several
pairs add their sums lane by lane (256; the UpperBound kernels are separate instantiations):
every pair's bracket and counts equal its own single run's (whole numbers, and neither run cuts
queries)."""
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


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("order", [(1, 2, 3, 4), (3, 1)])
@pytest.mark.parametrize("n_pairs", [255, 256, 700])
def test_each_pair_as_its_single_run(hd, precision, order, n_pairs):
    rng = np.random.default_rng(n_pairs)
    VB, FB, _ = mg.torus(1.0, 0.3, 14, 7)
    pairs = []
    for i in range(n_pairs):  # 1 to 9 faces each, so 32 items span several pairs
        n = 1 + i % 9
        V = (VB[rng.integers(len(VB), size=n)][:, None] + rng.normal(0, 0.15, (n, 3, 3))).reshape(-1, 3)
        pairs.append((V, np.arange(3 * n, dtype=np.int32).reshape(n, 3)))
    prec = hd.HD_MIXED if precision == "mixed" else hd.HD_FP64
    o = hd.hd_options_default(tol_mode=hd.HD_TOL_REL, precision=prec, bound_order=order, flags=hd.HD_FLAG_EXACT_QUERIES)
    bvh = hd.hd_build_B(VB, FB)
    batch = hd.hd_hausdorff_batched([bvh] * n_pairs, pairs, 1e-3, o)
    for (V, F), b in list(zip(pairs, batch))[:: max(1, n_pairs // 60)]:
        r = hd.hd_hausdorff(bvh, V, F, 1e-3, o)
        assert (b["lower"], b["upper"], b["status"]) == (r["lower"], r["upper"], r["status"])
        for k in ("rounds", "splits", "queries", "pointtri_evals", "leaf_tests", "box_tests", "discards", "retired",
                  "peak_frontier", "node_visits", "long_queries"):
            assert b["stats"][k] == r["stats"][k], k
