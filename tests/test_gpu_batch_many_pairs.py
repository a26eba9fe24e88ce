"""Batched runs on both sides of the number of pairs from which warps that hold items of several
pairs add their sums lane by lane (384; the UpperBound kernels are separate instantiations):
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
@pytest.mark.parametrize("n_pairs", [255, 256, 383, 384, 700])
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


def test_one_batch_costs_no_more_than_its_halves(hd):
    """260 pairs in one call against 130 and 130: a batch of more pairs fills the GPU better, so it
    must not take longer (2% for run-to-run differences)."""
    pairs, bvhs, rng = [], [], np.random.default_rng(2)
    for i in range(260):
        m = int(round(np.exp(rng.uniform(np.log(15), np.log(200)))))  # 900 to 160,000 faces
        P, F, N = mg.torus(1.0, 0.3, 2 * m, m)
        pairs.append((torch.from_numpy(P.astype(np.float32)).cuda(), torch.from_numpy(F).cuda()))
        Q = P + N * rng.normal(0, 10 ** rng.uniform(-4, -2), (len(P), 1))
        bvhs.append(hd.hd_build_B(torch.from_numpy(Q.astype(np.float32)).cuda(), pairs[-1][1]))
    o = hd.hd_options_default(tol_mode=hd.HD_TOL_REL, precision=hd.HD_MIXED)

    def ms(parts):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for s in parts:
            hd.hd_hausdorff_batched(bvhs[s], pairs[s], 1e-4, o)
        b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b)

    whole, halves = [slice(None)], [slice(0, 130), slice(130, 260)]
    ms(whole), ms(halves)
    t = np.median([(ms(whole), ms(halves)) for _ in range(7)], axis=0)
    print("one batch %.1f ms, two %.1f ms" % tuple(t))
    assert t[0] <= 1.02 * t[1]
