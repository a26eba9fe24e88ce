"""FP64 results are those of FP64 arithmetic alone, whatever FP32 decides on the way: distances,
triangles (the choice among equal distances too), closest points, lower bounds and counts bit for
bit against digests made by a library without the filters (tests/golden/fp64_bits.py).  Upper
bounds come from kernels whose roundings a compiler may contract in another way: they agree
within 1e-12 of the largest coordinate, as a bound takes under a few hundred roundings of it."""
import importlib.util
import json
import os

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

_spec = importlib.util.spec_from_file_location(
    "fp64_bits", os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "fp64_bits.py"))
G = importlib.util.module_from_spec(_spec)
_spec.loader.exec_module(G)


@pytest.fixture(scope="module")
def hd():
    from paper_2406_10357_gb300 import build

    build.build()
    import paper_2406_10357_gb300 as hd

    return hd


@pytest.fixture(scope="module")
def want():
    with open(G.PATH) as f:
        return json.load(f)


@pytest.mark.parametrize("case", G.NEAREST, ids=G.key)
def test_nearest(hd, want, case):
    assert G.nearest(hd, *case) == want["nearest"][G.key(case)]


@pytest.mark.parametrize("case", G.BRACKETS, ids=G.key)
def test_bracket(hd, want, case):
    got, ref = G.bracket(hd, *case), want["bracket"][G.key(case)]
    C = (case[1] + 25.0) * 2.0 ** case[0]
    assert abs(float.fromhex(got[1]) - float.fromhex(ref[1])) <= 1e-12 * C
    assert got[0] == ref[0] and got[2:] == ref[2:]
