"""GPU: the banded preconditioner made from both ends, at the shortest chains that it
takes (L = 2 D + 2; one row less goes from one end), halves of equal and unequal
length, and blocks large enough for a launch per block column: alone (by columns,
where the blocks are worth it) and among others (one cluster per problem) the same bits,
eigenvalues against the dense oracle, and the iteration count of a shift-and-invert
step; with a bound state the first shift fails and the cluster kernel searches on."""
import numpy as np
import pytest

from oracle import dense
from tests import _cases
from tests.test_gpu_band import _chain

pytestmark = pytest.mark.gpu

CASES = [(8, 1.5, extra, ()) for extra in (1, 2, 3, 6)] + [(20, 0.6, extra, ()) for extra in (1, 2, 3)] + \
        [(32, 1.2, 5, ()), (20, 0.6, 8, ((5, 3.0),))]


@pytest.mark.parametrize("m0,lowest,extra,defects", CASES)
def test_from_both_ends(m0, lowest, extra, defects):
    from paper_1702_00339_gb300 import fock

    kw = dict(m0=m0, lowest=lowest, k=4, per=1 if defects else 0, defects=defects)
    D = fock.problem_layout(_chain(L=40, **kw))["D"]
    p = _chain(L=2 * D + extra, **kw)
    assert fock.problem_layout(p)["D"] == D
    H, S = dense.build(p)
    ctx = fock.Context(0)
    out = ctx.solve([p])[0]
    _cases.check(_cases.reference(p, H, S), out["evals"], None)
    for o in ctx.solve([p] * 9):
        assert np.array_equal(o["evals"], out["evals"]) and o["iters"] == out["iters"]
    if not defects:
        assert out["iters"] <= 40
    ctx.close()
