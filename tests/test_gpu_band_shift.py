"""GPU: bound states that make the first shift fail while a ring's banded factor is made a
launch per block column: found on one side, on the other, on both, and only in the middle
rows.  The search then goes on with one cluster per problem, so the numbers are those of a
batch, which starts there, and the dense oracle's."""
import numpy as np
import pytest

from oracle import dense
from tests import _cases
from tests.test_gpu_band import _chain

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells", [(1,), (22,), (1, 22), (12,)])
def test_failed_first_shift_by_columns(cells):
    from paper_1702_00339_gb300 import fock

    kw = dict(m0=20, lowest=0.6, k=4, per=1)
    D = fock.problem_layout(_chain(L=40, defects=((5, 3.0),), **kw))["D"]
    assert D * (D + 1) // 2 * 20 ** 3 >= 150000 and D * (D + 1) // 2 >= 16 and 24 >= 2 * D + 2   # by columns, from both ends
    p = _chain(L=24, defects=tuple((c, 3.0) for c in cells), **kw)
    H, S = dense.build(p)
    ctx = fock.Context(0)
    out = ctx.solve([p])[0]
    _cases.check(_cases.reference(p, H, S), out["evals"], None)
    for o in ctx.solve([p] * 9):
        assert np.array_equal(o["evals"], out["evals"]) and o["iters"] == out["iters"]
    ctx.close()
