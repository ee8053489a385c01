"""GPU: banded solves whose step of coefficients is longer than 64 KB although a block has
at most eight functions (rings of 140 and 168 cells whose functions reach across the whole
ring, so that the planner's reach is the ring's): eigenvalues against the dense oracle, and
the same bits beside a chain whose own steps are taken in pieces."""
import numpy as np
import pytest

from oracle import dense
from tests import _cases
from tests.test_gpu_band import _chain

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m0,L,lowest", [(8, 140, 0.138), (7, 168, 0.093)])
def test_long_steps_of_small_blocks(m0, L, lowest):
    from paper_1702_00339_gb300 import fock

    p = _chain(L, m0, lowest=lowest, per=1, defects=((3, 0.0),), k=4, n0=4, eps=1e-300)
    D = fock.problem_layout(p)["D"]
    assert D == L - 1 and (D + 1) * m0 * m0 > 8192
    H, S = dense.build(p)
    ctx = fock.Context(0)
    out = ctx.solve([p])[0]
    _cases.check(_cases.reference(p, H, S), out["evals"], None)
    beside = ctx.solve([_chain(40, 16, k=4, lowest=0.6, eps=1e-300), p])[1]
    assert np.array_equal(beside["evals"], out["evals"]) and beside["iters"] == out["iters"]
    ctx.close()
