"""GPU: the Rayleigh-Ritz kernel at the sizes where it can go wrong -- small,
odd and largest bases, either side of the size that changes the launch, the
whole-space block -- against the dense oracle, and the same bits for every
number of problems (which sets the CTAs per problem)."""
import numpy as np
import pytest

import lattice_inputs as li
from oracle import dense, sinc
from tests import _cases

pytestmark = pytest.mark.gpu


def _chain(L, m0, k):
    n0 = 6
    p = li.Problem(L=(L, 1, 1), periodic=(0, 0, 0), N=(L * n0 + 8, 16, 16), n0=n0, b0=2.0, Z=np.array([1.0]),
                   frac=np.array([[0.5, 0.5, 0.5]]), exps=0.25 * 2.5 ** np.arange(m0), ang=np.zeros(m0, int),
                   centre=np.zeros(m0, int), R=16, k_eig=k)
    t, c, _ = sinc.table_for(p)
    return p.with_table(t, c)


# (cells, functions, wanted pairs): block k + max(4, k / 8), basis three times that
CASES = [(24, 4, 1), (31, 3, 2), (30, 4, 17), (30, 4, 18), (50, 4, 40), (76, 4, 75), (21, 4, 16)]


@pytest.mark.parametrize("L,m0,k", CASES)
def test_rayleigh_ritz_sizes(L, m0, k):
    from paper_1702_00339_gb300 import fock

    p = _chain(L, m0, k)
    H, S = dense.build(p)
    ctx = fock.Context(0)
    out = ctx.solve([p])[0]
    assert out["status"] == 0
    _cases.check(_cases.reference(p, H, S), out["evals"], None)
    for count in (3, 40, 80):
        for o in ctx.solve([p] * count):
            assert np.array_equal(o["evals"], out["evals"]) and o["iters"] == out["iters"]
    ctx.close()
