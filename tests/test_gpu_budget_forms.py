"""GPU: budgets near the least that a plan of the library's problems takes. A plan that does
not fit in its fast form gives up chunk workspace, split sums, the factor from both ends and
the factor, in this order, before it is refused: each form solves the problem, and the least
one takes no more bytes than these plans did before there were fast forms."""
import re

import numpy as np
import pytest

from oracle import dense
from tests import _cases
from tests.test_gpu_band import _chain
from tests.test_gpu_periodic_blocks import _lattice

pytestmark = pytest.mark.gpu


def _least(fock, ps):
    tiny = fock.Context(0, budget_bytes=1 << 12)
    with pytest.raises(fock.FockError) as e:
        tiny.plan(ps)
    tiny.close()
    assert e.value.code == fock.FOCK_ENOMEM
    return int(re.search(r"needs (\d+) bytes", str(e.value)).group(1))


@pytest.mark.parametrize("kw,took", [(dict(L=64, m0=8, k=16), 4445072), (dict(L=48, m0=16, k=8, lowest=0.4), 7453264)])
def test_chains_solve_in_every_form(kw, took):
    from paper_1702_00339_gb300 import fock
    p = _chain(**kw)
    H, S = dense.build(p)
    ref = _cases.reference(p, H, S)
    least = _least(fock, [p])
    assert least <= took
    its = []
    for f in (1.0, 1.1, 1.2, 1.3, 1.5, 4.0):
        ctx = fock.Context(0, budget_bytes=int(least * f))
        out = ctx.solve([p])[0]
        _cases.check(ref, out["evals"], None)
        its.append(out["iters"])
        ctx.close()
    assert its[0] > its[-1]                          # the circulant inverse at the least, the factor with room
    with pytest.raises(fock.FockError):
        fock.Context(0, budget_bytes=least - 1).plan([p])


def test_lattices_and_rings_beside_chains_solve_in_every_form():
    from paper_1702_00339_gb300 import fock
    ps = [_lattice((9, 5, 7), 12, True), _chain(L=40, m0=8, k=6), _chain(L=21, m0=4, k=4, per=1, defects=((3, 0.0),)), _lattice((14, 14, 14), 8)]
    wide = fock.Context(0)
    ref = wide.solve(ps)
    wide.close()
    least = _least(fock, ps)
    assert least <= 15138576
    for f in (1.0, 1.05, 1.2, 1.5):
        ctx = fock.Context(0, budget_bytes=int(least * f))
        for a, o, p in zip(ref, ctx.solve(ps), ps):
            if p.k_eig and a["block_of"] is None:
                assert np.allclose(o["evals"], a["evals"], rtol=0, atol=1e-9 * np.max(np.abs(a["evals"])))
            else:                                    # chunks do not change a periodic spectrum
                assert np.array_equal(o["evals"], a["evals"]) and np.array_equal(o["block_of"], a["block_of"])
        ctx.close()
