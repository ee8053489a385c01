"""GPU: the banded preconditioner's factor and solves at the sizes where they
can go wrong -- odd and single-function blocks, a ring planned as its whole
circulant (reach L - 1), more window rows than a CTA has threads, a block
column that does not fit shared memory, several column counts -- through the
block iteration, whose eigenvalues are compared with the dense oracle's and
whose iteration count (without defects) stays that of a shift-and-invert step."""
import numpy as np
import pytest

import lattice_inputs as li
from oracle import sinc
from tests import _cases

pytestmark = pytest.mark.gpu


def _tab(p):
    t, c, _ = sinc.table_for(p)
    return p.with_table(t, c)


def _chain(L, m0, b0=2.0, n0=6, k=6, lowest=0.25, ratio=2.2, per=0, defects=(), eps=1e-14):
    n = np.arange(m0)
    p = li.Problem(L=(L, 1, 1), periodic=(per, 0, 0), N=(L * n0 + (0 if per else 8), 16, 16), n0=n0, b0=b0, Z=np.array([1.0]),
                   frac=np.array([[0.5, 0.5, 0.5]]), exps=lowest * ratio ** (n % 8), ang=np.where(n < 8, 0, 1 + (n // 8 - 1) % 3),
                   centre=np.zeros(m0, int), R=16, k_eig=k, eps_support=eps)
    p.defects = [li.Defect(cell=(c, 0, 0), nucleus=0, newZ=z) for c, z in defects]
    return _tab(p)


CASES = [
    ("one function", dict(L=90, m0=1, lowest=0.6)),
    ("odd block", dict(L=29, m0=7, k=5)),
    ("band of reach L - 1 (short ring, defect)", dict(L=14, m0=7, per=1, defects=((3, 0.0),), k=4)),
    ("ring with a bound state (shift search)", dict(L=40, m0=4, per=1, defects=((5, 3.0),), k=6)),
    ("more window rows than threads", dict(L=40, m0=16, k=4, lowest=0.6, eps=1e-300)),
    ("block column beyond shared memory", dict(L=34, m0=32, k=4, lowest=0.6, eps=1e-220)),
    ("32 functions", dict(L=12, m0=32, k=8)),
    ("many columns", dict(L=40, m0=8, k=40)),
]


@pytest.mark.parametrize("name,kw", CASES, ids=[c[0] for c in CASES])
def test_band_preconditioner(name, kw):
    from oracle import dense
    from paper_1702_00339_gb300 import fock

    p = _chain(**kw)
    H, S = dense.build(p)
    ctx = fock.Context(0)
    out = ctx.solve([p])[0]
    _cases.check(_cases.reference(p, H, S), out["evals"], None)
    # the same problem among others (clusters of 8 instead of 16, two columns per CTA)
    many = ctx.solve([p] * 9 + [p] * (40 if p.m0 <= 8 else 0))
    for o in many:
        assert np.array_equal(o["evals"], out["evals"]) and o["iters"] == out["iters"]
    if not p.defects:
        assert out["iters"] <= 40
    ctx.close()
