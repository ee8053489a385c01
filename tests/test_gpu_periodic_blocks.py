"""GPU: spectra of periodic lattices over the shapes at which the pipeline of
Fourier-block kernels changes what it does: block orders at and around the
limits of its launch shapes (8, 16, 32), lattices whose last or only long
axis is not the third, numbers of blocks off the groups of eight, blocks with
directions cut and without.  Against LAPACK on the oracle's Fourier blocks
with the bar of tests/_cases.py; batched together the spectra are the same
numbers, whatever their neighbours and the chunks of the workspace."""
import numpy as np
import pytest

import lattice_inputs as li
from oracle import dense
from tests import _cases

pytestmark = pytest.mark.gpu

SHAPES = [((5, 1, 1), 1), ((7, 1, 1), 2), ((3, 4, 1), 7), ((2, 2, 3), 8), ((1, 1, 9), 9), ((1, 5, 1), 16),
          ((3, 1, 2), 17), ((2, 3, 1), 31), ((2, 1, 2), 32)]


def _lattice(L, m0, cut=False):
    """m0 functions: s and p about two centres in turn, exponents 0.4 * 3^i; cut: the last
    repeats the first."""
    rng = np.random.default_rng(m0)
    n0 = 12
    k = np.arange(m0)
    ex, ce, ang = 0.4 * 3.0 ** (k // 8), k % 2, (k // 2) % 4
    if cut:
        ex[-1], ce[-1], ang[-1] = ex[0], ce[0], ang[0]
    frac = np.array([[0.3, 0.45, 0.5], [0.7, 0.55, 0.4]]) + 0.02 * rng.random((2, 3))
    p = li.Problem(L=tuple(L), periodic=(1, 1, 1), N=tuple(l * n0 for l in L), n0=n0, b0=4.0, Z=np.array([1.0, 2.0]),
                   frac=frac, exps=ex, ang=ang, centre=ce, R=12)
    return _cases.with_table(p)


@pytest.fixture(scope="module")
def ctx():
    from paper_1702_00339_gb300 import build, fock
    build.build()
    c = fock.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("cut", [False, True])
@pytest.mark.parametrize("L,m0", SHAPES)
def test_spectrum_against_lapack(ctx, L, m0, cut):
    if cut and m0 < 2:
        pytest.skip("one function has nothing to repeat")
    p = _lattice(L, m0, cut)
    H, S = dense.build(p)
    o = ctx.solve([p])[0]
    assert o["status"] == 0
    _cases.report(f"periodic_blocks_{L}_{m0}_{cut}", _cases.check(_cases.reference(p, H, S), o["evals"], o["block_of"]))


def test_batches_and_budgets_give_the_same_numbers(ctx):
    from paper_1702_00339_gb300 import fock
    ps = [_lattice(L, m0, cut) for L, m0 in SHAPES for cut in (False, True) if m0 > 1]
    ps.insert(3, _lattice((9, 5, 7), 12, True))
    alone = [ctx.solve([p])[0] for p in ps]
    small = fock.Context(0, budget_bytes=3 << 20)     # less than the largest lattice takes in one chunk
    for outs in (ctx.solve(ps), small.solve(ps[3:4])):
        first = 0 if len(outs) == len(ps) else 3
        for a, o in zip(alone[first:], outs):
            assert np.array_equal(a["evals"], o["evals"]) and np.array_equal(a["block_of"], o["block_of"])
    small.close()
