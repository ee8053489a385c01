"""GPU: spectra with removed directions are sorted whole: the finite eigenvalues ascending,
then +inf, by the sort in shared memory and by the global one, of a plan and of a handle."""
import numpy as np
import pytest

from tests.test_gpu_periodic_blocks import _lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,m0", [((3, 4, 1), 7), ((5, 7, 11), 12), ((1, 1, 1), 2)])
def test_removed_directions_come_last(L, m0):
    from paper_1702_00339_gb300 import fock
    p = _lattice(L, m0, cut=True)
    ctx = fock.Context(0)
    b = ctx.assemble(p)
    out = ctx.solve([p])[0]
    for ev, blk in ((out["evals"], out["block_of"]), b.circulant_eig(), b.circulant_eig_range(0, p.ncell)):
        assert not np.isnan(ev).any() and np.isinf(ev[-1]) and np.isfinite(ev[0])
        assert np.all(ev[1:] >= ev[:-1])             # (a comparison, not a difference: inf - inf is no number)
        tie = ev[1:] == ev[:-1]
        assert np.all(blk[1:][tie] >= blk[:-1][tie])
        assert np.array_equal(np.bincount(blk, minlength=p.ncell), np.full(p.ncell, m0))
    ctx.close()
