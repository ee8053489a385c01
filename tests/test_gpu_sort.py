"""GPU: the sorts of eigenvalues with their Fourier indices, at sizes either side
of the shared-memory tile and of a power of two: a range of Fourier blocks
returns the full solve's pairs of that range, ascending."""
import numpy as np
import pytest

from tests import _cases

pytestmark = pytest.mark.gpu


def test_range_sizes_sort_like_the_full_solve():
    from paper_1702_00339_gb300 import fock

    p = _cases.periodic_3d_small(L=(8, 8, 6))     # 384 blocks of 16
    ctx = fock.Context(0)
    b = ctx.assemble(p)
    ev, blk = b.circulant_eig()
    assert np.all(np.diff(ev) >= 0) or not np.all(np.isfinite(ev))
    for j0, j1 in [(0, 1), (3, 4), (0, 128), (0, 129), (1, 128), (0, 256), (5, 262), (0, 384)]:
        e2, b2 = b.circulant_eig_range(j0, j1)
        inside = (blk >= j0) & (blk < j1)
        order = np.lexsort((blk[inside], ev[inside]))
        assert np.array_equal(e2, ev[inside][order]) and np.array_equal(b2, blk[inside][order])
    ctx.close()
