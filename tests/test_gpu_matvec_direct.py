"""GPU: small products with a chain's operator go block by block instead of through
the embedding's transforms: against the dense matrices, and against the
transforms (the entry point without allocations always takes them), for block orders that
do and do not divide the threads, column counts about the groups of four, and rings whose
boundary and defect blocks lie far from the diagonal.

Bar: both sum at most N_b products of entries below max|A| and max|x|, with
rounding 2^-53 per term; the transforms carry about log2 M such errors: 64 of them."""
import numpy as np
import pytest

from oracle import dense
from tests import _cases
from tests.test_gpu_band import _chain

pytestmark = pytest.mark.gpu

CASES = {
    "box m0 1": dict(L=9, m0=1, lowest=0.6, k=3), "box m0 7": dict(L=12, m0=7, k=3), "box m0 32": dict(L=5, m0=32, k=3),
    "two cells": dict(L=2, m0=8, k=3), "ring with defects": dict(L=14, m0=4, per=1, defects=((3, 0.0), (9, 2.0)), k=3),
    "short ring": dict(L=7, m0=7, per=1, defects=((2, 0.0),), k=3),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_small_products(name):
    torch = pytest.importorskip("torch")
    from paper_1702_00339_gb300 import build, fock
    build.build()
    p = _chain(**CASES[name])
    H, S = dense.build(p)
    ctx = fock.Context(0)
    b = ctx.assemble(p)
    g = torch.Generator().manual_seed(5)
    for nvec in (1, 3, 4, 9):
        x = torch.randn(nvec, p.Nb, dtype=torch.float64, generator=g)
        for which, A in ((fock.FOCK_OP_H, H), (fock.FOCK_OP_S, S)):
            bar = 64 * _cases.U64 * p.Nb * np.max(np.abs(A)) * float(x.abs().max())
            y = torch.full_like(x, float("nan")).cuda()
            z = torch.full_like(x, float("nan")).cuda()
            xd = x.cuda()
            b.matvec_device(xd.data_ptr(), y.data_ptr(), nvec, which)
            b.matvec_noalloc(xd.data_ptr(), z.data_ptr(), nvec, which)
            torch.cuda.synchronize()
            assert np.max(np.abs(y.cpu().numpy() - x.numpy() @ A.T)) <= bar + 1e-11 * np.max(np.abs(A)) * np.sqrt(p.Nb)
            assert float((y - z).abs().max()) <= bar
    ctx.close()
