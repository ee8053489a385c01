"""GPU: products with far more columns than one grid dimension has groups for (65535 of
four or eight): block by block and, above its limit, through the transforms, on the
smallest chain, against the dense matrix on the device (at most four products an entry,
with the transforms' rounding: 64 units)."""
import numpy as np
import pytest

from oracle import dense
from tests import _cases
from tests.test_gpu_band import _chain

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nvec", [4 * 65535 + 1, 1400001])
def test_more_columns_than_a_grid_dimension(nvec):
    torch = pytest.importorskip("torch")
    from paper_1702_00339_gb300 import fock
    p = _chain(L=2, m0=1, lowest=0.6, k=1)
    H, _ = dense.build(p)
    ctx = fock.Context(0)
    b = ctx.assemble(p)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(nvec, p.Nb, dtype=torch.float64, device="cuda", generator=g)
    y = torch.full_like(x, float("nan"))
    b.matvec_device(x.data_ptr(), y.data_ptr(), nvec, fock.FOCK_OP_H)
    torch.cuda.synchronize()
    ref = x @ torch.tensor(H.T.copy(), device="cuda")
    bar = (64 * _cases.U64 * p.Nb * float(x.abs().max()) + 1e-11 * np.sqrt(p.Nb)) * np.max(np.abs(H))
    assert float((y - ref).abs().max()) <= bar
    ctx.close()
