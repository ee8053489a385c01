"""GPU: the workspace that a context keeps between single calls stays within the context's
budget, beside its plans and handles, and is given back to a plan that needs the room."""
import pytest

from tests.test_gpu_handle_memory import _needs
from tests.test_gpu_periodic_blocks import _lattice

pytestmark = pytest.mark.gpu

PAGE = 2 << 20


def _product(torch, ctx):
    """A product of 1200 x 1200 with at least one range's partial sums: 11.5 MB of workspace or more."""
    A = torch.ones(1200, 4096, dtype=torch.float64, device="cuda")
    C = torch.zeros(1200, 1200, dtype=torch.float64, device="cuda")
    ctx.split_dgemm(1200, 1200, 4096, A.data_ptr(), 4096, 1, A.data_ptr(), 1, 4096, C.data_ptr(), 1200, 1, ksplit=2)
    assert bool((C == 4096.0).all())


def test_kept_workspace_counts_against_the_budget():
    torch = pytest.importorskip("torch")
    from paper_1702_00339_gb300 import fock
    p = _lattice((9, 5, 7), 12)                      # (a lattice's handle takes the same in every budget)
    need = _needs(fock, p)
    warm = fock.Context(0)                           # the kernels' own memory
    _product(torch, warm)
    warm.assemble(p)
    warm.close()
    free = lambda: torch.cuda.mem_get_info()[0]  # noqa: E731
    small = fock.Context(0, budget_bytes=1 << 20)
    before = free()
    _product(torch, small)
    assert before - free() <= 0                     # nothing of a context of 1 MB stays
    small.close()

    probe = fock.Context(0)
    before = free()
    _product(torch, probe)
    kept = before - free()
    assert kept >= 5 * PAGE                          # a context with room keeps it
    probe.close()
    ctx = fock.Context(0, budget_bytes=max(need, kept))
    before = free()
    _product(torch, ctx)
    assert before - free() == kept
    b = ctx.assemble(p)                              # beside which the workspace does not fit
    assert before - free() <= need + 2 * PAGE
    _product(torch, ctx)
    assert before - free() <= need + 2 * PAGE
    b.close()
    _product(torch, ctx)
    assert before - free() == kept
    ctx.close()
