"""Pivots of every column of a panel, the last one included: matrices whose
pivot rows are known (a row permutation of a dominant upper triangle with a
known exchange at every column), batched so that many panels are in flight,
at panel widths of 1 to 32 columns, one to several panels, and one to sixteen
blocks per panel.  A wrong exchange puts a wrong row on top, so the solution
is wrong by its own size; the bound is the solves' backward error 8 n u."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs():
    from paper_1608_06871_gb300.build import build
    build()
    import paper_1608_06871_gb300 as mod
    return mod


@pytest.mark.parametrize("dtype,u", [(torch.complex128, 2.0 ** -53), (torch.complex64, 2.0 ** -24)])
@pytest.mark.parametrize("batch,n", [(256, 1), (256, 2), (256, 7), (256, 31), (256, 32), (256, 33), (150, 64), (40, 97),
                                     (4, 300), (1, 600), (1, 1500)])
def test_last_pivot_of_a_panel(hs, dtype, u, batch, n):
    g = torch.Generator().manual_seed(n)
    U = torch.randn((batch, n, n), generator=g, dtype=torch.float64).triu(1) / (4.0 * n)
    A = (U + torch.eye(n, dtype=torch.float64)).to(dtype)
    order = (torch.arange(n) + 1) % n  # the pivot of every column but the last lies in the last row
    A = A[:, order].contiguous()
    X0 = torch.complex(torch.randn((batch, n, 1), generator=g, dtype=torch.float64),
                       torch.randn((batch, n, 1), generator=g, dtype=torch.float64)).to(dtype)
    B = (A.to(torch.complex128) @ X0.to(torch.complex128)).to(dtype)
    X = B.cuda().contiguous()
    hs.hs_lu_solve(A.cuda().contiguous(), X)
    r = (A.to(torch.complex128) @ X.cpu().to(torch.complex128) - B.to(torch.complex128)).abs().amax(dim=(1, 2))
    scale = A.abs().double().sum(dim=2).amax(dim=1) * X.cpu().abs().double().amax(dim=(1, 2)) + B.abs().double().amax(dim=(1, 2))
    assert bool((r <= 8 * n * u * scale).all())
