"""Emulated FP64 products at the lower end of the exponent range: rows of
subnormal and barely normal entries, whose products with large ones are
ordinary numbers."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def hs():
    from paper_1608_06871_gb300.build import build
    build()
    import paper_1608_06871_gb300 as mod
    return mod


def _randn(shape, seed):
    return torch.randn(shape, generator=torch.Generator().manual_seed(seed), dtype=torch.float64)


@pytest.mark.parametrize("e", [-1000, -1015, -1020, -1022, -1023, -1030, -1050])
def test_rows_of_tiny_entries(hs, e):
    """Scaling by powers of two is exact, so the product of the scaled-up rows is the reference; the
    bound is that of the scheme, 5 k 2^-55 max|A_i.| max|B_.j|, and the rounding of the result."""
    m, n, k = 200, 70, 300
    A = _randn((m, k), 1) * 2.0 ** e  # (rounded where subnormal: these are the inputs)
    A[:50] *= 0.125
    A[3, :] = 0.0
    B = _randn((k, n), 2) * 2.0 ** 900
    C = torch.empty((1, m, n), dtype=torch.float64, device="cuda")
    hs.hs_dgemm_emulated(A.cuda()[None], B.cuda()[None], C)
    up, down = A * 2.0 ** 900, B * 2.0 ** -900
    ref = up @ down
    bound = 5 * k * 2.0 ** -55 * up.abs().amax(1)[:, None] * down.abs().amax(0)[None, :] \
        + 2 * k * U * (up.abs() @ down.abs())
    assert bool(((C[0].cpu() - ref).abs() <= bound).all())


@pytest.mark.parametrize("tA,tB", [(False, False), (True, True)])
@pytest.mark.parametrize("e", [-1018, -1023, -1040])
def test_tiny_entries_of_the_complex_product(hs, e, tA, tB):
    """The same through the library's FP64 dispatch, at a size that it sends to the tensor cores."""
    m, n, k = 512, 300, 260
    A = torch.complex(_randn((m, k), 5) * 2.0 ** e, _randn((m, k), 6) * 2.0 ** e)
    B = torch.complex(_randn((k, n), 7) * 2.0 ** 900, _randn((k, n), 8) * 2.0 ** 900)
    C = torch.empty((m, n), dtype=torch.complex128, device="cuda")
    hs.hs_zgemm((A.T if tA else A).contiguous().cuda(), (B.T if tB else B).contiguous().cuda(), C, tA, tB, False)
    up = torch.complex(A.real * 2.0 ** 900, A.imag * 2.0 ** 900)
    down = torch.complex(B.real * 2.0 ** -900, B.imag * 2.0 ** -900)
    bound = 2 * (5 * 2 * k * 2.0 ** -55 * up.abs().amax(1)[:, None] * down.abs().amax(0)[None, :]
                 + 2 * k * U * (up.abs() @ down.abs()))
    assert bool(((C.cpu() - up @ down).abs() <= bound).all())
