"""FP64 and FP32 products and triangular solves at the edges of their kernels'
ranges: dot-product kernel (up to eight rows or columns, one to several
columns per warp, k below and above a warp's width), 16 x 16 and 32 x 32
tiles with remainders and k splits, the diagonal-block solves (one to
eight columns per block, sub-block remainders, both sweeps) and the panel
clusters (32 to 256 rows per CTA, 1 to 16 CTAs, the tournament above).

FP64 products: entry by entry against complex128 on the host within
2 k u |A||B|; FP32: against the float64 product within 4 k u32 |A||B| (each
real part is a sum of 2 k products).  Solves: backward error <= 8 n u."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs():
    from paper_1608_06871_gb300.build import build
    build()
    import paper_1608_06871_gb300 as mod
    return mod


def _rand(shape, g, cplx=True):
    re = torch.randn(shape, generator=g, dtype=torch.float64)
    return torch.complex(re, torch.randn(shape, generator=g, dtype=torch.float64)) if cplx else re


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (224, 1, 224), (1, 224, 33), (5, 300, 77), (300, 8, 31), (8, 8, 65),
                                   (9, 9, 15), (17, 16, 31), (33, 40, 700), (112, 113, 28), (250, 9, 1000)])
@pytest.mark.parametrize("tA,tB", [(False, False), (True, False), (False, True), (True, True)])
def test_zgemm_small(hs, m, n, k, tA, tB):
    g = torch.Generator().manual_seed(m * 31 + n * 7 + k)
    A, B, C0 = _rand((k, m) if tA else (m, k), g), _rand((n, k) if tB else (k, n), g), _rand((m, n), g)
    a, b = A.T if tA else A, B.T if tB else B
    C = C0.cuda().contiguous()
    hs.hs_zgemm(A.cuda().contiguous(), B.cuda().contiguous(), C, tA, tB, True)
    bound = 2 * k * 2.0 ** -53 * (a.abs() @ b.abs() + C0.abs())
    assert bool(((C.cpu() - (a @ b + C0)).abs() <= bound).all())


@pytest.mark.parametrize("m,n,k", [(700, 130, 260), (513, 300, 200), (200, 900, 1000)])
@pytest.mark.parametrize("tA,tB", [(False, False), (True, False), (False, True), (True, True)])
def test_zgemm_on_the_tensor_cores(hs, m, n, k, tA, tB):
    """Sizes the emulated product takes: one and several pieces of k, remainders, both transposes."""
    g = torch.Generator().manual_seed(m + n + k)
    A, B, C0 = _rand((k, m) if tA else (m, k), g), _rand((n, k) if tB else (k, n), g), _rand((m, n), g)
    A *= torch.logspace(-6, 6, A.shape[0], dtype=torch.float64)[:, None] if not tA else 1.0
    a, b = A.T if tA else A, B.T if tB else B
    C = C0.cuda().contiguous()
    hs.hs_zgemm(A.cuda().contiguous(), B.cuda().contiguous(), C, tA, tB, True)
    bound = 2 * k * 2.0 ** -53 * (a.abs() @ b.abs() + C0.abs())
    assert bool(((C.cpu() - (a @ b + C0)).abs() <= bound).all())


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_emulated_product_keeps_non_finite_rows(hs, bad):
    g = torch.Generator().manual_seed(3)
    A, B = _rand((1, 300, 500), g, False), _rand((1, 500, 70), g, False)
    A[0, 17, 3] = bad
    C = torch.empty((1, 300, 70), dtype=torch.float64, device="cuda")
    hs.hs_dgemm_emulated(A.cuda(), B.cuda(), C)
    finite = torch.isfinite(C.cpu()[0]).all(dim=1)
    assert not bool(finite[17]) and int(finite.sum()) == 299


@pytest.mark.parametrize("batch,m,n,k", [(1, 1, 1, 1), (3, 252, 5, 56), (2, 7, 200, 130), (1, 300, 8, 31),
                                         (2, 65, 9, 17), (1, 64, 64, 16), (3, 67, 130, 48), (1, 448, 81, 897),
                                         (40, 196, 140, 196), (300, 56, 48, 40), (300, 112, 96, 64)])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_gemm32_small(hs, batch, m, n, k, mode):
    g = torch.Generator().manual_seed(m + n * 7 + k)
    A, B = _rand((batch, m, k), g, mode == 2), _rand((batch, k, n), g, mode > 0)
    lo = {True: torch.complex64, False: torch.float32}
    A, B = A.to(lo[A.is_complex()]), B.to(lo[B.is_complex()])
    out = torch.empty((batch, m, n), dtype=B.dtype, device="cuda")
    hs.hs_set_tensor_cores(0)
    try:
        hs.hs_gemm32(A.cuda(), B.cuda(), out)
    finally:
        hs.hs_set_tensor_cores(1)
    wide = lambda t: t.to(torch.complex128)
    bound = 4 * k * 2.0 ** -24 * (A.abs().double() @ B.abs().double())
    assert bool(((wide(out.cpu()) - wide(A) @ wide(B)).abs() <= bound).all())


@pytest.mark.parametrize("dtype,u", [(torch.complex128, 2.0 ** -53), (torch.complex64, 2.0 ** -24)])
@pytest.mark.parametrize("batch,n,nrhs", [(1, 1, 1), (1, 15, 1), (2, 129, 1), (1, 224, 2), (1, 144, 700), (3, 130, 160),
                                          (1, 300, 1300), (9, 33, 2), (200, 31, 3), (20, 200, 2), (1, 513, 2),
                                         (2, 1025, 1), (1, 2050, 1), (1, 4300, 2)])
def test_block_solves(hs, dtype, u, batch, n, nrhs):
    g = torch.Generator().manual_seed(n * 7 + nrhs)
    A, B = _rand((batch, n, n), g).to(dtype), _rand((batch, n, nrhs), g).to(dtype)
    X = B.cuda().contiguous()
    hs.hs_lu_solve(A.cuda().contiguous(), X)
    A, X, B = (t.cpu().to(torch.complex128) for t in (A, X, B))
    r = (A @ X - B).abs().amax(dim=(1, 2))
    scale = A.abs().sum(dim=2).amax(dim=1) * X.abs().amax(dim=(1, 2)) + B.abs().amax(dim=(1, 2))
    assert bool((r <= 8 * n * u * scale).all())


@pytest.mark.parametrize("nL,M,P", [(1, 1, 3), (2, 3, 1), (4, 530, 7), (8, 2, 600)])
def test_fp64_solves_by_block_inverses(hs, nL, M, P):
    """Far fields and gradients of FP64 contexts whose root (and top merge) systems have one block, a
    remainder block, and more right-hand sides of either sweep than one chunk of columns, against the
    oracle with the bounds the other FP64 contexts are held to."""
    import numpy as np
    from oracle import forward as F
    k, c = 2.0 + nL / 4, np.array([[0.05, -0.02], [0.01, 0.03]])
    al, th = np.linspace(0.1, 6.0, M), np.linspace(0.2, 6.1, P)
    fw = F.forward_from_coeffs(c, k, nL)
    ref, _ = fw.solve_plane(al, th)
    S = hs.Solver(nL, 2, 2).build(c, k)
    uf = S.solve(al, th)
    assert np.linalg.norm(uf - ref) < 1e-10 * np.linalg.norm(ref)
    g, _ = S.gradient(ref * 1.1, al, th)
    go = F.misfit_gradient(fw.jacobian(al, th, 2, 2), ref.ravel(), ref.ravel() * 1.1)
    assert np.linalg.norm(g.ravel() - go) < 1e-9 * np.linalg.norm(go)
    S.close()


@pytest.mark.parametrize("nL,M,P,k", [(1, 2, 1, 0.7), (2, 1, 9, 3.0), (4, 3, 17, 6.0)])
def test_mixed_adjoint_residuals(hs, nL, M, P, k):
    """Jacobians of mixed contexts (adjoint residuals for one to seventeen receivers: part of a block's
    eight, and one more than one or two blocks; leaves with one to four boundary sides) against the
    oracle within the FP64 contexts' 1e-9."""
    import numpy as np
    from oracle import forward as F
    c = np.array([[0.05, -0.02], [0.01, 0.03]])
    al, th = np.linspace(0.1, 6.0, M), np.linspace(0.2, 6.1, P)
    S = hs.Solver(nL, 2, 2, precision=hs.HS_MIXED).build(c, k)
    J, Jo = S.jacobian(al, th), F.forward_from_coeffs(c, k, nL).jacobian(al, th, 2, 2)
    assert np.linalg.norm(J - Jo) < 1e-9 * np.linalg.norm(Jo)
    S.close()
