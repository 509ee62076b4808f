"""What the emulated FP64 product (csrc/ozaki.cu) promises of its results.

With entries of at most 27 bits no slice pair is left out, so the slices, their
products and the recombination are exact and a result of one piece of k is the
exact sum rounded once, also where it cancels down to the last bits.

Otherwise the error of an entry is bounded by the largest entries of its row
and column: 2^-56 of each from the fixed point and 3.6 2^-55 from the slice
pairs left out, together below 1.25 k u max|A_i.| max|B_.j| (u = 2^-53; the
larger part of a complex entry, and 2 k terms a part), besides the roundings of
the result and of the sum of the pieces, 2 k u |A||B| at most.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs():
    from paper_1608_06871_gb300.build import build
    build()
    import paper_1608_06871_gb300 as mod
    return mod


@pytest.mark.parametrize("k", [16, 100, 384])
@pytest.mark.parametrize("bits", [12, 27])
def test_short_entries_are_summed_exactly_and_rounded_once(hs, k, bits):
    rng = np.random.default_rng(k + bits)
    m, n = 130, 40
    A = rng.integers(-2 ** bits, 2 ** bits, size=(m, k))
    B = rng.integers(-2 ** bits, 2 ** bits, size=(k, n))
    A[:, -1], B[-1, :] = 2 ** bits - 1, 1  # (every row has an entry of full length)
    B[0, :] = 2 ** bits - 1
    # the last rows cancel: the second half of k repeats the first with the other sign, but for one entry
    h = k // 2
    A[100:, h:2 * h] = -A[100:, :h]
    B[h:2 * h, :] = B[:h, :]
    A[100:, 0] += 1
    exact = A.astype(object) @ B.astype(object)
    C = torch.empty((1, m, n), dtype=torch.float64, device="cuda")
    hs.hs_dgemm_emulated(torch.tensor(A, dtype=torch.float64, device="cuda")[None],
                         torch.tensor(B, dtype=torch.float64, device="cuda")[None], C)
    want = np.array([[float(x) for x in row] for row in exact])  # (int -> float rounds to nearest even)
    assert np.array_equal(C[0].cpu().numpy(), want)


U = 2.0 ** -53


@pytest.mark.parametrize("spread", [0, 5, 8, 14])
@pytest.mark.parametrize("k", [128, 500])
def test_rows_graded_along_k(hs, k, spread):
    """A's columns fall over 10^spread, B's rows rise: every product has terms of one size, and rows and
    columns whose largest entries meet none of their own size."""
    g = torch.Generator().manual_seed(k + spread)
    grade = torch.logspace(0, -spread, k, dtype=torch.float64)[torch.randperm(k, generator=g)]
    A = torch.randn((140, k), generator=g, dtype=torch.float64) * grade
    B = torch.randn((k, 50), generator=g, dtype=torch.float64) / grade[:, None]
    C = torch.empty((1, 140, 50), dtype=torch.float64, device="cuda")
    hs.hs_dgemm_emulated(A.cuda()[None], B.cuda()[None], C)
    bound = 1.25 * k * U * A.abs().amax(1)[:, None] * B.abs().amax(0)[None, :] + 4 * k * U * (A.abs() @ B.abs())
    assert bool(((C[0].cpu() - A @ B).abs() <= bound).all())


@pytest.mark.parametrize("emulated", [True, False])
@pytest.mark.parametrize("rows,cols", [(0, 0), (8, 0), (0, 8), (8, 8)])
def test_factors_of_graded_systems(hs, rows, cols, emulated):
    """L U against the permuted matrix for rows and columns over 10^rows and 10^cols: the FP64 bound
    8 n u |L||U| and, with emulation, that of the trailing updates with 128 columns of L at a time."""
    n = 640
    g = torch.Generator().manual_seed(rows * 3 + cols)
    rand = lambda: torch.randn((n, n), generator=g, dtype=torch.float64)
    d = lambda s: torch.logspace(0, -s, n, dtype=torch.float64)[torch.randperm(n, generator=g)]
    A = torch.complex(rand(), rand()) * d(rows)[:, None] * d(cols)[None, :]
    F, X = A.clone().cuda()[None].contiguous(), torch.ones((1, n, 300), dtype=torch.complex128, device="cuda")
    hs.hs_set_fp64_emulation(emulated)
    try:
        hs.hs_lu_solve(F, X)
    finally:
        hs.hs_set_fp64_emulation(True)
    F = F[0].cpu()
    L, R = F.tril(-1) + torch.eye(n, dtype=torch.complex128), F.triu()
    PA = L @ R
    flat = lambda t: torch.view_as_real(t / t.abs().amax(1, keepdim=True)).reshape(n, -1)
    order = torch.cdist(flat(PA), flat(A)).argmin(1)  # which row of A became row i
    assert len(set(order.tolist())) == n
    bound = 8 * n * U * (L.abs() @ R.abs())
    if emulated:
        for j in range(0, n, 128):
            part = lambda t: torch.maximum(t.real.abs(), t.imag.abs())
            l, r = part(L[:, j:j + 128]).amax(1), part(R[j:j + 128, :]).amax(0)
            bound += 2 ** 0.5 * 2 * 128 * 1.25 * U * l[:, None] * r[None, :]
    assert bool(((PA - A[order]).abs() <= bound).all())
