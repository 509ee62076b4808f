"""What the emulated FP64 product (csrc/ozaki.cu) promises of its results.

With entries of at most 27 bits no slice pair is left out, so the slices, their
products and the recombination are exact and a result of one piece of k is the
exact sum rounded once, also where it cancels down to the last bits.
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
