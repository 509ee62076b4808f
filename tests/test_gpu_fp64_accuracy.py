"""Far fields of FP64 contexts against the dense solution of the same discrete
system (perf/cases.py): with the FP64 products on the tensor cores they are as
close to it as with all of them on the FP64 pipe, within a tenth (another order
of the sums moves the error by a few per cent)."""
import numpy as np
import pytest

pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs():
    from paper_1608_06871_gb300.build import build
    build()
    import paper_1608_06871_gb300 as mod
    return mod


@pytest.mark.parametrize("impedance", [False, True])
@pytest.mark.parametrize("k,leaves,seed", [(3.1, 4, 301), (3.1, 4, 307), (5.0, 4, 302)])
def test_emulated_products_do_not_cost_accuracy(hs, k, leaves, seed, impedance):
    from perf import cases
    case = dict(cases.listed()[0], k=k, leaves=leaves, S1=8, S2=8, M=5, P=24, leaf_impedance=impedance)
    ref = np.asarray(cases.exact(case, seed)).ravel()
    err = []
    for on in (True, False):
        hs.hs_set_fp64_emulation(on)
        try:
            far = np.asarray(cases.run(cases.prepare(case, seed))).ravel()
        finally:
            hs.hs_set_fp64_emulation(True)
        err.append(np.linalg.norm(far - ref) / np.linalg.norm(ref))
    assert err[0] <= 1.1 * err[1], err
