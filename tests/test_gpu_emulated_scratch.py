"""FP64 products that are cut to a context's scratch: chunks of columns whose
remainder has fewer tiles than SMs (its pieces of k run as separate tiles and
want room that a full chunk does not), against the same products on the FP64
pipe.  Chunks of a context with 4 x 4 leaves (32 MB of scratch): the far field
of 436 incidences at 1184 receivers is one of 1216 and one of 1152 real
columns, that of 300 at 3392 two of 3392 columns and smaller ones."""
import numpy as np
import pytest

import synth
from parity import rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs():
    from paper_1608_06871_gb300.build import build
    build()
    import paper_1608_06871_gb300 as mod
    return mod


@pytest.mark.parametrize("M,P", [(436, 1184), (300, 3392), (436, 1183), (301, 3391)])
def test_remainder_chunks_are_computed(hs, M, P):
    c = synth.random_coeffs(3, 3, seed=5, scale=0.04)
    al, th = np.linspace(0.05, 6.2, M), np.linspace(0.01, 6.25, P)
    s = hs.Solver(4, 3, 3).build(c, 5.0)
    far = s.solve(al, th)
    hs.hs_set_fp64_emulation(False)
    try:
        ref = s.solve(al, th)
    finally:
        hs.hs_set_fp64_emulation(True)
    s.close()
    assert rel(far, ref) < 1e-10  # the far-field bar of the FP64 contexts
