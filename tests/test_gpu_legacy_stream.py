"""Calls of a mixed context on CUDA's legacy default stream (handle 1, the one
that autograd.misfit passes for torch's default stream), which cannot be
captured: repeated calls run launch by launch and give the same bits."""
import pytest

import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs():
    from paper_1608_06871_gb300.build import build
    build()
    import paper_1608_06871_gb300 as mod
    return mod


def test_repeated_mixed_calls_on_the_legacy_stream(hs):
    c = synth.random_coeffs(4, 4, seed=12, scale=0.04)
    s = hs.Solver(4, 4, 4, precision=hs.HS_MIXED).build(c, 5.0)
    al, th = torch.tensor(synth.directions(5), device="cuda"), torch.tensor(synth.receivers(7), device="cuda")
    data, grad = torch.zeros((5, 7, 2), dtype=torch.float64, device="cuda"), []
    for _ in range(4):
        g, m = torch.zeros((4, 4), dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
        hs.hs_gradient_dev(s.ctx, data, al, th, g, m, stream=1)
        grad.append(torch.cat([g.ravel(), m]))
    torch.cuda.synchronize()
    assert bool(grad[0].abs().max() > 0) and all(torch.equal(x, grad[0]) for x in grad)
    s.close()
