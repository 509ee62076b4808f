"""hs_solve_noalloc beside the context's other calls: its scratch is the static
array alone, so calls on one stream and full forward solves of the same context
on another, enqueued without waiting, give the bits that each gives alone."""
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


@pytest.mark.parametrize("leaves,M,P,M2", [(4, 20, 24, 60), (4, 1, 3, 40), (8, 33, 40, 64)])
def test_noalloc_and_forward_on_two_streams(hs, leaves, M, P, M2):
    c = synth.random_coeffs(5, 5, seed=17, scale=0.05)
    S = hs.Solver(leaves, 5, 5).build(c, 5.0)
    dev = lambda x: torch.tensor(x, device="cuda")
    a, t, a2 = dev(synth.directions(M)), dev(synth.receivers(P)), dev(synth.directions(M2) + 0.3)
    far = lambda m: torch.zeros((m, P, 2), dtype=torch.float64, device="cuda")
    ref, ref2 = far(M), far(M2)
    u = torch.zeros((M2, leaves * leaves * 256, 2), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    hs.hs_solve_noalloc(S.ctx, a, t, ref)
    torch.cuda.synchronize()
    hs.hs_forward_dev(S.ctx, a2, t, ref2, u)
    torch.cuda.synchronize()
    ref_u = u.clone()
    n = 30
    outs, outs2 = [far(M) for _ in range(n)], [far(M2) for _ in range(n)]
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for i in range(n):
        hs.hs_solve_noalloc(S.ctx, a, t, outs[i], stream=s1.cuda_stream)
        hs.hs_forward_dev(S.ctx, a2, t, outs2[i], u, stream=s2.cuda_stream)
    torch.cuda.synchronize()
    assert all(torch.equal(o, ref) for o in outs)
    assert all(torch.equal(o, ref2) for o in outs2)
    assert torch.equal(u, ref_u)
    S.close()
