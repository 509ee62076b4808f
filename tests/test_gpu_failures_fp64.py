"""Failures on FP64 contexts, made on the host as in test_gpu_failures.py: a
tensor-core wait that gave up (the flag that it would set, set from the host)
is reported by every call that synchronises, and once; scratch that only
speeds the FP64 products up and cannot be had is not an error, and results do
not depend on whether an earlier call allocated it."""
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


def _problem():
    return synth.random_coeffs(4, 4, seed=12, scale=0.04), synth.directions(24), synth.receivers(32)


def _calls(hs, data):
    return {"solve": lambda s, al, th: s.solve(al, th),
            "jacobian": lambda s, al, th: s.jacobian(al, th),
            "gradient": lambda s, al, th: s.gradient(data, al, th)[0]}


@pytest.mark.parametrize("M", [1, 24])
@pytest.mark.parametrize("name", ["solve", "jacobian", "gradient"])
def test_timeout_is_reported_by_fp64_calls(hs, name, M):
    c, al, th = _problem()
    al = al[:M]
    s = hs.Solver(4, 4, 4).build(c, 5.0)
    call = _calls(hs, 1.1 * s.solve(al, th))[name]
    before = call(s, al, th)
    hs.hs_raise_tc_timeout(0)
    with pytest.raises(hs.HSError) as e:
        call(s, al, th)
    assert e.value.code == hs.HS_ETIMEOUT
    assert rel(call(s, al, th), before) == 0.0  # reported once; the same numbers again
    s.close()


def test_timeout_of_a_device_call_is_reported_by_the_next_that_synchronises(hs):
    import torch
    c, al, th = _problem()
    s, other = hs.Solver(4, 4, 4).build(c, 5.0), hs.Solver(2, 4, 4)
    far = torch.empty((len(al), len(th), 2), dtype=torch.float64, device="cuda")
    a, t = torch.tensor(al, device="cuda"), torch.tensor(th, device="cuda")
    hs.hs_raise_tc_timeout(0)
    hs.hs_solve_dev(s.ctx, a, t, far)
    torch.cuda.synchronize()
    with pytest.raises(hs.HSError) as e:
        s.solve(al, th)
    assert e.value.code == hs.HS_ETIMEOUT
    other.build(c, 3.0)  # nothing is left over for another context
    s.close()
    other.close()


def test_build_and_gradient_without_the_product_scratch(hs):
    c, al, th = _problem()
    ref = hs.Solver(4, 4, 4).build(c, 5.0)
    far = ref.solve(al, th)
    grad = ref.gradient(1.1 * far, al, th)[0]
    s, m = hs.Solver(4, 4, 4), hs.Solver(4, 4, 4, precision=hs.HS_MIXED).build(c, 5.0)
    try:
        hs.hs_fail_next_allocs(1)  # the first allocation of each is the scratch
        s.build(c, 5.0)
        hs.hs_fail_next_allocs(1)
        gm = m.gradient(1.1 * far, al, th)[0]
    finally:
        hs.hs_fail_next_allocs(0)
    assert rel(s.solve(al, th), far) < 1e-10
    assert rel(s.gradient(1.1 * far, al, th)[0], grad) < 1e-9
    assert rel(gm, grad) < 1e-8
    for x in (ref, s, m):
        x.close()


@pytest.mark.parametrize("precision", ["HS_FP64", "HS_MIXED"])
def test_results_do_not_depend_on_earlier_calls(hs, precision):
    # (32 x 32 leaves, 64 x 64 modes: q on the leaf grid is a product worth the tensor cores)
    c, al, th = synth.random_coeffs(64, 64, seed=12, scale=0.004), synth.directions(24), synth.receivers(32)
    s = hs.Solver(32, 64, 64, precision=getattr(hs, precision)).build(c, 16.0)
    first = s.solve(al, th)
    s.gradient(1.1 * first, al, th)
    s.gn_step(1.1 * first, al, th, 1e-3, c)
    s.build(c, 16.0)
    assert np.array_equal(s.solve(al, th), first)
    s.close()
