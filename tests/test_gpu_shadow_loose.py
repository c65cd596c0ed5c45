"""The shadow boundary at loose tolerances, where the fates of traced rays are not
monotone in the impact parameter near the critical one.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_05635_gb300 as B
    B.lib()
    return B


@pytest.mark.parametrize("lanes", [1, 2, 8])
@pytest.mark.parametrize("metric,chi,incl,rtol", [(1, 0.5, 17.0, 1e-2), (1, 0.5, 17.0, 3e-2),
                                                  (2, 0.95, 85.0, 1e-3), (0, 0.9, 60.0, 1e-2)])
def test_brackets_are_ordered(B, metric, chi, incl, rtol, lanes):
    """b_in <= b_out and no wider than b_tol in every direction without a flag."""
    psi = np.linspace(0.0, 2.0 * math.pi, 3000, endpoint=False)
    st = B.Spacetime(metric=metric, chi=chi, lambda_E=0.3)
    cam = B.Camera(incl=math.radians(incl))
    it = B.Integrator(rtol=rtol, atol=1e-2 * rtol, max_steps=20000)
    b_in, b_out, fl = (x.cpu().numpy() for x in
                       B.shadow_boundary(st, cam, it, psi, 1.0, 9.0, 1e-6, lanes=lanes))
    ok = (fl & 3) == 0
    assert np.all(b_in[ok] <= b_out[ok])
    assert np.all((b_out - b_in)[ok] <= 1e-6)


@pytest.mark.parametrize("metric,chi,incl", [(0, 0.9, 60.0), (1, 0.5, 17.0), (2, 0.95, 85.0)])
@pytest.mark.parametrize("lanes", [0, 1, 4])
def test_ends_have_their_fates(B, metric, chi, incl, lanes):
    """At rtol 1e-4 the bracket is that of the FP64 integrator: the rays at its ends,
    traced as FP64 points (each 28 times over: enough points for the kernel that
    gives a ray one thread, as the shadow's; the four-lane kernel of fewer points
    rounds in another order, which at this tolerance moves the transition by more
    than the bracket), are captured and not captured.  The two builds may still
    round apart, so a few ends next to a fold of the fates may fall on its other
    side: one in twenty."""
    psi = np.sort(np.random.default_rng(1).uniform(0, 2 * math.pi, 400))
    st = B.Spacetime(metric=metric, chi=chi, lambda_E=0.3)
    cam = B.Camera(incl=math.radians(incl))
    it = B.Integrator(rtol=1e-4, atol=1e-6)
    b_in, b_out, fl = (x.cpu().numpy() for x in
                       B.shadow_boundary(st, cam, it, psi, 1.0, 9.0, 1e-9, lanes=lanes))
    assert np.all(fl == 0)
    wrong = 0
    for b, captured in ((b_in, True), (b_out, False)):
        xy = np.tile(np.stack([b * np.cos(psi), b * np.sin(psi)], 1), (28, 1))
        status = np.asarray(B.trace_points(st, cam, B.Emission(), it, xy)["status"])[:400]
        wrong += int(np.sum((status == 1) != captured))
    assert wrong <= 40
