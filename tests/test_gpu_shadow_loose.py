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
