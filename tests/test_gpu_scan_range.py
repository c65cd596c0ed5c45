"""The geometry scan at constants far outside the floats, against limits in closed
form: an Einasto scale below the scan's smallest radius is Kerr, a cored-NFW
core beyond every radius is H = e^-eta - 2/R, a core below every radius with no
mass is Kerr.

Bar as test_gpu_scan.py: 1e-12 relative, R_e 1e-7; flags exact.
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


def _scan(B, sts):
    return {k: v.cpu().numpy() for k, v in B.geometry_scan(sts, (0.0, 0.5 * math.pi)).items()}


def test_einasto_kerr_limit(B):
    # from 1e-7 on, e^-x is 0 at every radius of the scan above 9.7e-5
    lams = [10.0 ** -k for k in (7, 9, 12, 18, 19, 20, 21, 22, 23, 24, 40, 152, 153, 154, 156, 158,
                                 200, 300)]
    for chi in (0.0, 0.3, 0.9, 1.1):
        r = _scan(B, [B.Spacetime(metric=B.EINASTO, chi=chi, lambda_E=x) for x in lams])
        assert np.all(r["flags"] == (1 if chi > 1.0 else 0))
        assert np.allclose(r["chi_e"], 1.0, rtol=1e-12) and np.allclose(r["R_e"], 1.0, rtol=1e-7)
        if chi < 1.0:
            want = 1.0 + math.sqrt(1.0 - chi * chi)
            assert np.allclose(r["r_plus"], want, rtol=1e-12)
            assert np.allclose(r["R_s"], [want, 2.0], rtol=1e-12)


def test_cored_nfw_limits(B):
    # R << lambda_c: S = -eta, so R^2 H = e^-eta R^2 - 2 R
    for eta in (0.0, 1e-6, 0.02, 1.5):
        lcs = (1e18, 1e29, 1e31, 1e37, 1e38, 1e39, 1e45, 1e100, 1e200)
        r = _scan(B, [B.Spacetime(metric=B.CNFW, chi=0.5, eta=eta, lambda_c=x) for x in lcs])
        assert np.all(r["flags"] == 0)
        assert np.allclose(r["R_e"], math.exp(eta), rtol=1e-7)
        assert np.allclose(r["chi_e"], math.exp(0.5 * eta), rtol=1e-12)
        want = math.exp(eta) * (1.0 + math.sqrt(1.0 - 0.25 * math.exp(-eta)))
        assert np.allclose(r["r_plus"], want, rtol=1e-12)
    # lambda_c << R: S -> 0 with the halo's mass eta lambda_c log(R / lambda_c)
    lcs = (1e-25, 1e-30, 1e-31, 1e-38, 1e-40, 1e-200, 1e-300)
    r = _scan(B, [B.Spacetime(metric=B.CNFW, chi=0.5, eta=0.02, lambda_c=x) for x in lcs])
    assert np.all(r["flags"] == 0) and np.allclose(r["chi_e"], 1.0, rtol=1e-12)
    # the halo outweighs everything: H < 0 up to the top of the scan
    r = _scan(B, [B.Spacetime(metric=B.CNFW, chi=0.7, eta=3e77, lambda_c=1e-38)])
    assert r["flags"][0] == 1 and r["R_e"][0] > 50.0
