"""Which images take split arithmetic (split_allowed in api.cu): constants beyond the
floats, a capture radius next to the horizon and an observer next to the axis
keep the FP64 kernel.

A batch runs all its images on one kernel, so an image beside one whose atol is
below the split line gives the FP64 kernel's planes: an image that has to stay
FP64 gives the same bits alone, one that may be split does not (the constraint
drift shows the arithmetic), but agrees to the bar of test_gpu_split.py.
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


def _item(B, metric=0, chi=0.9, incl=math.radians(50.0), r_obs=1000.0, lam=0.1, eta=0.02, lc=10.0,
          em={}, **it):
    st = B.Spacetime(metric=metric, chi=chi, lambda_E=lam, eta=eta, lambda_c=lc)
    cam = B.Camera(r_obs=r_obs, incl=incl, x_min=-9.0, x_max=9.0, y_min=-9.0, y_max=9.0, nx=20,
                   ny=18, refine_levels=1)
    it.setdefault("max_steps", 20000)
    return st, cam, B.Emission(**em), B.Integrator(**it)


def _both(B, **kw):
    import dataclasses
    item = _item(B, **kw)
    other = (B.Spacetime(), item[1], B.Emission(), dataclasses.replace(item[3], atol=0.999e-12))
    alone = B.trace_image(*item)
    beside = B.trace_batch([item, other])[0]
    return ({k: v.cpu().numpy() for k, v in o.items() if k != "refine_keys"} for o in (alone, beside))


FP64 = [dict(em=dict(R_out=1e300)), dict(em=dict(R_out=-1e300)), dict(em=dict(R_out=1e39)),
        dict(em=dict(sigma_in=1e-300)), dict(em=dict(sigma_out=1e-39)), dict(em=dict(R_s=1e-3)),
        dict(em=dict(p=1e3)), dict(em=dict(p=-1e3)), dict(em=dict(j0=1e39)), dict(em=dict(j0=1e-38)),
        dict(esc_factor=1e16), dict(esc_factor=1e20), dict(r_obs=1e13),
        dict(chi=0.998, cap_factor=1.0001), dict(chi=0.9999), dict(chi=0.5, cap_factor=1.000001),
        dict(metric=1, chi=0.997, cap_factor=1.001), dict(metric=2, chi=1.0, cap_factor=1.0001),
        dict(incl=1e-6), dict(incl=math.pi - 1e-6), dict(incl=1e-3),
        dict(metric=1, lam=1e-25), dict(metric=2, lc=1e35, eta=1e-3)]
SPLIT = [dict(), dict(metric=1), dict(metric=2), dict(chi=0.99), dict(chi=0.9, cap_factor=1.003),
         dict(em=dict(R_out=1e9)), dict(em=dict(sigma_in=1e-3, sigma_out=1e-3)),
         dict(em=dict(p=20.0, j0=1e-9)), dict(em=dict(R_s=1e300)), dict(em=dict(j0=0.0)),
         dict(esc_factor=1e6), dict(r_obs=1e6), dict(incl=0.01), dict(rtol=1e-6, atol=1e-8)]


def _name(kw):
    return "-".join(f"{k}={v}" for k, v in kw.items()) or "default"


@pytest.mark.parametrize("kw", FP64, ids=_name)
def test_fp64(B, kw):
    alone, beside = _both(B, **kw)
    for k, v in alone.items():
        assert np.array_equal(v, beside[k], equal_nan=True), k
    if "incl" not in kw:  # rays through the axis may need more than max_steps
        assert np.all(alone["status"] < 2)


@pytest.mark.parametrize("kw", SPLIT, ids=_name)
def test_split(B, kw):
    alone, beside = _both(B, **kw)
    assert not np.array_equal(alone["h_drift"], beside["h_drift"])
    for k in ("status", "ncross", "refine_level"):
        assert np.array_equal(alone[k], beside[k]), k
    for k in ("I", "I_n", "R_em", "T_em", "g"):
        top = max(np.abs(beside[k]).max(), 1e-300)
        assert np.abs(alone[k] - beside[k]).max() <= 1e-6 * top, k
    assert alone["h_drift"].max() <= 1.1 * beside["h_drift"].max()
    assert abs(alone["steps"].sum() / beside["steps"].sum() - 1.0) <= 0.01


def test_promoted_rays(B):
    """The mixed path's promoted pass by the same rule: a kernel more per level when
    it is split."""
    counts = []
    for em in ({}, dict(R_out=1e300)):
        item = _item(B, em=em, precision=B.MIXED, rtol=1e-8, atol=1e-8)
        p = B.Plan([item])
        p.launch()
        p.check()
        counts.append(p.stats()["kernel_launches"])
        assert np.all(np.isfinite(p.outputs[0]["I"].cpu().numpy()))
        p.close()
    assert counts[0] == counts[1] + 2
