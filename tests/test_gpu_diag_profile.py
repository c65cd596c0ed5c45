"""The radial profile of the diagnostics: every number of bins that fits pass 2's
shared memory, images whose range is far beyond a float's 24 bits, and screens
far smaller or larger than the unit.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# In a process of its own: the opt-in to more shared memory is kept per process.
SIZES = """
import sys
import numpy as np, torch
import paper_2605_05635_gb300 as B
from oracle.diagnostics import NAMES, diagnostics
rng = np.random.default_rng(5)
for nx in (2195, 2196, 3000, 4094, 4095, 10238, 10239, 17000):
    I = (rng.random((3, nx)) + 0.1).astype(np.float32)
    cam = B.Camera(nx=nx, ny=3, x_min=0.0, x_max=float(nx), y_min=-0.5, y_max=0.5)
    got = B.diagnostics(torch.from_numpy(I).cuda(), cam).cpu().numpy()
    ref = diagnostics(I, 0.0, float(nx), -0.5, 0.5)
    for k, name in enumerate(NAMES):
        if name != "theta_peak":
            assert abs(got[k] - ref[name]) <= 1e-11 * max(1.0, abs(ref[name])), (nx, name)
"""


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_05635_gb300 as B
    B.lib()
    return B


def test_bin_counts(B):
    """nx + 2 bins of 12 bytes: around the 24 KB from which pass 2 opts in to more
    shared memory, 48 KB and the largest that fits."""
    r = subprocess.run([sys.executable, "-c", SIZES], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]


def _diag(B, I, ext):
    import torch
    cam = B.Camera(nx=I.shape[1], ny=I.shape[0], x_min=ext[0], x_max=ext[1], y_min=ext[2],
                   y_max=ext[3])
    return B.diagnostics(torch.from_numpy(I).cuda(), cam).cpu().numpy()


@pytest.mark.parametrize("mask", [-1e12, -1e20, -3.4028235e38, -1.0, 1e30])
def test_masked_pixels(B, mask):
    """A ring with four corner pixels set to a mask value: a negative one leaves the
    peak on the ring, a large positive one is the peak."""
    y, x = np.mgrid[0:128, 0:128] - 63.5
    rho = np.hypot(x, y) * (24.0 / 128)
    I = (np.exp(-0.5 * ((rho - 5.2) / 0.15) ** 2) *
         (0.9 + 0.2 * np.random.default_rng(1).random(rho.shape))).astype(np.float32)
    I[:2, :2] = mask
    b = np.floor(rho / (24.0 / 128)).astype(int)
    mean = np.bincount(b.ravel(), I.astype(np.float64).ravel()) / np.maximum(np.bincount(b.ravel()), 1)
    want = (np.argmax(mean) + 0.5) * (24.0 / 128)
    got = _diag(B, I, (-12.0, 12.0, -12.0, 12.0))
    assert got[9] == pytest.approx(want, rel=1e-15)
    assert got[10] == pytest.approx(2.0 * want, rel=1e-15)


@pytest.mark.parametrize("small", [2.0 ** -10, 0.0, -2.0 ** -10])
def test_near_tie(B, small):
    """Four corner pixels, one of 2^40 and three of `small`, against a centre pixel of
    2^38: the means differ by 2^-48 of their value, exact in FP64, and an exact
    tie goes to the smaller radius."""
    I = np.zeros((65, 65), dtype=np.float32)
    I[0, 0], I[0, 64], I[64, 0], I[64, 64] = 2.0 ** 40, small, small, small
    I[32, 32] = 2.0 ** 38
    got = _diag(B, I, (-32.5, 32.5, -32.5, 32.5))
    assert got[9] == (np.floor(np.hypot(32, 32)) + 0.5 if small > 0 else 0.5)


@pytest.mark.parametrize("half", [1e-150, 1e-30, 1e-22, 0.99e-12, 1e-12, 1e12, 1.01e12, 1e20, 1e150])
def test_screen_scale(B, half):
    """The peak's bin does not depend on the unit of the screen."""
    I = np.random.default_rng(3).random((128, 128)).astype(np.float32)
    one = _diag(B, I, (-1.0, 1.0, -1.0, 1.0))
    got = _diag(B, I, (-half, half, -half, half))
    assert round(got[9] / (2.0 * half / 128) - 0.5) == round(one[9] / (2.0 / 128) - 0.5)
