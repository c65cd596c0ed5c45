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
