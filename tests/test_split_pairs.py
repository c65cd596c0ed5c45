"""The paired operations of a split step (csrc/step_split.cuh): products with the
tableau's coefficients, the stage sums and the three-float state, compiled for
the host and compared with long double.

Bounds, with v = 2^-48: a product within 8 v of itself; a sum of seven products
within 128 v of the sum of their magnitudes (the low parts, up to 7 * 2^-23 of
it, are rounded twice a term); the state within 2^-54 a step, as the scalar sum
of test_split_arith.py (the same increments).
"""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
V = 2.0 ** -48
BOUND = dict(v_prod=8 * V, v_acc=128 * V, v_add3=2.0 ** -54)


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    from paper_2605_05635_gb300 import _build
    out = str(tmp_path_factory.mktemp("split_pairs") / "probe")
    cmd = [_build._nvcc(), *_build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr",
           "-Xcompiler", "-ffp-contract=off", "-I", _build.CSRC, "-I",
           os.path.join(ROOT, "include"), os.path.join(HERE, "split_pairs_probe.cu"), "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    run = subprocess.run([out], capture_output=True, text=True, check=True)
    return {w.split()[0]: float(w.split()[1]) for w in run.stdout.splitlines()}


@pytest.mark.parametrize("name", sorted(BOUND))
def test_within_bound(errors, name):
    assert errors[name] <= BOUND[name]
