"""The room that the ray adjoint works in: the workspace that
bh_backward_workspace_size asks for is enough for every metric, more of it makes
fewer forward / reverse pairs, an image whose trajectories it cannot hold well
takes the kernel that replays from checkpoints, and rays next to the critical
curve, longer than the default room per ray, are held by both.

Gradients of the same replay in other portions differ by the order of their sum
alone (1e-10 of the largest component).  The two kernels round differently, and
tangents of rays next to the critical curve amplify that: 1e-4, the bar of the
adjoint tests.  A cored NFW of eta = 0 is Kerr, on the other kernel.
"""
import ctypes as C
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


def _item(B, metric, nx, levels, eta=0.02, chi=0.7, incl=50.0, ext=(-12.0, 12.0, -12.0, 12.0), **it):
    st = B.Spacetime(metric=metric, chi=chi, eta=eta)
    cam = B.Camera(incl=math.radians(incl), x_min=ext[0], x_max=ext[1], y_min=ext[2], y_max=ext[3],
                   nx=nx, ny=nx, refine_levels=levels)
    return st, cam, B.Emission(r_in_mode=1), B.Integrator(**it)


def _least(B, cam):
    n = C.c_size_t(0)
    assert B.lib().bh_backward_workspace_size(C.byref(cam._c()), C.byref(n)) == 0
    return n.value


def _weights(nx):
    import torch
    return torch.from_numpy(np.random.default_rng(9).normal(size=(nx, nx))).float().cuda()


def _gradient(B, item, w, nbytes):
    import torch
    st, cam, em, it = item
    ws = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    at = (ws.data_ptr() + 255) // 256 * 256
    g = np.zeros(10)
    code = B.lib().bh_trace_backward(
        C.byref(st._c()), C.byref(cam._c()), C.byref(em._c()), C.byref(it._c()),
        C.c_void_p(w.data_ptr()), C.c_void_p(0), C.c_void_p(0), C.c_void_p(g.ctypes.data),
        C.c_void_p(0), C.c_void_p(0), C.c_void_p(at), C.c_size_t(nbytes), C.c_void_p(0))
    return code, g


def _close(a, b, tol):
    assert np.all(np.isfinite(a)) and np.any(b != 0.0)
    assert np.max(np.abs(a - b)) <= tol * np.max(np.abs(b)), (a, b)


@pytest.mark.parametrize("metric,nx,levels", [(0, 48, 1), (1, 48, 1), (2, 48, 1), (0, 128, 1),
                                              (1, 128, 0), (2, 100, 0)])
def test_least_workspace(B, metric, nx, levels):
    """The size that is asked for, 64 checkpoints a thread and the forward image's
    (0.38 GB at 48^2 on 152 SMs), suffices; 128^2 then takes several pairs."""
    import torch
    item, w = _item(B, metric, nx, levels), _weights(nx)
    least = _least(B, item[1])
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert least <= (3.0e6 * sms if nx == 48 else 4.0e6 * sms)
    code, g = _gradient(B, item, w, least)
    assert code == 0
    full, _, _ = B.trace_backward(*item, dL_dI=w)
    _close(g, full, 1e-10)
    assert _gradient(B, item, w, least - 256)[0] == 4


def test_pool_too_small(B):
    """256^2 Kerr: with the least workspace the pool holds too few of the longest rays,
    and the checkpoint kernel takes the image."""
    item, w = _item(B, 0, 256, 0), _weights(256)
    code, g = _gradient(B, item, w, _least(B, item[1]))
    assert code == 0
    full, _, _ = B.trace_backward(*item, dL_dI=w)
    _close(g, full, 1e-4)


@pytest.mark.parametrize("tol,steps", [(1e-10, 0), (1e-15, 4096)])
def test_critical_rays_on_both_kernels(B, tol, steps):
    """A screen straddling the critical curve.  At rtol 1e-10 the forward image's split
    rays and the FP64 replay part next to it; at 1e-15 the longest ray takes more
    than the 64 checkpoints of 64 steps that a thread has by default."""
    ext = (3.9, 4.9, -0.5, 0.5)
    kw = dict(chi=0.9, incl=80.0, ext=ext, rtol=tol, atol=1e-2 * tol)
    kerr, nfw = _item(B, 0, 32, 3, **kw), _item(B, 2, 32, 3, eta=0.0, **kw)
    p = B.Plan([kerr])
    p.launch()
    p.check()
    assert p.stats()["max_ray_steps"] > steps
    p.close()
    w = _weights(32)
    a, _, _ = B.trace_backward(*kerr, dL_dI=w)
    b, _, _ = B.trace_backward(*nfw, dL_dI=w)
    keep = [0, 1, 4, 5, 6, 7, 8, 9]  # the halo's entries have no counterpart
    _close(b[keep], a[keep], 1e-4)
