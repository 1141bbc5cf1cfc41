"""Scatterings beyond |x| = 300, where u_par is a plain Gaussian and not the
sampler's, take the same path in a group of lanes as in a lane of its own:
a beam enters, through a transparent moving layer, gas at rest whose opacity
at the shifted frequency is tens per cell, so that runs of such scatterings
end at faces, by absorption and by destruction. Records are compared bit for
bit, as in test_gpu_tail."""
import dataclasses

import numpy as np
import pytest

import workloads as W
from _gpu_common import gpu_run, need_gpu

pytestmark = pytest.mark.gpu

A_DAMP = 0.149


def _far(x, tau_cell, nz=9, moving=False):
    """Layers of optical depth tau_cell at frequency x behind one transparent
    layer that moves at x Doppler widths along the beam."""
    p = W.slab(tau0=1.0, a=A_DAMP, nz=nz)
    b = np.sqrt(2.0 * 1.380649e-16 * p.T_K / (p.line.mass_amu * 1.66053906660e-24))
    p.source = W.Source(kind="beam", axis=2)
    # H(a, x) = a / (sqrt(pi) x^2) in the wing
    p.opacity = np.full(p.shape, tau_cell * np.sqrt(np.pi) * x * x / A_DAMP, dtype=np.float32)
    p.opacity[0] = 0.0
    p.vel_cms = np.zeros((3, *p.shape), dtype=np.float32)
    if moving:
        p.vel_cms[:] = np.linspace(-3e5, 3e5, nz, dtype=np.float32)[:, None, None]
    p.vel_cms[2, 0] = x * b
    p.spectrum = (-600.0, 600.0, 120)
    return p


def _destroyed(x):
    p = _far(x, 25.0)
    p.line = dataclasses.replace(p.line, k_ul=1e-9)
    # epsilon = k n / (A + k n) = 5e-3
    p.n_coll = np.full(p.shape, 5e-3 * p.line.A_ul / 1e-9, dtype=np.float32)
    return p


def _absorbed(x):
    p = _far(x, 25.0)
    p.tau_abs = np.full(p.shape, 5.0, dtype=np.float32)     # to the weight cut in tens of scatterings
    return p


CASES = {
    "beyond": lambda: _far(400.0, 20.0),
    "about the edge": lambda: _far(302.0, 30.0),
    "moving": lambda: _far(340.0, 20.0, nz=12, moving=True),
    "destroyed": lambda: _destroyed(350.0),
    "absorbed": lambda: _absorbed(320.0),
}


@pytest.mark.parametrize("few", [1, 304 * 9 + 5])
@pytest.mark.parametrize("name", sorted(CASES))
def test_far_group_walk_equals_lane_walk(name, few):
    krl = need_gpu()
    p = CASES[name]()
    a = gpu_run(krl, p, krl.KRL_PREC_FP32, n=few, seed=23, max_iters=20000)
    b = gpu_run(krl, p, krl.KRL_PREC_FP32, n=300_000, seed=23, max_iters=20000)
    ra, rb = a["records"], b["records"][:few]
    if few > 1:                     # the runs in question are there
        assert np.mean((np.abs(ra["x"]) > 250.0) & (ra["nscat"] > 2 * ra["ncross"])) > 0.02
    for f in ("status", "nscat", "ncross", "cell0"):
        assert np.array_equal(ra[f], rb[f]), f
    assert np.array_equal(ra["x"].view(np.uint32), rb["x"].view(np.uint32))
