"""The channel-map trace with several lanes per ray (many channels on images of
few or widely spaced pixels), in each of its lane counts and with full and
partly filled lanes, against the trace that evaluates the profile per segment
(no_scratch). Both sum the same segments with compensated sums and differ in
the exponentials' rounding only: inside the 1e-5 that either keeps to the FP64
trace."""
import dataclasses

import numpy as np
import pytest

import workloads as W
from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ch,pixels,fov", [
    (13, (120, 121), 11.0), (16, (121, 120), 11.0),             # 4 lanes per ray, images of some size
    (17, (5, 3), 11.0), (32, (33, 9), 11.0),                    # 8
    (40, (1, 1), 11.0), (64, (30, 21), 11.0),                   # 16
    (65, (7, 5), 11.0), (128, (20, 20), 11.0),                  # 32
    (24, (260, 200), 260.0), (85, (200, 201), 150.0)])          # pixels far apart
@pytest.mark.parametrize("jl", [False, True])
def test_lanes_share_a_ray(n_ch, pixels, fov, jl):
    krl = need_gpu()
    import torch
    p = W.envelope(n=9, n_ch=n_ch)
    p = dataclasses.replace(p, tallies=(), cameras=())
    p.opacity = p.opacity * np.float32(30.0)           # thick cells among thin ones
    p.tau_abs = np.full(p.shape, 0.02, np.float32)
    g = krl.Grid(p)
    try:
        gen = torch.Generator(device="cuda").manual_seed(n_ch)
        size = p.ncell * n_ch
        store = torch.rand(size + 8, generator=gen, device="cuda")
        jline = torch.rand(p.ncell, generator=gen, device="cuda") if jl else None
        for shift, theta in ((0, 0.9), (1, 0.0)):
            em = store[shift:shift + size]
            a = g.raytrace(-1, *pixels, fov, emiss=em, jline=jline, theta=theta, phi=0.4).double()
            b = g.raytrace(-1, *pixels, fov, emiss=em, jline=jline, theta=theta, phi=0.4, no_scratch=True).double()
            assert float(b.max()) > 0
            assert float(((a - b).abs() / torch.maximum(b.abs(), 1e-3 * b.max())).max()) <= 1e-5
            assert torch.equal(a == 0, b == 0)
    finally:
        g.close()
