"""The channel-map trace of narrow images, whose warps follow tiles of other
shapes than 8 x 4, against the trace that evaluates the profile per segment
(no_scratch): the same segments, compensated sums, exponentials that differ in
their rounding only, well inside the 1e-5 that either keeps to the FP64 trace."""
import dataclasses

import numpy as np
import pytest

import workloads as W
from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ch,pixels", [
    (1, (1, 300)), (5, (300, 1)), (8, (2, 77)), (5, (77, 2)), (2, (3, 50)), (5, (4, 33)), (8, (9, 41)), (5, (41, 3)),
    (64, (1, 40000)), (64, (40000, 1)), (12, (70000, 2)), (20, (3, 40001))])
def test_narrow_images(n_ch, pixels):
    krl = need_gpu()
    import torch
    p = W.envelope(n=9, n_ch=n_ch)
    p = dataclasses.replace(p, tallies=(), cameras=())
    p.opacity = p.opacity * np.float32(30.0)           # thick cells among thin ones
    g = krl.Grid(p)
    try:
        gen = torch.Generator(device="cuda").manual_seed(n_ch)
        em = torch.rand(p.ncell * n_ch, generator=gen, device="cuda")
        fov = 11.0 * pixels[0] / max(pixels)           # the long side spans the box
        a = g.raytrace(-1, *pixels, fov, emiss=em, theta=0.9, phi=0.4).double()
        b = g.raytrace(-1, *pixels, fov, emiss=em, theta=0.9, phi=0.4, no_scratch=True).double()
        assert float(b.max()) > 0
        assert float(((a - b).abs() / torch.maximum(b.abs(), 1e-3 * b.max())).max()) <= 1e-5
        assert torch.equal(a == 0, b == 0)
    finally:
        g.close()
