"""A channel grid whose origin is NaN gives NaN, not numbers, in every pixel
that the box covers, in each layout of the ray trace."""
import dataclasses
import math

import pytest

import workloads as W
from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("no_scratch", [False, True])
@pytest.mark.parametrize("n_ch,pixels", [(5, 40), (8, 700), (32, 60), (64, 400)])
def test_trace(n_ch, pixels, no_scratch):
    krl = need_gpu()
    import torch
    p = dataclasses.replace(W.envelope(n=9, n_ch=n_ch), tallies=(), cameras=())
    em = torch.ones(p.ncell * n_ch, device="cuda")
    maps = []
    for v0 in (p.channels[0], math.nan):
        g = krl.Grid(dataclasses.replace(p, channels=(v0, *p.channels[1:])))
        try:
            maps.append(g.raytrace(-1, pixels, pixels, 13.0, emiss=em, theta=0.9, phi=0.4, no_scratch=no_scratch))
        finally:
            g.close()
    assert torch.isfinite(maps[0]).all() and float(maps[0].min()) == 0.0
    assert torch.equal(torch.isnan(maps[1]), maps[0] > 0)
