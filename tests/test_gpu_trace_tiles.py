"""The channel-map trace over the per-camera cube at the edges of its tiles,
channel blocks and row alignments, against the trace that evaluates the
profile per segment (no_scratch). Both sum the same segments with compensated
sums and differ in the exponentials' rounding only: a few 2^-22 per segment
factor, well inside the 1e-5 that either keeps to the FP64 trace."""
import dataclasses
import math

import numpy as np
import pytest

import workloads as W
from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def _grid(krl, n_ch, dust):
    p = W.envelope(n=9, n_ch=n_ch)
    p = dataclasses.replace(p, tallies=(), cameras=())
    p.opacity = p.opacity * np.float32(30.0)           # thick cells among thin ones
    if dust:
        p.tau_abs = np.full(p.shape, 0.02, np.float32)
    return krl.Grid(p), p


@pytest.mark.parametrize("n_ch", [1, 2, 5, 8, 9, 12, 16, 33, 64, 100, 128])
@pytest.mark.parametrize("pixels", [(1, 1), (7, 5), (33, 9), (700, 500)])
def test_tiles_and_channel_blocks(n_ch, pixels):
    krl = need_gpu()
    import torch
    g, p = _grid(krl, n_ch, dust=n_ch % 2 == 0)
    try:
        gen = torch.Generator(device="cuda").manual_seed(n_ch)
        size = p.ncell * n_ch
        store = torch.rand(size + 8, generator=gen, device="cuda")
        jline = torch.rand(p.ncell, generator=gen, device="cuda")
        for shift, jl, theta in ((0, None, 0.9), (1, jline, math.pi / 2), (4, None, 0.0), (0, jline, 2.0)):
            em = store[shift:shift + size]
            a = g.raytrace(-1, *pixels, 11.0, emiss=em, jline=jl, theta=theta, phi=0.4)
            b = g.raytrace(-1, *pixels, 11.0, emiss=em, jline=jl, theta=theta, phi=0.4, no_scratch=True)
            a, b = a.double(), b.double()
            assert float(b.max()) > 0
            assert float(((a - b).abs() / torch.maximum(b.abs(), 1e-3 * b.max())).max()) <= 1e-5
            assert torch.equal(a == 0, b == 0)
    finally:
        g.close()
