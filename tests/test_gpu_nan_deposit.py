"""A channel grid whose origin is NaN gives NaN, not zeros, in the emissivity,
whether the walk deposits it or the second stage does."""
import dataclasses
import math

import pytest

import workloads as W
from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("records", [0, -1])
def test_deposit(records):
    krl = need_gpu()
    import torch
    p = W.envelope(n=9, n_ch=8)
    p = dataclasses.replace(p, channels=(math.nan, *p.channels[1:]))
    g = krl.Grid(p)
    try:
        g.run(n=500, seed=1, emiss_records=records)
        torch.cuda.synchronize()
        assert torch.isnan(g.tally("emiss")).any()
    finally:
        g.close()
