"""The table build at the ends of its range: damping parameters on both sides
of the small-a expansion's limit (1e-6) and near one, and a set-up without
the R_IIA table after one with it (its scratch shares a buffer)."""
import dataclasses

import numpy as np
import pytest

import workloads as W
from oracle import tables as OT
from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a", [1e-7, 9.9e-7, 1e-6, 0.7, 1.0])
@pytest.mark.parametrize("with_r", [True, False])
def test_tables_at_the_ends_of_the_range(a, with_r):
    krl = need_gpu()
    p = W.thin_slab()
    p.line = dataclasses.replace(p.line, a_fixed=a)
    if not with_r:
        p.tallies = ("exc",)
    g = krl.Grid(p)
    try:
        lnH = g.tally("voigt").cpu().numpy()
        lnc = g.tally("us_lncdf").cpu().numpy().reshape(40, 251)
        rt = g.tally("rtab")
        rt = None if rt is None else rt.cpu().numpy().reshape(40, 200, 201)
    finally:
        g.close()
    assert (rt is not None) == with_r
    # float32 storage (half an ulp, 6e-8) of FP64 sums: the bounds of the
    # element-wise table test
    assert np.allclose(lnH, OT.voigt_table(a)[0], rtol=3e-7, atol=1e-7)
    assert np.allclose(lnc, OT.usampler_table(a)[1], rtol=1e-6, atol=1e-6)
    if with_r:
        ref = OT.rtable(a)
        assert np.allclose(rt, ref, rtol=1e-5, atol=1e-9 * ref.max())
