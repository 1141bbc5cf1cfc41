"""Explicit CTA sizes, in the form of the walk for 256 threads and fewer and in
the one for more, walk the same paths as the default."""
import numpy as np
import pytest

import workloads as W
from _gpu_common import gpu_run, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [32, 128, 256, 288, 512])
def test_explicit_blocks_same_records(block):
    krl = need_gpu()
    p = W.sphere(vmax_kms=60.0, tau0=1e3, n=16, a=4.7e-3)
    a = gpu_run(krl, p, krl.KRL_PREC_FP32, n=20_000, seed=9, block=block)["records"]
    b = gpu_run(krl, p, krl.KRL_PREC_FP32, n=20_000, seed=9)["records"]
    assert np.array_equal(a.view(np.uint8), b.view(np.uint8))
