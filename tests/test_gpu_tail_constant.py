"""The tables in the constant bank leave a packet's path as it is, whether a
CTA's packets all go to groups of lanes at once (up to 32 per CTA) or its
last ones do, in fewer groups: records against the shared-memory walk, bit for
bit."""
import numpy as np
import pytest

import workloads as W
from _gpu_common import gpu_run, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [304 * 2 + 1, 304 * 32, 304 * 32 + 1, 304 * 75])
@pytest.mark.parametrize("vmax", [0.0, 60.0])
def test_constant_tables_same_records(n, vmax):
    krl = need_gpu()
    p = W.sphere(vmax_kms=vmax, tau0=1e3, n=16, a=4.7e-3)
    a = gpu_run(krl, p, krl.KRL_PREC_FP32, n=n, seed=9, table_space=krl.KRL_TABLES_CONSTANT)["records"]
    b = gpu_run(krl, p, krl.KRL_PREC_FP32, n=n, seed=9)["records"]
    assert np.array_equal(a.view(np.uint8), b.view(np.uint8))
