"""The last packets of a launch, each walked by a group of lanes, take the
same path as in a lane of their own: a run of a few packets (which groups
walk from their first events on) against the same ids in a run that keeps
every lane busy with one packet. Records are compared bit for bit, in the
cases that end or divert a packet inside a group's chain: escape, moving
cells, periodic faces, destruction, continuum absorption to the weight cut,
the event budget, frequencies far from the sampler rows at hand."""
import dataclasses

import numpy as np
import pytest

import workloads as W
from _gpu_common import gpu_run, need_gpu

pytestmark = pytest.mark.gpu


def _destroying():
    p = W.box(tau0=2e3, n=8, tallies=("exc", "J"))
    p.line = dataclasses.replace(p.line, k_ul=1e-9)
    # epsilon = k n / (A + k n) = 5e-4
    p.n_coll = np.full(p.shape, 5e-4 * p.line.A_ul / 1e-9, dtype=np.float32)
    p.channels = (-4e5, 1e5, 8)
    return p


def _emitting():
    p = _destroying()
    p.cameras = ((0.3, 0.2), (1.2, 2.0))
    p.tallies = ("exc", "J", "emiss")
    p.vel_cms = np.stack([np.linspace(-2e4, 2e4, p.ncell, dtype=np.float32).reshape(p.shape)] * 3)
    return p


CASES = {
    "static": lambda: W.sphere(tau0=3e3, n=16, tallies=("scatmap",)),
    "moving": lambda: W.sphere(vmax_kms=60.0, tau0=3e4, n=17, a=4.7e-3),
    "wing": lambda: W.slab(tau0=2e3, a=0.149, nz=33),
    "destroyed": _destroying,
    "emissivity": _emitting,
    "absorbed": lambda: W.dusty_slab(60.0, tau0=3e3, nz=31),
    "thin dust": lambda: W.dusty_slab(0.05, tau0=3e3, nz=31),
}


@pytest.mark.parametrize("max_iters", [0, 777])
@pytest.mark.parametrize("few", [1, 304 * 9 + 5])
@pytest.mark.parametrize("name", sorted(CASES))
def test_group_walk_equals_lane_walk(name, few, max_iters):
    krl = need_gpu()
    p = CASES[name]()
    a = gpu_run(krl, p, krl.KRL_PREC_FP32, n=few, seed=11, max_iters=max_iters)
    b = gpu_run(krl, p, krl.KRL_PREC_FP32, n=300_000, seed=11, max_iters=max_iters)
    ra, rb = a["records"], b["records"][:few]
    for f in ("status", "nscat", "ncross", "cell0"):
        assert np.array_equal(ra[f], rb[f]), f
    assert np.array_equal(ra["x"].view(np.uint32), rb["x"].view(np.uint32))
    st = a["stats_tally"]
    assert st[0] == few == st[1] + st[2] + st[3] + st[6]
    assert st[4] == ra["nscat"].sum(dtype=np.uint64) and st[5] == ra["ncross"].sum(dtype=np.uint64)
    if a["scatmap"] is not None:
        assert a["scatmap"].sum() == st[4]


@pytest.mark.parametrize("name", ["destroyed", "emissivity", "thin dust"])
def test_group_walk_tallies(name):
    """Floating tallies of the same packets in one run and split over runs of
    a few packets each (other groups, other chains): equal up to the order of
    the additions, whose float32 partial sums round to 2^-24 each."""
    krl = need_gpu()
    import torch
    p = CASES[name]()
    n = 2000
    g = krl.Grid(p)
    try:
        out = []
        for step in (n, 137):
            g.reset()
            for first in range(0, n, step):
                g.run(n=min(step, n - first), first=first, seed=5, want_stats=False)
            torch.cuda.synchronize()
            out.append({k: g.tally(k) for k in ("spec_w", "exc", "J", "emiss", "absw")})
    finally:
        g.close()
    for k, a in out[0].items():
        if a is None:
            continue
        a, b = a.cpu().numpy().astype(np.float64), out[1][k].cpu().numpy().astype(np.float64)
        assert a.sum() > 0
        assert np.abs(a - b).sum() <= 1e-6 * np.abs(a).sum(), k
