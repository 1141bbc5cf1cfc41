"""Packets with few events: the emission position in integers, the guided pick
of the emission cell, the escape bin in single precision, and the segment
buffer's chunks, each at the sizes where it can go wrong."""
import dataclasses

import numpy as np
import pytest

import oracle
import workloads as W
from _gpu_common import gpu_run, need_gpu

pytestmark = pytest.mark.gpu


def _thin(shape, source, periodic=(False, False, False)):
    p = W.box(tau0=1e-3, n=4)
    return dataclasses.replace(p, name="thin", shape=shape, opacity=np.full(shape, 1e-6, np.float32), source=source,
                               periodic=periodic, n_packets=20000, spectrum=(-4.0, 4.0, 64))


def _rates(shape, zero):
    r = np.random.default_rng(1).random(shape).astype(np.float32) ** 8
    if zero:
        r.reshape(-1)[::3] = 0.0
        r.reshape(-1)[-2:] = 0.0
    return r


SOURCES = {
    "one cell": _thin((1, 1, 1), W.Source("volume", rate=np.ones((1, 1, 1), np.float32))),
    "zero cells": _thin((7, 5, 3), W.Source("volume", rate=_rates((7, 5, 3), True))),
    "more cells than guide bins": _thin((41, 41, 41), W.Source("volume", rate=_rates((41, 41, 41), False))),
    "plane on a face": _thin((5, 3, 7), W.Source("plane", axis=0, plane=3.0)),
    "plane inside, periodic": _thin((5, 3, 7), W.Source("plane", axis=2, plane=4.75), (True, True, False)),
    "plane on the domain's face, periodic": _thin((4, 3, 6), W.Source("plane", axis=1, plane=0.0), (True, True, True)),
    "point outside": _thin((3, 4, 5), W.Source("point", pos=(5.5, 1.0, 1.0))),
    "point on a vertex": _thin((3, 4, 5), W.Source("point", pos=(2.0, 1.0, 2.0))),
    "beam": _thin((3, 4, 5), W.Source("beam", axis=1)),
    "beam in a band": _thin((6, 4, 5), W.Source("beam", axis=0, band_axis=2, band=(1.25, 4.5))),
}


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("name", sorted(SOURCES))
def test_emission_cells(name, prec):
    krl = need_gpu()
    p = SOURCES[name]
    if all(p.periodic):
        p = dataclasses.replace(p, opacity=np.full(p.shape, 1e3, np.float32))   # no open face: end by the budget
    ref = oracle.run(p, records=True, max_iters=40)["records"]
    out = gpu_run(krl, p, krl.KRL_PREC_FP32 if prec == "fp32" else krl.KRL_PREC_FP64, max_iters=40)["records"]
    assert np.array_equal(out["cell0"], ref["cell0"])


@pytest.mark.parametrize("bins", [(-20.0, 20.0, 1), (-3.0, 3.0, 7), (-0.37, 2.9, 400), (-20.0, 20.0, 200_000),
                                  (1e3, 1e4, 50), (-1e-3, 1e-3, 1000)])
def test_escape_bins(bins):
    """Every packet in the bin that the FP64 form gives its recorded x."""
    krl = need_gpu()
    p = dataclasses.replace(W.box(tau0=30.0, n=6, n_packets=50_000), spectrum=bins)
    out = gpu_run(krl, p, krl.KRL_PREC_FP32)
    lo, hi, n = bins
    x = out["records"]["x"].astype(np.float64)
    b = np.clip(1 + np.floor((x - lo) / (hi - lo) * n).astype(np.int64), 1, n)
    b = np.where(x < lo, 0, np.where(x >= hi, n + 1, b))
    assert np.array_equal(out["spec_n"], np.bincount(b, minlength=n + 2))
    assert np.array_equal(out["spec_w"], out["spec_n"].astype(np.float64))


# chunk sizes of the 2432 warps of a run on 152 SMs: none, 32, 128, 256
@pytest.mark.parametrize("records", [1, 33, 100_000, 2432 * 64, 2432 * 256 + 7, 2432 * 1024])
@pytest.mark.parametrize("n", [1, 700, 30_000])
def test_segment_chunks(records, n):
    krl = need_gpu()
    p = W.envelope(n=12, n_ch=9)
    a = gpu_run(krl, p, krl.KRL_PREC_FP32, n=n, emiss_records=-1)
    b = gpu_run(krl, p, krl.KRL_PREC_FP32, n=n, emiss_records=records)
    for f in a["records"].dtype.names:
        assert np.array_equal(a["records"][f], b["records"][f]), f
    x, y = a["emiss"].astype(np.float64), b["emiss"].astype(np.float64)
    assert x.sum() > 0 or n == 1
    assert np.abs(x - y).sum() <= 1e-5 * np.abs(x).sum()
