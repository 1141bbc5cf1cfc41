"""Memory of the library's pools: the trim call gives the scratch of past calls
back, also while it is being freed behind work in flight, and a run with an
emissivity tally, whose segment buffer comes from the scratch pool, replays
from a CUDA graph."""
import dataclasses

import numpy as np
import pytest

import workloads as W
from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def test_trim_gives_scratch_back():
    krl = need_gpu()
    import torch
    p = dataclasses.replace(W.envelope(n=64, n_ch=128), tallies=(), cameras=())
    scratch = p.ncell * 128 * 4
    em = torch.ones(p.ncell * 128, device="cuda")
    g = krl.Grid(p)
    try:
        maps = g.raytrace(-1, 64, 64, 64.0, emiss=em)       # (in flight when the memory is asked back)
        krl.krl_memory_trim()
        free0 = torch.cuda.mem_get_info()[0]
        g.raytrace(-1, 64, 64, 64.0, emiss=em)
        torch.cuda.synchronize()
        free1 = torch.cuda.mem_get_info()[0]
        krl.krl_memory_trim()
        free2 = torch.cuda.mem_get_info()[0]
        assert free0 - free1 >= scratch and free2 - free1 >= scratch
        assert torch.equal(maps, g.raytrace(-1, 64, 64, 64.0, emiss=em))
    finally:
        g.close()


def test_emissivity_run_replays_from_a_graph():
    krl = need_gpu()
    import torch
    p = W.envelope(n=16, n_ch=16)
    g = krl.Grid(p)
    try:
        def run():
            g.run(n=3000, seed=4, want_stats=False, stream=s)
        s = torch.cuda.Stream()
        run()
        s.synchronize()
        want = {k: g.tally(k).cpu().numpy().astype(np.float64) for k in ("spec_n", "stats", "exc", "J", "emiss")}
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            run()
        for replays in (1, 3):
            g.reset()
            torch.cuda.synchronize()
            for _ in range(replays):
                graph.replay()
            torch.cuda.synchronize()
            for k, w in want.items():
                got = g.tally(k).cpu().numpy().astype(np.float64)
                if k in ("spec_n", "stats"):
                    assert np.array_equal(got, replays * w), k
                else:
                    # float32 partial sums in another order: 2^-24 times the root of the additions per bin
                    assert np.abs(got - replays * w).sum() <= 1e-5 * replays * w.sum(), k
    finally:
        g.close()
