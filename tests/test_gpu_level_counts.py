"""The statistical-equilibrium solve at every level count: one kernel per
count, unrolled over it. Every pair radiative, ragged cell counts, cells
without molecules, and one grid larger than a full launch (each thread takes
several cells)."""
import numpy as np
import pytest

import workloads as W
from oracle import levels as LV
from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_lev,n", [(2, 5), (3, 68), (4, 7), (5, 9), (6, 6), (7, 5), (8, 7)])
def test_solve_matches_numpy_at_every_level_count(n_lev, n):
    krl = need_gpu()
    import torch
    p, n_mol, spec = W.cloud(n=n, seed=5)
    nm = n_mol.reshape(-1).copy()
    nm[3::11] = 0.0
    lev = LV.rotor(n_lev, spec.B_K, spec.A1, spec.k_ul, spec.mass_amu)
    rng = np.random.default_rng(n_lev)
    for u in range(1, n_lev):
        for lo in range(u):
            lev.A[u, lo] = 1e-7 * rng.lognormal(sigma=1.0)
    trans = lev.transitions()
    assert len(trans) == n_lev * (n_lev - 1) // 2
    gam = rng.lognormal(mean=-16.0, sigma=2.0, size=(len(trans), p.ncell))
    old = rng.random((p.ncell, n_lev)) * nm[:, None]
    g = krl.Grid(p)
    try:
        pops = torch.from_numpy(old).cuda()
        nm_t = torch.from_numpy(nm).cuda()
        ch = g.levels_solve(krl.levels_desc(lev.E_K, lev.g, lev.A, lev.k_coll, lev.mass_amu, nm_t),
                            torch.from_numpy(gam).cuda(), pops)
        got = pops.cpu().numpy()
    finally:
        g.close()
    pick = np.unique(np.r_[np.arange(min(p.ncell, 400)), np.arange(p.ncell - 100, p.ncell)])
    ref = LV.solve(lev, p.T_K, p.n_coll.reshape(-1)[pick], nm[pick], {tr: gam[i, pick] for i, tr in enumerate(trans)})
    assert np.all(np.abs(got[pick] - ref) <= 1e-4 * ref)          # the stated bar; cells without molecules: exactly 0
    assert np.allclose(got.sum(axis=1), nm, rtol=1e-12, atol=0)
    full = nm > 0
    assert abs(ch / (np.abs(got - old)[full] / nm[full, None]).max() - 1) < 1e-12
