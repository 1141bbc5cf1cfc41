"""The largest population change leaves out a cell whose molecule density is
infinite (its quotients are 0 or NaN): the other cells' change comes back."""
import numpy as np
import pytest

from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_lev", [2, 5, 8])
def test_infinite_density_is_left_out(n_lev):
    krl = need_gpu()
    import torch
    import workloads as W
    p, n_mol, spec = W.cloud(n=4, seed=7, packets_per_line=1000)
    J = np.arange(n_lev, dtype=np.float64)
    A, k = np.zeros((n_lev, n_lev)), np.zeros((n_lev, n_lev))
    for u in range(1, n_lev):
        A[u, u - 1] = 1e-7 * u ** 3
        k[u, :u] = 1e-11
    gamma = torch.rand((n_lev - 1, p.ncell), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1)) * 1e-7
    g = krl.Grid(p)
    try:
        change = []
        for bad in (0.0, np.inf):
            nm = torch.from_numpy(n_mol.reshape(-1).copy()).cuda()
            nm[17] = bad
            pops = torch.zeros((p.ncell, n_lev), dtype=torch.float64, device="cuda")
            change.append(g.levels_solve(krl.levels_desc(2.77 * J * (J + 1), 2 * J + 1, A, k, 28.0, nm), gamma, pops))
    finally:
        g.close()
    assert 0.0 < change[0] <= 1.0 and change[1] == change[0]
