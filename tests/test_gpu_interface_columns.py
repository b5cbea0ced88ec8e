"""The interface sweeps at every number of loads: one to sixteen columns in
passes of one, two, four and eight, few and many rows a level, rows on and off
16 bytes, FP64 and FP32 factors."""
from __future__ import annotations

import numpy as np
import pytest

import oracle.global_solve as gs
import paper_2503_04033_gb300 as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,nb", [(5, (2, 1, 1)), (8, (2, 2, 2)), (9, (4, 3, 2)), (12, (4, 4, 2))])
@pytest.mark.parametrize("iprec", [H.HPS_FP64, H.HPS_FP32_IR])
def test_every_column_count_solves_the_interface_system(p, nb, iprec):
    """Maps I + 0.15 (a symmetric Gaussian of norm about 2 sqrt 2): the system is
    A = sum of their interface blocks, of condition below 5, so a backward-stable
    solve leaves ||A u + h|| below 1e-12 of ||h||."""
    import torch
    grid = gs.InterfaceGrid(p, nb)
    m = 6 * (p - 2) ** 2
    rng = np.random.default_rng(p)
    a = rng.standard_normal((grid.nbox, m, m)) / np.sqrt(m)
    T = np.eye(m) + 0.15 * (a + a.transpose(0, 2, 1))
    h = rng.standard_normal((grid.nbox, 16, m))
    maps = [grid.local_to_global(bx) for bx in range(grid.nbox)]
    ctx = H.hps_create(0, 0)
    F = H.hps_interface_factor(ctx, p, grid.nb, torch.from_numpy(T).cuda(), 16, iprec)
    try:
        for nrhs in list(range(1, 10)) + [12, 16]:
            hv = torch.from_numpy(np.ascontiguousarray(h[:, :nrhs])).cuda()
            ub = torch.full((grid.nbox, nrhs, m), np.nan, dtype=torch.float64, device="cuda")
            H.hps_interface_solve(F, nrhs, hv, None, ub)
            u = ub.cpu().numpy()
            res, size = np.zeros((grid.n_iface, nrhs)), np.zeros((grid.n_iface, nrhs))
            for bx, (isi, gid) in enumerate(maps):
                i = np.nonzero(isi)[0]
                res[gid[i]] += (T[bx][i][:, i] @ u[bx][:, i].T) + h[bx, :nrhs][:, i].T
                size[gid[i]] += h[bx, :nrhs][:, i].T
            assert (np.linalg.norm(res, axis=0) < 1e-12 * np.linalg.norm(size, axis=0)).all(), nrhs
    finally:
        H.hps_interface_destroy(F)
        H.hps_destroy(ctx)
