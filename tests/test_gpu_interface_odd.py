"""FP32 interface factors of separators whose size is no multiple of 4: the
columns of the last LU block end inside a 16-byte unit that right-hand sides
share."""
from __future__ import annotations

import numpy as np
import pytest

import oracle.global_solve as gs
import paper_2503_04033_gb300 as H

pytestmark = pytest.mark.gpu


def _maps(rng, nbox, m):
    """Symmetric positive definite box maps of condition about 4 (any maps do: the solve is algebra on them)."""
    import torch
    a = rng.standard_normal((nbox, m, m)) / np.sqrt(m)
    return torch.from_numpy(np.eye(m) + 0.15 * (a + a.transpose(0, 2, 1))).cuda()


@pytest.mark.parametrize("p,nb", [(9, (3, 3, 5)), (11, (5, 3, 2)), (13, (3, 3, 2)), (9, (5, 5, 2))])
def test_odd_separators_match_fp64_factors(p, nb):
    """The refined solve of both factor precisions is the same system's: they
    agree to rounding times its condition number, far below 1e-11."""
    import torch
    grid = gs.InterfaceGrid(p, nb)
    m = 6 * (p - 2) ** 2
    rng = np.random.default_rng(100 * p + nb[0])
    T = _maps(rng, grid.nbox, m)
    hv = torch.from_numpy(rng.standard_normal((grid.nbox, 2, m))).cuda()
    ctx = H.hps_create(0, 0)
    out = {}
    try:
        for iprec in (H.HPS_FP64, H.HPS_FP32_IR):
            F = H.hps_interface_factor(ctx, p, grid.nb, T, 2, iprec)
            try:
                assert H.hps_interface_info(F)[2] >= 256
                u = torch.empty(grid.nbox, 2, m, dtype=torch.float64, device="cuda")
                H.hps_interface_solve(F, 2, hv, None, u)
                torch.cuda.synchronize()
                out[iprec] = u.cpu().numpy(), H.hps_interface_last_refinement(F)
            finally:
                H.hps_interface_destroy(F)
    finally:
        H.hps_destroy(ctx)
    u64, u32 = out[H.HPS_FP64][0], out[H.HPS_FP32_IR][0]
    assert np.abs(u32 - u64).max() < 1e-11 * np.abs(u64).max()
    # factors right to FP32 (6e-8 times a modest growth) contract by more than 1e-4 a correction
    assert out[H.HPS_FP32_IR][1][0] <= 4
