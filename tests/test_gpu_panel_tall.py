"""FP64 panels of more than 8192 rows (blocks of eight columns, eight rows a thread)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def test_tall_panels_solve_the_collocation_equations():
    """p = 23, n = 9261, variable b: S solves A_ii S = -A_ib.  The residual of a
    column of each face, taken matrix-free in FP64, is that of a backward-stable
    solve: below 1e-12 of ||A|| times the column's largest entry (n eps = 2e-12
    times a small constant is what pivoted elimination can leave, 1e-14 is usual)."""
    import torch
    import paper_2503_04033_gb300 as H
    p, h, kappa = 23, 0.5, 6.0
    q = p - 2
    n, m = H.hps_leaf_sizes(p)
    b = np.random.default_rng(2).uniform(0.5, 1.5, (1, p ** 3))
    T = torch.empty(1, m, m, dtype=torch.float64, device="cuda")
    S = torch.full((1, n, m), np.nan, dtype=torch.float64, device="cuda")
    st = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    ctx = H.hps_create(0, 0)
    try:
        H.hps_leaf_build_dtn(ctx, H.LeafKind(p, h, kappa), 1, torch.from_numpy(b).cuda(), T, S, H.HPS_FP64, st)
        assert int(st.item()) == 0
    finally:
        H.hps_destroy(ctx)
    D2 = (2.0 / h) ** 2 * (oracle.diff(p) @ oracle.diff(p))
    bg = b[0].reshape(p, p, p)                       # [k][j][i]
    size = 3 * np.abs(D2[1:-1]).sum(axis=1).max() + kappa ** 2 * bg.max()
    rng = np.random.default_rng(3)
    for f in range(6):
        a, c = rng.integers(0, q, 2)
        col = f * q * q + a + q * c
        u = np.zeros((p, p, p))
        s = S[0, :, col].cpu().numpy()
        assert np.isfinite(s).all()
        u[1:-1, 1:-1, 1:-1] = s.reshape(q, q, q)
        e = p - 1 if f & 1 else 0
        at = [(c + 1, a + 1, e), (c + 1, e, a + 1), (e, c + 1, a + 1)][f >> 1]
        u[at] = 1.0
        lap = np.einsum("il,kjl->kji", D2, u) + np.einsum("jl,kli->kji", D2, u) + np.einsum("kl,lji->kji", D2, u)
        res = (-lap - kappa ** 2 * bg * u)[1:-1, 1:-1, 1:-1]
        assert np.abs(res).max() < 1e-12 * size * max(1.0, np.abs(s).max()), (f, np.abs(res).max() / size)
