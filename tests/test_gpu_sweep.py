"""Few right-hand sides through the streamed sweeps: every column count they
take (1 .. 4, with the padded 3) and some that they leave to the tensor-core
products (5 .. 9), at orders whose LU has one ragged unit (p = 5, 8),
a ragged last step (p = 9: 343 = 2 x 128 + 87) and several units (p = 12, 13).
Reference: the FP64 path's solves of the same boxes; both forms refine to
1e-11 of the solution, so they agree to 1e-10."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [5, 8, 9, 12, 13])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 5, 7, 8, 9])
def test_few_columns_match_fp64(p, nrhs):
    import torch
    import paper_2503_04033_gb300 as H
    rng = np.random.default_rng(10 * p + nrhs)
    nbox = 3
    n, m = H.hps_leaf_sizes(p)
    b = torch.from_numpy(rng.uniform(0.5, 1.5, (nbox, p ** 3))).cuda()
    f = torch.from_numpy(rng.standard_normal((nbox, nrhs, p ** 3))).cuda()
    ub = torch.from_numpy(rng.standard_normal((nbox, nrhs, m))).cuda()
    kind = H.LeafKind(p, 0.25, 5.0)
    ctx = H.hps_create(0, 0)
    got = {}
    try:
        for prec in (H.HPS_FP64, H.HPS_FP32_IR, H.HPS_BF16_IR):
            v = torch.full((nbox, nrhs, n), np.nan, dtype=torch.float64, device="cuda")
            hf = torch.full((nbox, nrhs, m), np.nan, dtype=torch.float64, device="cuda")
            ui = torch.full((nbox, nrhs, n), np.nan, dtype=torch.float64, device="cuda")
            st = torch.full((nbox,), -1, dtype=torch.int32, device="cuda")
            F = H.hps_leaf_factor(ctx, kind, nbox, b, nrhs, prec)
            H.hps_leaf_solve_factored(F, nrhs, f, v, hf, st)
            H.hps_leaf_reconstruct_factored(F, nrhs, v, ub, ui, st)
            torch.cuda.synchronize()
            H.hps_leaf_factors_destroy(F)
            assert (st.cpu().numpy() == 0).all()
            got[prec] = [t.cpu().numpy() for t in (v, hf, ui)]
    finally:
        H.hps_destroy(ctx)
    for prec in (H.HPS_FP32_IR, H.HPS_BF16_IR):
        for x, y in zip(got[prec], got[H.HPS_FP64]):
            assert np.linalg.norm(x - y) <= 1e-10 * np.linalg.norm(y)
