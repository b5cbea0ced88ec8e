"""The panel factorisation over its cluster sizes and edges.

The 2-D leaves give LU sizes n = q^2 = 1 .. 484 for q = 1 .. 22 (one column to
eight panels of 64, ragged last panels and blocks of columns), batches of 1, 40
and 700 boxes the cluster and row splits; the 3-D leaves reach n = 10648, where
a cluster holds the panel in blocks of 8 columns.  Reference: the oracle's
dense LU of the same collocation.  Bound: both solves are backward stable, so S is
within a few cond(A_ii) eps of the truth; kappa = 1 keeps A_ii positive definite
with cond below 3 q^4, and 1e-11 is 50 times that eps at q = 22.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", list(range(3, 25)))
@pytest.mark.parametrize("nbox", [1, 40, 700])
def test_leaf2d_every_order_and_batch(p, nbox):
    import torch
    import oracle
    import paper_2503_04033_gb300 as H
    rng = np.random.default_rng(p)
    n, m = H.hps_leaf2d_sizes(p)
    h = (0.5, 0.4)
    b = rng.uniform(0.5, 1.5, (nbox, p * p))
    T = torch.full((nbox, m, m), np.nan, dtype=torch.float64, device="cuda")
    S = torch.full((nbox, n, m), np.nan, dtype=torch.float64, device="cuda")
    st = torch.full((nbox,), -1, dtype=torch.int32, device="cuda")
    H.hps_leaf2d_solve(p, h, 1.0, nbox, torch.from_numpy(b).cuda(), 0, None, T, S, None, None, st)
    assert (st.cpu().numpy() == 0).all()
    for i in sorted({0, nbox // 2, nbox - 1}):
        To, So, info = oracle.leaf_dtn_2d(p, h, 1.0, b[i])
        assert info == 0
        assert np.linalg.norm(S[i].cpu().numpy() - So) <= 1e-11 * np.linalg.norm(So), i
        assert np.linalg.norm(T[i].cpu().numpy() - To) <= 1e-11 * np.linalg.norm(To), i


@pytest.mark.parametrize("prec", ["fp64", "fp32ir"])
def test_results_do_not_depend_on_the_batch(prec):
    """A box alone and the same box among 300 take different clusters, with the same arithmetic."""
    import torch
    import paper_2503_04033_gb300 as H
    pr = {"fp64": H.HPS_FP64, "fp32ir": H.HPS_FP32_IR}[prec]
    p = 10
    n, m = H.hps_leaf_sizes(p)
    b = torch.from_numpy(np.random.default_rng(1).uniform(0.5, 1.5, (300, p ** 3))).cuda()
    ctx = H.hps_create(0, 0)
    try:
        T = torch.empty(300, m, m, dtype=torch.float64, device="cuda")
        T1 = torch.empty(1, m, m, dtype=torch.float64, device="cuda")
        kind = H.LeafKind(p, 0.125, 20.0)
        H.hps_leaf_build_dtn(ctx, kind, 300, b, T, None, pr)
        H.hps_leaf_build_dtn(ctx, kind, 1, b[123:124].contiguous(), T1, None, pr)
        assert torch.equal(T[123], T1[0])
    finally:
        H.hps_destroy(ctx)


def test_largest_order_fp64():
    """n = 10648: panels taller than 8192 rows."""
    import torch
    import paper_2503_04033_gb300 as H
    p = 24
    n, m = H.hps_leaf_sizes(p)
    b = torch.ones(1, p ** 3, dtype=torch.float64, device="cuda")
    T = torch.empty(1, m, m, dtype=torch.float64, device="cuda")
    st = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    ctx = H.hps_create(0, 0)
    try:
        H.hps_leaf_build_dtn(ctx, H.LeafKind(p, 1.0, 0.0), 1, b, T, None, H.HPS_FP64, st)
        assert int(st.item()) == 0
    finally:
        H.hps_destroy(ctx)
    # kappa = 0: a constant has no flux, x has flux +-1 on the x faces (|T| entries reach q^2, sums of m of them)
    one = T[0] @ torch.ones(m, dtype=torch.float64, device="cuda")
    assert float(one.abs().max()) <= 1e-9 * float(T.abs().max())
