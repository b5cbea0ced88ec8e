"""FP64 products from exact digits (hps_digit.cu) against higher precision.

``hps_lowrank_dtn`` is one such product with a separate source (T = T0 + s U V^T);
the leaf tests run the other modes.  Bound: with x, y below 2^Ea, 2^Eb in
magnitude per row of U and of V, an entry of U V^T is off by the cut of the
operands (2^-62 each, K terms), the digit pairs left out (7 K 2^14 2^-76 at
i + j = 8, the rest a 256th of that), the unit of the joined sum (2^-58) and
its rounding to FP64; s times it and the source's sum are rounded once more.
The left-out pairs are the largest, 2^-53.2 2^(Ea + Eb) if every digit had its
largest magnitude and one sign, so an entry is within 2^-53 2^(Ea + Eb) +
2^-52 (|s U V^T| + |T0|) at K <= 64; each further 64 terms of K add their own
and one rounding of the entry.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _lowrank(m, r, nbox, seed, graded=False):
    import torch
    import paper_2503_04033_gb300 as H
    rng = np.random.default_rng(seed)
    U, V, T0 = rng.standard_normal((nbox, m, r)), rng.standard_normal((nbox, m, r)), rng.standard_normal((m, m))
    if graded:   # rows and entries over many orders of magnitude, zeros and zero rows among them
        U *= np.exp2(rng.integers(-60, 60, (nbox, m, 1))) * np.exp2(rng.integers(-30, 1, (nbox, m, r)))
        V *= np.exp2(rng.integers(-60, 60, (nbox, m, 1))) * np.exp2(rng.integers(-30, 1, (nbox, m, r)))
        U[rng.random(U.shape) < 0.2] = 0.0
        V[:, ::7] = 0.0
    s = 0.37
    T = torch.full((nbox, m, m), np.nan, dtype=torch.float64, device="cuda")
    H.hps_lowrank_dtn(nbox, m, r, torch.from_numpy(T0).cuda(), s, torch.from_numpy(U).cuda(),
                      torch.from_numpy(V).cuda(), T)
    L = np.longdouble
    ref, bound = np.empty((nbox, m, m), dtype=L), np.empty((nbox, m, m))
    for b in range(nbox):
        P = U[b].astype(L) @ V[b].astype(L).T
        ref[b] = T0.astype(L) + L(s) * P
        tops = np.abs(U[b]).max(axis=1)[:, None] * np.abs(V[b]).max(axis=1)[None, :] * 4.0
        chunks = (r + 63) // 64
        bound[b] = chunks * (2.0 ** -53 * tops * s + 2.0 ** -52 * (
            np.abs(np.abs(U[b]) @ np.abs(V[b]).T) * s * (0.0 if chunks == 1 else 1.0)
            + np.abs(s * P.astype(np.float64)) + np.abs(T0)))
    return T.cpu().numpy(), ref, bound


@pytest.mark.parametrize("m,r,nbox", [(1, 1, 1), (6, 1, 2), (24, 3, 5), (31, 16, 3), (32, 17, 2), (33, 32, 1),
                                      (127, 63, 2), (128, 64, 1), (129, 64, 2), (150, 65, 1), (257, 130, 1),
                                      (600, 32, 3)])
@pytest.mark.parametrize("graded", [False, True])
def test_digit_product_is_exact_to_fp64_rounding(m, r, nbox, graded):
    T, ref, bound = _lowrank(m, r, nbox, 100 * m + r, graded)
    err = np.abs((T - ref).astype(np.float64))
    assert (err <= bound).all(), (err / np.maximum(bound, 1e-300)).max()


def test_digit_product_exact_integers():
    """Small integers: every product and sum is a whole number, so the result is exact."""
    import torch
    import paper_2503_04033_gb300 as H
    rng = np.random.default_rng(3)
    m, r = 200, 64
    U = rng.integers(-(1 << 20), 1 << 20, (m, r)).astype(np.float64)
    V = rng.integers(-(1 << 20), 1 << 20, (m, r)).astype(np.float64)
    T = torch.empty(1, m, m, dtype=torch.float64, device="cuda")
    H.hps_lowrank_dtn(1, m, r, torch.zeros(m, m, dtype=torch.float64, device="cuda"), 1.0,
                      torch.from_numpy(U).cuda(), torch.from_numpy(V).cuda(), T)
    assert (T.cpu().numpy()[0] == (U.astype(np.int64) @ V.astype(np.int64).T).astype(np.float64)).all()


def test_digit_product_extremes():
    """NaN and infinities reach their row or column only, as in plain sums; the largest and the smallest normal
    values survive."""
    import torch
    import paper_2503_04033_gb300 as H
    m, r = 40, 8
    rng = np.random.default_rng(4)
    U, V = rng.standard_normal((m, r)), rng.standard_normal((m, r))
    U[3, 2], V[5, 0] = np.nan, np.inf
    U[7] *= 2.0 ** 1000
    V[9] *= 2.0 ** -1000
    U[11] = 0.0
    U[13] = np.finfo(np.float64).max / 16
    T0 = np.zeros((m, m))
    T = torch.empty(1, m, m, dtype=torch.float64, device="cuda")
    H.hps_lowrank_dtn(1, m, r, torch.from_numpy(T0).cuda(), 1.0, torch.from_numpy(U).cuda(),
                      torch.from_numpy(V).cuda(), T)
    got = T.cpu().numpy()[0]
    bad = np.zeros((m, m), dtype=bool)
    bad[3], bad[:, 5] = True, True
    with np.errstate(over="ignore", invalid="ignore"):
        plain = U @ V.T
        assert (np.isnan(got[bad]) == np.isnan(plain[bad])).all()
        assert (got == plain)[bad & np.isinf(plain)].all() and np.isinf(plain[bad]).any()
        ref = (U.astype(np.longdouble) @ V.astype(np.longdouble).T).astype(np.float64)
        tops = np.abs(U).max(axis=1)[:, None] * np.abs(V).max(axis=1)[None, :] * 4.0
        ok = ~bad & np.isfinite(ref) & np.isfinite(tops)
        assert (np.abs(got - ref)[ok] <= (2.0 ** -53 * tops + 2.0 ** -52 * np.abs(ref))[ok]).all()
    assert (got[11][~bad[11]] == 0.0).all()
    assert np.isfinite(got[7][~bad[7]]).all()
