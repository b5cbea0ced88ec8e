"""Entry-wise accuracy of the FP64 products from exact digits.

Rows of A and columns of B share one scale each, so an entry whose sum of
|a||b| is far below the product of its scales has to be summed as it stands.
``hps_lowrank_dtn`` (T = T0 + s U V^T) holds every entry to the bound of an FP64
sum, K 2^-53 sum |u||v| per 64 terms (asserted with a factor of two) and one
rounding each for s and T0.  The LU of a matrix whose scales lie far apart runs
on plain FP64 sums.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _factors(kind, m, r, rng):
    U, V = rng.standard_normal((m, r)), rng.standard_normal((m, r))
    k = np.arange(r)
    if kind == "opposed":            # columns of U graded one way, of V the other
        U, V = U * np.exp2(-1.0 * k), V * np.exp2(1.0 * k)
    elif kind == "opposed_mild":
        U, V = U * np.exp2(-0.5 * k), V * np.exp2(0.5 * k)
    elif kind == "spread":           # entries over 400 binary orders, a third of them zero
        U *= np.exp2(rng.integers(-400, 1, U.shape))
        V *= np.exp2(rng.integers(-400, 1, V.shape))
        U[rng.random(U.shape) < 0.33] = 0.0
    elif kind == "few":              # one row and one column whose large entries do not meet
        U[m // 2, 0], U[m // 2, 1:] = 1.0, np.exp2(-70.0)
        V[m // 3, 0] = 0.0
    elif kind == "subnormal":        # subnormal entries against large ones, subnormal rows among them
        U[1::3] *= 2.0 ** -1060
        U[::3, ::2] *= 2.0 ** -1070
        V *= 2.0 ** 600
    return U, V


@pytest.mark.parametrize("kind", ["plain", "opposed", "opposed_mild", "spread", "few", "subnormal"])
@pytest.mark.parametrize("m,r,nbox", [(2, 2, 1), (33, 17, 1), (33, 17, 130), (129, 64, 1), (160, 65, 1), (200, 8, 110),
                                      (300, 7, 2)])
def test_lowrank_entries_are_as_good_as_fp64_sums(kind, m, r, nbox):
    """Sizes on both sides of the lines between plain sums and digits."""
    import torch
    import paper_2503_04033_gb300 as H
    rng = np.random.default_rng(10 * m + r)
    U, V = (np.stack(x) for x in zip(*(_factors(kind, m, r, rng) for _ in range(nbox))))
    T = torch.full((nbox, m, m), np.nan, dtype=torch.float64, device="cuda")
    H.hps_lowrank_dtn(nbox, m, r, torch.zeros(m, m, dtype=torch.float64, device="cuda"), 1.0,
                      torch.from_numpy(U).cuda(), torch.from_numpy(V).cuda(), T)
    L = np.longdouble
    for b in {0, nbox // 2, nbox - 1}:
        ref = U[b].astype(L) @ V[b].astype(L).T
        size = np.abs(U[b]).astype(L) @ np.abs(V[b]).astype(L).T
        err = np.abs(T[b].cpu().numpy().astype(L) - ref)
        bound = (2 * min(r, 64) + 2 * ((r + 63) // 64)) * L(2.0) ** -53 * size + L(2.0) ** -1073
        assert (err <= bound).all(), float((err / np.maximum(bound, L(1e-4000))).max())


def _lu_longdouble(A, B):
    """A^-1 B by partial-pivot elimination in long double."""
    M = np.hstack([A, B]).astype(np.longdouble)
    n = len(A)
    for c in range(n):
        r = c + int(np.argmax(np.abs(M[c:, c])))
        M[[c, r]] = M[[r, c]]
        M[c + 1:, c:] -= np.outer(M[c + 1:, c] / M[c, c], M[c, c:])
    for c in range(n - 1, -1, -1):
        M[c, n:] = (M[c, n:] - M[c, c + 1:n] @ M[c + 1:, n:]) / M[c, c]
    return M[:, n:]


def _s_2d(p, h, kappa, b):
    """S of 2-D boxes with fields b [nbox, p^2] from the library, and A_ii, A_ib of each."""
    import torch
    import paper_2503_04033_gb300 as H
    n, m = oracle.sizes_2d(p)
    S = torch.full((len(b), n, m), np.nan, dtype=torch.float64, device="cuda")
    T = torch.empty(len(b), m, m, dtype=torch.float64, device="cuda")
    st = torch.full((len(b),), -1, dtype=torch.int32, device="cuda")
    H.hps_leaf2d_solve(p, h, kappa, len(b), torch.from_numpy(b).cuda(), T=T, S=S, box_status=st)
    assert (st.cpu().numpy() == 0).all()
    A = [oracle.leaf_matrix_2d(p, h, kappa, x) for x in b]
    return S.cpu().numpy(), [(a[:n, :n], a[:n, n:]) for a in A]


@pytest.mark.parametrize("p", [10, 16])
def test_flat_boxes_keep_small_entries(p):
    """Sides 1 : 1e-6: S has entries many orders below its largest; each keeps 28 bits (a plain elimination 43)."""
    b = np.random.default_rng(p).uniform(0.5, 1.5, (2, p * p))
    S, blocks = _s_2d(p, [1.0, 1e-6], 10.0, b)
    for got, (Aii, Aib) in zip(S, blocks):
        ref = -_lu_longdouble(Aii, Aib)
        big = np.abs(ref) > 1e-300
        rel = (np.abs(got - ref)[big] / np.abs(ref)[big]).astype(np.float64)
        assert rel.max() < 2.0 ** -28, rel.max()


@pytest.mark.parametrize("decades", [2, 8, 10, 12, 14, 16])
def test_coefficients_that_jump_from_node_to_node(decades):
    """b between 1 and 10^decades, independently at every node: the LU's blocks
    hold pivots as far apart.  S of ten boxes is as close to long double as a
    plain FP64 elimination (geometric means of the norms of the errors and of
    the worst row's, each relative to its own size; a factor of four for another
    order of operations)."""
    p = 16
    rng = np.random.default_rng(decades)
    b = 10.0 ** rng.uniform(0, decades, (10, p * p))
    S, blocks = _s_2d(p, [1.0 / 64] * 2, 10.0, b)
    e = []
    for got, (Aii, Aib) in zip(S, blocks):
        ref = -_lu_longdouble(Aii, Aib)
        plain = -np.linalg.solve(Aii, Aib)
        d = [np.abs(x - ref) for x in (got, plain)]
        e.append([f(x) for x in d for f in (lambda x: float(np.sqrt((x ** 2).sum() / (ref ** 2).sum())),
                                            lambda x: float((x.max(axis=1) / np.abs(ref).max(axis=1)).max()))])
    fro, row, fro0, row0 = np.exp(np.log(np.array(e)).mean(axis=0))
    print(f"decades {decades}: norm {fro:.2e} (plain {fro0:.2e}), worst row {row:.2e} (plain {row0:.2e})")
    assert fro < 4 * fro0 and row < 4 * row0


@pytest.mark.parametrize("h", [1.0, 1.0 / 64, 1.0 / 1024])
def test_small_impedance_leaves(h):
    """The impedance system's face rows are of order 1 / h, its interior rows of
    order 1 / h^2.  The face values behind R = I - 2 i eta x are as close to long
    double as a plain FP64 elimination's (factor of four as above, and the
    rounding of I - R)."""
    import torch
    import paper_2503_04033_gb300 as H
    p, kappa, eta = 6, 10.0, 10.0
    n, m = oracle.sizes(p)
    b = np.random.default_rng(5).uniform(0.5, 1.5, (3, p ** 3))
    R = torch.empty(3, m, m, dtype=torch.complex128, device="cuda")
    H.hps_leaf_iti(H.LeafKind(p, [h] * 3, kappa), eta, 3, torch.from_numpy(b).cuda(), R)
    got = R.cpu().numpy()
    e = []
    for i in range(3):
        A = oracle.leaf_matrix(p, [h] * 3, kappa, b[i])
        E = np.diag(np.r_[np.zeros(n), np.ones(m)])
        K, F = np.block([[A, -eta * E], [eta * E, A]]), np.zeros((2 * (n + m), m))
        F[n:n + m] = np.eye(m)
        ref, plain = _lu_longdouble(K, F), np.linalg.solve(K, F)
        faces = [slice(n, n + m), slice(2 * n + m, None)]
        x = [got[i].imag / (-2 * eta), (got[i].real - np.eye(m)) / (2 * eta)]
        size = np.sqrt(sum((ref[s] ** 2).sum() for s in faces))
        e.append([float(np.sqrt(sum(((y - ref[s]) ** 2).sum() for y, s in zip(v, faces))) / size)
                  for v in (x, [plain[s] for s in faces])] + [float(2.0 ** -52 * np.sqrt(m) / (2 * eta) / size)])
    err, err0, unit = np.exp(np.log(np.array(e)).mean(axis=0))
    print(f"h {h}: {err:.2e} (plain {err0:.2e}, rounding of I - R {unit:.2e})")
    assert err < 4 * err0 + unit
