"""The eigensolvers' FP64 products keep the error bound of FP64 arithmetic element by
element, |error| <= (number of operations) 2^-53 sum |a||b|, where the large elements
of the operands do not meet as well as where they do."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
TINY = 2.0 ** -1074             # one rounding among the subnormal numbers
TILE = 64


def operand(kind, n, w, seed):
    """n x w doubles."""
    rng = np.random.default_rng(seed)
    M = rng.standard_normal((n, w))
    if kind == "apart":         # one element of 1 in each column's tile, at other rows for other columns and seeds
        M *= 1e-8
        r = np.arange(0, n, TILE)[:, None] + rng.integers(0, TILE, (-(-n // TILE), w))
        for j in range(w):
            M[np.minimum(r[:, j], n - 1), j] = 1.0
    elif kind == "wide":        # every element of its own size
        M *= np.exp(12 * rng.standard_normal((n, w)))
    elif kind == "disjoint":    # columns with supports of their own
        M[(np.arange(n)[:, None] + 7 * seed) % w != np.arange(w)] = 0.0
    elif kind == "small":       # products among the subnormal numbers
        M *= 1e-158
    elif kind == "subnormal":
        M *= 1e-311
    elif kind == "large":
        M *= 1e150
    return M


KINDS = ["even", "apart", "wide", "disjoint", "small", "subnormal", "large"]


@pytest.mark.parametrize("kinds", [(k, k) for k in KINDS] + [("apart", "even"), ("wide", "disjoint"), ("subnormal", "large")])
@pytest.mark.parametrize("n,p,q", [(40, 3, 5), (1000, 48, 16), (4099, 33, 20)])
def test_tn_error_is_that_of_fp64(kinds, n, p, q):
    """Per tile at most the bound of an FP64 sum of 64 products, then one addition per tile and
    the tree over the row groups."""
    import torch
    from paper_1602_02864_gb300 import probe
    A, B = operand(kinds[0], n, p, 1), operand(kinds[1], n, q, 2)
    ops = TILE + -(-n // TILE) + 16
    for L, R in ((A, B), (A, A)):
        Lg = torch.from_numpy(L).cuda()
        Rg = Lg if R is L else torch.from_numpy(R).cuda()
        C = torch.empty((L.shape[1], R.shape[1]), dtype=torch.float64, device="cuda")
        probe.spmm_probe_ts_tn(Lg, Rg, C)
        Lq, Rq = L.astype(np.longdouble), R.astype(np.longdouble)
        err = np.abs(C.cpu().numpy().astype(np.longdouble) - Lq.T @ Rq)
        assert np.all(err <= ops * U * (np.abs(Lq).T @ np.abs(Rq)) + ops * n * TINY)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n,p,q,alpha,beta", [(17, 5, 3, 1.0, 0.0), (1000, 48, 16, -1.0, 1.0), (333, 64, 24, 1.0, 0.0),
                                              (500, 33, 9, 2.5, -0.5)])
@pytest.mark.parametrize("c_kind", ["even", "wide", "near identity"])
def test_nn_error_is_that_of_fp64(kind, n, p, q, alpha, beta, c_kind):
    """p products summed, scaled, and added to the scaled Out; Out from far below the product to
    far above it."""
    import torch
    from paper_1602_02864_gb300 import probe
    A = operand(kind, n, p, 3)
    C = operand("even" if c_kind == "near identity" else c_kind, p, q, 4)
    if c_kind == "near identity":
        C = np.triu(C * 1e-9) + np.eye(p, q)
    O = np.abs(A @ C) * np.exp(6 * np.random.default_rng(5).standard_normal((n, q)))
    Og = torch.from_numpy(O.copy()).cuda()
    probe.spmm_probe_ts_nn(torch.from_numpy(A).cuda(), torch.from_numpy(C).cuda(), Og, alpha, beta)
    Aq, Cq, Oq = A.astype(np.longdouble), C.astype(np.longdouble), O.astype(np.longdouble)
    err = np.abs(Og.cpu().numpy().astype(np.longdouble) - (beta * Oq + alpha * (Aq @ Cq)))
    bound = U * ((p + 3) * abs(alpha) * (np.abs(Aq) @ np.abs(Cq)) + 3 * abs(beta) * np.abs(Oq)) + 4 * p * TINY
    assert np.all(err <= bound)


def test_localised_vectors_stay_orthonormal():
    """A block Krylov-Schur solve on 400 separate weighted paths, whose eigenvectors live on one
    path each: the vectors are orthonormal to m^2 roundings per cycle (the small rotations that
    make them have as many, and their lengths carry over from restart to restart), and the
    eigenvalues are those of the dense paths within the float32 products' rounding."""
    import scipy.linalg
    import torch
    from paper_1602_02864_gb300 import spmm
    rng = np.random.default_rng(0)
    blocks, exact = [], []
    for i in range(400):
        m = 20 + i % 31
        w = rng.random(m - 1) * (0.2 + 0.7 * i / 400)
        D = np.diag(w.astype(np.float32).astype(np.float64), 1)
        blocks.append(D + D.T)
        exact.append(np.linalg.eigvalsh(D + D.T))
    S = scipy.linalg.block_diag(*blocks)
    n = len(S)
    rows, cols = np.nonzero(S)
    rp = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))]).astype(np.int64)
    h = spmm.SparseMatrix(n, n, rp, cols.astype(np.int32), S[rows, cols].astype(np.float32))
    try:
        nev, m = 8, 64
        V0 = torch.rand((n, 16), dtype=torch.float64, generator=torch.Generator().manual_seed(1)).cuda() * 2 - 1
        U_ = torch.empty((n, nev), dtype=torch.float64, device="cuda")
        ev, res, restarts = h.eigs(nev, V0, block=16, max_basis=m, max_restarts=300, tol=1e-6, evecs=U_)
        G = (U_.T @ U_).cpu().numpy()
        assert np.abs(G - np.eye(nev)).max() <= (restarts + 1) * m * m * U
        assert np.all(res <= 1e-6)
        np.testing.assert_allclose(ev, np.sort(np.concatenate(exact))[::-1][:nev], atol=2e-6)
    finally:
        h.close()
