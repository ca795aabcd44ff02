"""The eigensolvers' FP64 products of tall, narrow matrices (tensor-core digits)
against quadruple precision on the host, at the edges of their tiles."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
TILE = 64                       # rows per tile of the inner dimension


def columns(n, p, ld, seed, tail):
    """n x p inside a row-major array of ld columns; tail: rows of very different size."""
    rng = np.random.default_rng(seed)
    M = rng.standard_normal((n, ld))
    if tail:
        M *= np.exp(3 * rng.standard_normal((n, 1)))
    return M


def tn_bound(A, B):
    """Each tile leaves out at most 2^-59 of the product of its columns' scales (twice the
    largest magnitudes) per row and rounds once; the tiles are added in FP64."""
    n = A.shape[0]
    left_out = np.zeros((A.shape[1], B.shape[1]))
    for r in range(0, n, TILE):
        a, b = np.abs(A[r:r + TILE]), np.abs(B[r:r + TILE])
        left_out += a.shape[0] * 2.0 ** -59 * 4 * np.outer(a.max(0), b.max(0))
    adds = -(-n // TILE) + 16
    return left_out + adds * U * (np.abs(A).T @ np.abs(B))


@pytest.mark.parametrize("n,p,q,extra,tail", [(1, 1, 1, 0, False), (63, 5, 3, 1, False), (64, 16, 16, 0, False),
                                              (65, 17, 16, 3, True), (1000, 48, 16, 16, True), (4097, 64, 64, 0, False),
                                              (3001, 33, 24, 7, True), (20000, 24, 8, 0, True)])
def test_tn_matches_quad(n, p, q, extra, tail):
    import torch
    from paper_1602_02864_gb300 import probe
    A, B = columns(n, p, p + extra, 1, tail), columns(n, q, q + extra, 2, tail)
    C = torch.empty((p, q), dtype=torch.float64, device="cuda")
    probe.spmm_probe_ts_tn(torch.from_numpy(A).cuda()[:, :p], torch.from_numpy(B).cuda()[:, :q], C)
    ref = A[:, :p].T.astype(np.longdouble) @ B[:, :q].astype(np.longdouble)
    err = np.abs(C.cpu().numpy().astype(np.longdouble) - ref)
    assert np.all(err <= tn_bound(A[:, :p], B[:, :q]))
    # A^T A takes the symmetric form
    G = torch.empty((p, p), dtype=torch.float64, device="cuda")
    At = torch.from_numpy(A).cuda()[:, :p]
    probe.spmm_probe_ts_tn(At, At, G)
    G = G.cpu().numpy()
    ref = A[:, :p].T.astype(np.longdouble) @ A[:, :p].astype(np.longdouble)
    assert np.array_equal(G, G.T)
    assert np.all(np.abs(G.astype(np.longdouble) - ref) <= tn_bound(A[:, :p], A[:, :p]))


@pytest.mark.parametrize("n,p,q,extra,alpha,beta", [(1, 1, 1, 0, 1.0, 0.0), (15, 16, 16, 0, -1.0, 1.0),
                                                    (17, 24, 7, 1, -1.0, 1.0), (1000, 56, 24, 8, 1.0, 0.0),
                                                    (4099, 64, 64, 0, 2.5, -0.5), (2500, 33, 9, 2, -1.0, 1.0)])
def test_nn_matches_quad(n, p, q, extra, alpha, beta):
    import torch
    from paper_1602_02864_gb300 import probe
    A, C = columns(n, p, p + extra, 3, True), columns(p, q, q, 4, False)
    O = columns(n, q, q + extra, 5, True)
    Og = torch.from_numpy(O.copy()).cuda()
    probe.spmm_probe_ts_nn(torch.from_numpy(A).cuda()[:, :p], torch.from_numpy(C).cuda(), Og[:, :q], alpha, beta)
    A = A[:, :p]
    ref = beta * O[:, :q].astype(np.longdouble) + alpha * (A.astype(np.longdouble) @ C.astype(np.longdouble))
    scales = 4 * np.outer(np.abs(A).max(1), np.abs(C).max(0))
    bound = (abs(alpha) * (p * 2.0 ** -59 * scales + 4 * U * (np.abs(A) @ np.abs(C))) + 4 * U * abs(beta) * np.abs(O[:, :q]))
    out = Og.cpu().numpy()
    assert np.all(np.abs(out[:, :q].astype(np.longdouble) - ref) <= bound)
    assert np.array_equal(out[:, q:], O[:, q:])                   # nothing beside the block is written


def test_special_values():
    """Zeros, subnormals and the largest magnitudes; an infinity or a NaN spoils its own column or row only."""
    import torch
    from paper_1602_02864_gb300 import probe
    n = 200
    A = columns(n, 6, 6, 7, False)
    A[:, 1] = 0.0
    A[:, 2] *= 1e-310
    A[:, 3] *= 1e200
    A[5, 4] = np.inf
    A[150, 5] = np.nan
    At = torch.from_numpy(A).cuda()
    G = torch.empty((6, 6), dtype=torch.float64, device="cuda")
    probe.spmm_probe_ts_tn(At, At, G)
    G = G.cpu().numpy()
    assert np.all(G[1, :4] == 0.0) and abs(G[2, 0]) <= 1e-306
    assert np.isinf(G[3, 3]) and np.isclose(G[3, 0], A[:, 3] @ A[:, 0], rtol=1e-10)
    assert np.all(np.isnan(G[4:])) and np.all(np.isnan(G[:, 4:]))
    O = torch.zeros((n, 6), dtype=torch.float64, device="cuda")
    probe.spmm_probe_ts_nn(At, torch.eye(6, dtype=torch.float64, device="cuda"), O, 1.0, 0.0)
    O = O.cpu().numpy()
    bad = np.zeros(n, bool)
    bad[[5, 150]] = True
    assert np.all(np.isnan(O[bad])) and np.all(np.isfinite(O[~bad]))
    # A times the identity, to within 2^-59 of each row's largest element
    off = np.abs(O[~bad][:, [0, 3]] - A[~bad][:, [0, 3]])
    assert np.all(off <= 6 * 2.0 ** -59 * 4 * np.abs(A[~bad]).max(1)[:, None] + 4 * U * np.abs(A[~bad][:, [0, 3]]))
