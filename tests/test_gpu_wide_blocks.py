"""Block widths above 16 and not powers of two in the eigensolvers, whose kernels differ from those
of narrow blocks; and the strides and alignments that lead to a whole warp per X row."""
import numpy as np
import pytest

import oracle
import synth
from tests import graphs

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def sp():
    from paper_1602_02864_gb300 import spmm
    return spmm


def start(n, b, seed):
    import torch
    return (torch.rand((n, b), dtype=torch.float64, generator=torch.Generator().manual_seed(seed)) * 2 - 1).cuda()


def weighted_path(n, seed):
    """A symmetric tridiagonal matrix as CSR and its eigenvalues (float32 values, exact spectrum)."""
    import scipy.linalg
    w = (0.1 + 0.8 * np.random.default_rng(seed).random(n - 1)).astype(np.float32)
    deg = np.full(n, 2)
    deg[[0, -1]] = 1
    rp = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    ci = np.concatenate([[1]] + [[i - 1, i + 1] for i in range(1, n - 1)] + [[n - 2]]).astype(np.int32)
    vals = np.concatenate([[w[0]]] + [[w[i - 1], w[i]] for i in range(1, n - 1)] + [[w[-1]]]).astype(np.float32)
    ev = scipy.linalg.eigh_tridiagonal(np.zeros(n), w.astype(np.float64), eigvals_only=True)[::-1]
    return rp, ci, vals, ev


# Orthonormality: the block is orthonormal to a few b^2 roundings per cycle (Cholesky QR twice) and the
# Ritz vectors are products with up to 64 x 64 rotations: 64^2 roundings per cycle bound both.  A Ritz value
# lies within its residual of an eigenvalue; the residual's own rounding is that of the float32 products,
# 2^-24 times the row length and norm (below 2e-6 for rows of two entries, norm below 2).

@pytest.mark.parametrize("block,nev", [(17, 5), (24, 8), (31, 2)])
def test_krylov_schur_wide_blocks(sp, block, nev):
    import torch
    n = 3000
    rp, ci, vals, ev_ref = weighted_path(n, 1)
    h = sp.SparseMatrix(n, n, rp, ci, vals)
    try:
        V = torch.empty((n, nev), dtype=torch.float64, device="cuda")
        m = min(64, nev + 3 * block) if nev + 2 * block <= 64 else 64
        ev, res, restarts = h.eigs(nev, start(n, block, block), block=block, max_basis=m, max_restarts=400, tol=1e-5, evecs=V)
        assert np.all(res <= 1e-5)
        dist = np.abs(ev[:, None] - ev_ref[None, :]).min(1)
        assert np.all(dist <= res + 2e-6)
        assert np.all(np.abs(ev - ev_ref[:nev]) <= 1e-4)
        G = (V.T @ V).cpu().numpy()
        assert np.abs(G - np.eye(nev)).max() <= (restarts + 1) * 64 * 64 * U
    finally:
        h.close()


@pytest.mark.parametrize("block,nev", [(17, 4), (24, 8), (33, 8), (63, 8), (64, 20)])
def test_filtered_wide_blocks(sp, block, nev):
    import torch
    n = 3000
    rp, ci, vals, ev_ref = weighted_path(n, 2)
    h = sp.SparseMatrix(n, n, rp, ci, vals)
    try:
        V = torch.empty((n, nev), dtype=torch.float64, device="cuda")
        ev, res, iters = h.eigs_filtered(nev, start(n, block, block), degree=16, lower=-2.0, max_iters=80, tol=1e-5, evecs=V)
        assert np.all(res <= 1e-5)
        dist = np.abs(ev[:, None] - ev_ref[None, :]).min(1)
        assert np.all(dist <= res + 2e-6)
        assert np.all(np.abs(ev - ev_ref[:nev]) <= 1e-4)
        G = (V.T @ V).cpu().numpy()
        assert np.abs(G - np.eye(nev)).max() <= (iters + 1) * 64 * 64 * U
    finally:
        h.close()


@pytest.mark.parametrize("block,nsv", [(24, 3), (31, 1)])
def test_svds_wide_blocks(sp, block, nsv):
    A = graphs.random_csr(900, 300, 0.03, 5)
    h = sp.SparseMatrix.from_csr(A, transpose=True)
    try:
        sv, res, _ = h.svds(nsv, start(300, block, 3), block=block, max_basis=64, max_restarts=300, tol=1e-4)
        ref = np.linalg.svd(graphs.dense_of(A), compute_uv=False)[:nsv]
        assert np.all(np.abs(sv - ref) <= 1e-5 * ref[0])
    finally:
        h.close()


@pytest.mark.parametrize("xdtype", ["float32", "bfloat16", "float16"])
@pytest.mark.parametrize("k,pad,shift", [(34, 0, 1), (48, 1, 0), (64, 3, 1), (64, 1, 0), (40, 5, 3), (33, 4, 0)])
def test_whole_warp_rows_by_stride(sp, xdtype, k, pad, shift):
    """Even widths above 32 on an odd row stride or a shifted start take one element a lane, as odd
    widths do; Y is a column block of a wider array, whose other columns stay."""
    import torch
    A = synth.rmat_csr(12, seed=6)
    n = A.n_rows
    h = sp.SparseMatrix.from_csr(A, transpose=True)
    try:
        for tr in (False, True):
            X = synth.dense(n, k, seed=k, mode="int")
            buf = torch.full((n * (k + pad) + shift,), 9.0, dtype=getattr(torch, xdtype), device="cuda")
            Xg = buf[shift:].view(n, k + pad)[:, :k]
            Xg.copy_(torch.from_numpy(X).to(Xg.dtype))
            W = torch.full((n, k + 7), -1.0, device="cuda")
            h.apply(Xg, transpose=tr, Y=W[:, 3:3 + k])
            ref = oracle.spmm(n, n, A.row_ptr, A.col_idx, None, X, transpose=tr)
            got = W.cpu().numpy()
            assert np.array_equal(got[:, 3:3 + k].astype(np.float64), ref)
            assert np.all(got[:, :3] == -1.0) and np.all(got[:, 3 + k:] == -1.0)
    finally:
        h.close()
