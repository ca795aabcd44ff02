"""NMF's fused update, Gram and cross-term pass at the edges of its tiles and
chunks, against the update rules in float64."""
import numpy as np
import pytest

from tests import graphs

pytestmark = pytest.mark.gpu

STEPS = 2


def nmf64(D, W, H):
    obj = [np.sum((D - W @ H.T) ** 2)]
    for _ in range(STEPS):
        H = H * (D.T @ W) / (H @ (W.T @ W))
        W = W * (D @ H) / (W @ (H.T @ H))
        obj.append(np.sum((D - W @ H.T) ** 2))
    return W, H, np.array(obj)


@pytest.mark.parametrize("k", [8, 16, 32, 64])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_fused_step_edges(k, dtype):
    """One graph per size: one row, a tile of 4096 / k rows and its neighbours, a chunk of 2048
    rows and its neighbours, three tiles and a bit.  Every term is positive, so relative
    errors add up: per half step the product (row or column length), the Gram (128 rows in
    FP32, then FP64), the quadratic form (k) and a few operations, in units of 2^-24 (2^-9 on
    top for the BF16 copies that the products read)."""
    import torch
    from paper_1602_02864_gb300 import spmm
    T = 4096 // k
    sizes = [1, T - 1, T, T + 1, 3 * T + 5, 2047, 2048, 2049]
    gs = [graphs.random_csr(n, n, min(0.5, 12.0 / n), i, empty_rows=0.0) for i, n in enumerate(sizes)]
    h = spmm.SparseMatrix.batched(gs, transpose=True, weighted=False)
    try:
        n = sum(sizes)
        g = torch.Generator().manual_seed(k)
        W, H = torch.rand((n, k), generator=g) + 0.1, torch.rand((n, k), generator=g) + 0.1
        Wg, Hg = W.cuda(), H.cuda()
        obj = h.nmf(k, STEPS, Wg, Hg, ftype=spmm.SPMM_F32 if dtype == "f32" else spmm.SPMM_BF16)
        at = 0
        for i, (m, A) in enumerate(zip(sizes, gs)):
            D = (graphs.dense_of(A) != 0).astype(np.float64)
            longest = max(D.sum(0).max(), D.sum(1).max(), 1)
            w, hh, o = nmf64(D, W[at:at + m].double().numpy(), H[at:at + m].double().numpy())
            per_half = (longest + 128 + 2 * k + 8) * 2.0 ** -24 + (2.0 ** -8 if dtype == "bf16" else 0.0)
            tol = 3 * 2 * STEPS * per_half
            for got, ref in ((Wg, w), (Hg, hh)):
                got = got[at:at + m].double().cpu().numpy()
                assert np.all(np.abs(got - ref) <= tol * np.abs(ref) + 1e-30)
            # the objective is a difference of sums as large as these
            size = D.sum() + 2 * np.sum(w * (D @ hh)) + np.sum((w.T @ w) * (hh.T @ hh))
            assert np.all(np.abs(obj[i] - o) <= 4 * tol * max(size, o.max()))
            at += m
    finally:
        h.close()
