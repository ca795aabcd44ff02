"""Variants of the task kernel that are chosen by size: the weighted merge over
lane groups with two or three blocks per SM, and the tasks claimed at a time."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    from paper_1602_02864_gb300 import spmm
    return spmm


@pytest.mark.parametrize("xdtype", ["float32", "bfloat16", "float16"])
@pytest.mark.parametrize("k", [2, 4, 6, 12, 16, 32])
def test_large_x_variant_same_sums(sp, xdtype, k):
    """A row stride that makes X count as larger than L2 takes the two-block form:
    the same pieces and sums, so the same bits as the three-block form on a dense X, and
    both match the oracle."""
    import torch
    A = synth.rmat_csr(14, seed=5, weighted=True)
    h = sp.SparseMatrix.from_csr(A, transpose=True, opts=sp.spmm_opts(short_runs=2))
    try:
        n, dt = A.n_rows, getattr(torch, xdtype)
        X = torch.from_numpy(synth.dense(n, k, seed=k)).cuda().to(dt)
        wide = torch.zeros((n, 1536 if xdtype == "float32" else 3072), dtype=dt, device="cuda")
        assert wide.numel() * wide.element_size() > 64 << 20
        wide[:, :k] = X
        Xh = X.float().cpu().numpy()
        for tr in (False, True):
            Y, Yw = h.apply(X, transpose=tr), h.apply(wide[:, :k], transpose=tr)
            assert torch.equal(Y, Yw)
            ref = oracle.spmm(n, n, A.row_ptr, A.col_idx, A.values, Xh, transpose=tr)
            scale = oracle.spmm(n, n, A.row_ptr, A.col_idx, A.values, np.abs(Xh), transpose=tr)
            assert np.all(np.abs(Y.cpu().numpy() - ref) <= 1e-5 * scale + 1e-30)
    finally:
        h.close()


@pytest.mark.parametrize("n_tasks", [1, 4000, 16383, 16384, 32768, 60000, 131072, 140000])
@pytest.mark.parametrize("k", [1, 2])
def test_every_task_claimed_once(sp, n_tasks, k):
    """Lists of as many one-row tasks as make the claim size change (1 to 8 at a time):
    every row is written, with its exact sum."""
    import torch
    rng = np.random.default_rng(n_tasks)
    deg = rng.integers(0, 5, n_tasks)
    rp = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    cols = rng.integers(0, 1000, rp[-1]).astype(np.int32)
    h = sp.SparseMatrix(n_tasks, 1000, rp, cols, None, opts=sp.spmm_opts(task_rows=1))
    try:
        assert h.info()["n_tasks"] == n_tasks
        X = synth.dense(1000, k, seed=1, mode="int")
        Y = torch.full((n_tasks, k), -1.0, device="cuda")
        h.apply(torch.from_numpy(X).cuda(), Y=Y)
        ref = oracle.spmm(n_tasks, 1000, rp, cols, None, X)
        assert np.array_equal(Y.cpu().numpy().astype(np.float64), ref)
    finally:
        h.close()


def _hubs(n_hubs, n_short, n_cols, seed):
    """Rows of 513..3000 entries (split) among short ones."""
    rng = np.random.default_rng(seed)
    deg = rng.integers(0, 4, n_hubs + n_short)
    deg[rng.choice(len(deg), n_hubs, replace=False)] = rng.integers(513, 3000, n_hubs)
    rp = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    return rp, rng.integers(0, n_cols, rp[-1]).astype(np.int32)


@pytest.mark.parametrize("n_hubs,n_short", [(1, 0), (40, 3000), (1000, 20000), (5000, 60000)])
def test_split_rows_call_after_call(sp, n_hubs, n_short):
    """Split rows are added by the launch itself on short task lists and by a second
    launch on long ones; widths that take different kernels follow one another on one
    handle, alone and in a batched call, and every sum is exact every time."""
    import torch
    n, m = n_hubs + n_short, 700
    rp, ci = _hubs(n_hubs, n_short, m, n_hubs)
    h = sp.SparseMatrix(n, m, rp, ci, None, transpose=True)
    h2 = sp.SparseMatrix(n, m, rp, ci, None)
    try:
        assert h.info()["n_split_rows"] == n_hubs
        assert (h.info()["n_tasks"] <= 16384) == (n_hubs <= 1000)
        for k in (1, 64, 2, 3, 4, 8, 33, 16, 1, 8):
            X = synth.dense(m, k, seed=k, mode="int")
            Xg = torch.from_numpy(X).cuda()
            ref = oracle.spmm(n, m, rp, ci, None, X)
            for _ in range(2):
                Y = torch.full((n, k), -1.0, device="cuda")
                h.apply(Xg, Y=Y)
                assert np.array_equal(Y.cpu().numpy().astype(np.float64), ref), k
            Ys = [torch.full((n, k), -1.0, device="cuda") for _ in range(2)]
            sp.spmm_apply_batched([h.handle, h2.handle], [Xg, Xg], Ys)
            for Y in Ys:
                assert np.array_equal(Y.cpu().numpy().astype(np.float64), ref), k
            Xt = synth.dense(n, k, seed=k + 1, mode="int")
            Yt = h.apply(torch.from_numpy(Xt).cuda(), transpose=True)
            assert np.array_equal(Yt.cpu().numpy().astype(np.float64),
                                  oracle.spmm(n, m, rp, ci, None, Xt, transpose=True)), k
        sp.spmm_replan(h.handle, sp.spmm_opts(task_nnz=64, long_row=64))
        X = synth.dense(m, 8, seed=9, mode="int")
        Y = h.apply(torch.from_numpy(X).cuda())
        assert np.array_equal(Y.cpu().numpy().astype(np.float64), oracle.spmm(n, m, rp, ci, None, X))
    finally:
        h.close()
        h2.close()


def test_streaming_default_slots(sp):
    """Enough entries for several blocks of the default slot size (16 MiB and more): the
    resident result bit for bit, call after call, at the widths that take other kernels."""
    import torch
    A = synth.rmat_csr(20, n_edges=14 << 20, seed=8)
    assert A.nnz * 4 > 2 * (16 << 20)
    hs = sp.SparseMatrix(A.n_rows, A.n_cols, A.row_ptr, A.col_idx, None, streaming=True)
    hr = sp.SparseMatrix(A.n_rows, A.n_cols, A.row_ptr, A.col_idx, None)
    try:
        for k in (1, 4, 33):
            X = torch.from_numpy(synth.dense(A.n_cols, k, seed=k)).cuda()
            Yr = hr.apply(X)
            for _ in range(3):
                assert torch.equal(hs.apply(X), Yr), k
        hs.sync_status()
    finally:
        hs.close()
        hr.close()


@pytest.mark.parametrize("xdtype", ["float32", "bfloat16", "float16"])
@pytest.mark.parametrize("k", [33, 47, 63])
@pytest.mark.parametrize("weighted", [False, True])
def test_whole_warp_rows(sp, xdtype, k, weighted):
    """Odd widths above 32 (a warp per X row): runs with empty rows at both ends, tasks of 0 to
    512 entries around the batches of 8, against the oracle; small integers exactly."""
    import torch
    rng = np.random.default_rng(k)
    deg = np.concatenate([[0, 0, 7, 8, 9, 0, 15, 16, 17, 1], rng.integers(0, 3, 500), np.zeros(70, np.int64),
                          rng.integers(0, 64, 600), [63] * 64, [0, 600, 0, 64], rng.integers(0, 2, 131), [0]])
    rp = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    n, m = len(deg), 3001
    ci = rng.integers(0, m, rp[-1]).astype(np.int32)
    vals = rng.random(rp[-1]).astype(np.float32) if weighted else None
    h = sp.SparseMatrix(n, m, rp, ci, vals, transpose=True)
    try:
        for tr in (False, True):
            rows, cols = (m, n) if tr else (n, m)
            Xi = synth.dense(cols, k, seed=1, mode="int")
            Xf = torch.from_numpy(synth.dense(cols, k, seed=2)).to(getattr(torch, xdtype))
            Xf_h = Xf.float().numpy()
            Y = torch.full((rows, k), np.nan, device="cuda")
            h.apply(Xf.cuda(), transpose=tr, Y=Y)
            ref = oracle.spmm(n, m, rp, ci, vals, Xf_h, transpose=tr)
            scale = oracle.spmm(n, m, rp, ci, vals, np.abs(Xf_h), transpose=tr)
            assert np.all(np.abs(Y.cpu().numpy() - ref) <= 1e-5 * scale + 1e-30)
            if not weighted:
                Yi = h.apply(torch.from_numpy(Xi).to(getattr(torch, xdtype)).cuda(), transpose=tr)
                assert np.array_equal(Yi.cpu().numpy().astype(np.float64),
                                      oracle.spmm(n, m, rp, ci, None, Xi, transpose=tr))
    finally:
        h.close()
