"""Split rows by each route: added inside the launch, by a second launch on rows of one
element a lane, and both in turn on one handle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("xdtype", ["float32", "bfloat16", "float16"])
@pytest.mark.parametrize("weighted", [False, True])
def test_odd_widths_on_16_and_32_lanes(xdtype, weighted):
    """Widths on 4 to 32 lanes of one element follow one another; small integers, so every sum is
    exact: pattern entries, or values of a power of two."""
    import torch
    from paper_1602_02864_gb300 import spmm
    rng = np.random.default_rng(3)
    n, m = 4000, 900
    deg = rng.integers(0, 6, n)
    deg[rng.choice(n, 60, replace=False)] = rng.integers(513, 2500, 60)
    rp = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    ci = rng.integers(0, m, rp[-1]).astype(np.int32)
    vals = 2.0 ** rng.integers(-1, 2, rp[-1]).astype(np.float32) if weighted else None
    h = spmm.SparseMatrix(n, m, rp, ci, vals, transpose=True)
    try:
        assert h.info()["n_split_rows"] == 60 and h.info()["n_tasks"] <= 16384
        for k in (13, 5, 31, 7, 9, 17, 3, 31, 13, 8):
            for tr in (False, True):
                X = synth.dense(n if tr else m, k, seed=k, mode="int")
                Y = torch.full((m if tr else n, k), -1.0, device="cuda")
                h.apply(torch.from_numpy(X).to(getattr(torch, xdtype)).cuda(), transpose=tr, Y=Y)
                ref = oracle.spmm(n, m, rp, ci, vals, X, transpose=tr)
                assert np.array_equal(Y.cpu().numpy().astype(np.float64), ref), (k, tr)
    finally:
        h.close()
