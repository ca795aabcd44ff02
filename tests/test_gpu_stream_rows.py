"""Row pointers of the streaming mode: streamed through the slots or kept in HBM, with
the same result and never with more device memory than streamed."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    from paper_1602_02864_gb300 import spmm
    return spmm


def long_and_thin(n):
    """n rows of 0 to 3 entries: the row pointers outweigh the column indices."""
    rng = np.random.default_rng(n)
    rp = np.concatenate([[0], np.cumsum(rng.integers(0, 4, n))]).astype(np.int64)
    return rp, rng.integers(0, 5000, rp[-1]).astype(np.int32)


@pytest.mark.parametrize("slot_kib", [64, 1024, 0])
@pytest.mark.parametrize("weighted", [False, True])
def test_no_more_memory_than_streamed(sp, slot_kib, weighted):
    """Two slots of the block's column indices, values and row pointers, the task list and a page
    of counters: the bytes of a handle that streams its row pointers."""
    import torch
    from paper_1602_02864_gb300 import probe
    n = 1 << 20
    rp, ci = long_and_thin(n)
    vals = np.random.default_rng(1).random(len(ci)).astype(np.float32) if weighted else None
    kw = {"opts": sp.spmm_opts(stream_slot_kib=slot_kib)} if slot_kib else {}
    hs = sp.SparseMatrix(n, 5000, rp, ci, vals, streaming=True, **kw)
    hr = sp.SparseMatrix(n, 5000, rp, ci, vals)
    try:
        info = hs.info()
        block = min(len(ci), (slot_kib << 8) or (64 << 20)) + 32          # entries of a slot
        # a block of so many entries has at most a run of rows more than its share, plus runs of empty rows
        gaps = np.searchsorted(rp, rp[:-1] + block, side="right") - np.arange(n)
        rows = min(n + 5, int(gaps.max()) + 128)
        allowed = 2 * (block * (8 if weighted else 4) + rows * 8) + 16 * (info["n_tasks"] + 1) + 4096
        assert info["device_bytes"] <= allowed
        # streamed with a slot of the caller's, kept in HBM by default here
        per_call = len(ci) * (8 if weighted else 4) + (8 * (n + 1) if slot_kib else 0)
        assert probe.spmm_probe_stream_bytes(hs.handle) == per_call
        assert probe.spmm_probe_stream_bytes(hr.handle) == 0
        for k in (1, 4, 33):
            X = torch.from_numpy(synth.dense(5000, k, seed=k)).cuda()
            Y = hr.apply(X)
            for _ in range(2):
                assert torch.equal(hs.apply(X), Y), k
        hs.sync_status()
    finally:
        hs.close()
        hr.close()
