"""The work that users of this library have it do, as cases to be timed.

Every case goes through the public binding (paper_1602_02864_gb300.spmm): plain
products Y = A X and Y = A^T X on power-law graphs (float32, bfloat16 and float16 X,
pattern and weighted A, k = 1..64), PageRank, the two eigensolvers, NMF and products
over batches of graphs, and the streaming mode (A in pinned host memory).  Graphs are
drawn on the GPU from the seed: R-MAT (a/b/c/d = 0.57/0.19/0.19/0.05, duplicates
merged), symmetrised and degree-normalised R-MAT (largest component) and Chung-Lu
(exponent 2.1).  Sizes are the repository's own configurations, tests and benchmark,
scaled so that a graph is made and planned in about a second.
"""
import math

import numpy as np
import torch

from paper_1602_02864_gb300 import spmm

RMAT = (0.57, 0.19, 0.19, 0.05)
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
CODES = {"f32": spmm.SPMM_F32, "bf16": spmm.SPMM_BF16, "f16": spmm.SPMM_F16}
BYTES = {"f32": 4, "bf16": 2, "f16": 2}


def listed():
    return [
        # the smallest call: one product on a graph of a few thousand vertices (smoke and unit
        # test size), where the host call and the launches are the time
        {"name": "product_4k_k8", "kind": "product", "n": 1 << 12, "deg": 16, "k": 8, "x": "f32", "values": "f32",
         "transpose": False},
        # the plain-SpMM configuration: R-MAT scale 16, weighted, one column
        {"name": "product_64k_k1", "kind": "product", "n": 1 << 16, "deg": 16, "k": 1, "x": "f32", "values": "f32",
         "transpose": False},
        # a ragged middle size with an odd number of half-precision columns, A^T X
        {"name": "product_700k_k33_f16_t", "kind": "product", "n": 700001, "deg": 16, "k": 33, "x": "f16",
         "values": "pattern", "transpose": True},
        # the k sweep at sizes whose X does not fit L2: the paper's headline width, k = 8
        {"name": "product_8m_k8", "kind": "product", "n": 1 << 23, "deg": 16, "k": 8, "x": "f32",
         "values": "pattern", "transpose": False},
        # the precision configuration: bfloat16 X, 16 columns, weighted A
        {"name": "product_4m_k16_bf16", "kind": "product", "n": 1 << 22, "deg": 16, "k": 16, "x": "bf16",
         "values": "f32", "transpose": False},
        # the widest product, A^T X
        {"name": "product_2m_k64_t", "kind": "product", "n": 1 << 21, "deg": 16, "k": 64, "x": "f32",
         "values": "pattern", "transpose": True},
        # PageRank: 30 iterations, damping 0.85 (k = 1 products on A^T)
        {"name": "pagerank_4m", "kind": "pagerank", "n": 1 << 22, "deg": 16, "iters": 30},
        # block Krylov-Schur, block 16, basis 64: the work of a solve (expansions, projections, a thick
        # restart), bounded to one restart, since rounding grows from restart to restart until the outputs
        # of a whole solve are no more alike than its tolerance
        {"name": "eigs_256k", "kind": "eigs", "n": 1 << 18, "nev": 8, "restarts": 1},
        # Chebyshev-filtered subspace iteration, block 16, degree 20, as for the clustered top spectra
        {"name": "eigs_filtered_1m", "kind": "eigs_filtered", "n": 1 << 20, "nev": 8, "degree": 20, "iters": 4},
        # the batching configuration: NMF on Chung-Lu graphs held by one block-diagonal handle
        {"name": "nmf_64_graphs_k16", "kind": "nmf", "graphs": 64, "nmax": 200000, "k": 16, "steps": 10, "x": "f32"},
        # the same graphs as separate handles, each with its own k, one call
        {"name": "batched_48_graphs", "kind": "batched", "graphs": 48, "nmax": 200000, "k": 32, "x": "f32"},
        # semi-external: A streamed from pinned host memory, X and Y resident, k = 4
        {"name": "streaming_4m_k4", "kind": "streaming", "n": 1 << 22, "deg": 16, "k": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product"] * 6 + ["pagerank", "eigs", "eigs_filtered", "nmf", "batched", "streaming"])
    if kind == "product":
        k = rng.choice([1, 2, 3, 4, 5, 7, 8, 13, 16, 24, 31, 32, 33, 48, 64])
        hi = min(1 << 23, (1 << 27) // k)             # X of at most 512 MB
        x = rng.choice(["f32", "f32", "f32", "bf16", "f16"])
        values = rng.choice(["pattern", "f32"] + (["own"] if x != "f32" else []))
        return {"kind": kind, "n": _log(rng, 1000, hi), "deg": rng.choice([8, 16, 16, 24]) if hi < (1 << 23) else 16,
                "k": k, "x": x, "values": values, "transpose": rng.random() < 0.4}
    if kind == "pagerank":
        return {"kind": kind, "n": _log(rng, 2000, 1 << 22), "deg": rng.choice([8, 16]),
                "iters": rng.choice([10, 20, 30])}
    if kind == "eigs":
        return {"kind": kind, "n": _log(rng, 1 << 14, 1 << 18), "nev": rng.choice([3, 4, 6, 8]),
                "restarts": rng.choice([0, 1])}
    if kind == "eigs_filtered":
        return {"kind": kind, "n": _log(rng, 1 << 15, 1 << 20), "nev": rng.choice([4, 6, 8]),
                "degree": rng.choice([10, 16, 20]), "iters": rng.choice([2, 3, 4])}
    if kind == "nmf":
        return {"kind": kind, "graphs": rng.randint(1, 64), "nmax": rng.choice([20000, 60000, 200000]),
                "k": rng.choice([5, 8, 10, 16, 16]), "steps": rng.choice([4, 8, 10]),
                "x": rng.choice(["f32", "f32", "bf16"])}
    if kind == "batched":
        return {"kind": kind, "graphs": rng.randint(2, 48), "nmax": rng.choice([20000, 60000, 200000]),
                "k": rng.choice([0, 8, 16, 32]), "x": rng.choice(["f32", "bf16"])}   # 0: widths 1, 8, 33 in turn
    return {"kind": kind, "n": _log(rng, 1 << 18, 1 << 22), "deg": 16, "k": rng.choice([1, 4, 8])}


# ------------------------------------------------------------------ inputs
class _Graph:
    """A host CSR matrix (int64 row pointers, int32 columns, float32 values or None)."""

    def __init__(self, n_rows, n_cols, row_ptr, col_idx, values=None):
        self.n_rows, self.n_cols = n_rows, n_cols
        self.row_ptr, self.col_idx, self.values = row_ptr, col_idx, values


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _rmat_edges(n, m, g):
    """m R-MAT edges on n vertices (drawn on the next power of two, scaled down to n)."""
    levels = max(1, (n - 1).bit_length())
    src = torch.zeros(m, dtype=torch.int32, device="cuda")
    dst = torch.zeros(m, dtype=torch.int32, device="cuda")
    a, b, c, _ = RMAT
    for _level in range(levels):
        u = torch.rand(m, generator=g, device="cuda")
        row = u >= a + b
        col = ((u >= a) & ~row) | (u >= a + b + c)
        src.mul_(2).add_(row)
        dst.mul_(2).add_(col)
    if n != 1 << levels:
        src = (src.long() * n) >> levels
        dst = (dst.long() * n) >> levels
    return src.long(), dst.long()


def _coo_to_csr(n_rows, n_cols, src, dst):
    """Duplicates merged; (row_ptr, cols) on the GPU, int64."""
    key = torch.unique(src * n_cols + dst)
    rows = torch.div(key, n_cols, rounding_mode="floor")
    cols = key - rows * n_cols
    rp = torch.zeros(n_rows + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=n_rows), 0)
    return rp, rows, cols


def _to_host(n_rows, n_cols, rp, cols, values=None):
    return _Graph(n_rows, n_cols, rp.cpu().numpy(), cols.to(torch.int32).cpu().numpy(),
                  None if values is None else values.cpu().numpy())


def _rmat(case, g):
    n = case["n"]
    src, dst = _rmat_edges(n, n * case["deg"], g)
    rp, _, cols = _coo_to_csr(n, n, src, dst)
    values = None
    if case.get("values", "pattern") != "pattern":
        values = torch.rand(cols.numel(), generator=g, device="cuda")
    return rp, cols, values


def _symmetric(case):
    """Largest component of the symmetrised R-MAT graph with lognormal weights, D^-1/2 A D^-1/2.  One graph
    for every seed (the size of the component is drawn too); the start block is the seed's."""
    n = case["n"]
    g = _generator(n)
    src, dst = _rmat_edges(n, 8 * n, g)
    rp, rows, cols = _coo_to_csr(n, n, torch.cat([src, dst]), torch.cat([dst, src]))
    inside = torch.zeros(n, dtype=torch.bool, device="cuda")
    inside[torch.argmax(rp[1:] - rp[:-1])] = True
    while True:
        before = int(inside.sum())
        inside[cols[inside[rows]]] = True
        if int(inside.sum()) == before:
            break
    new = torch.cumsum(inside, 0) - 1
    keep = inside[rows]
    rows, cols, m = new[rows[keep]], new[cols[keep]], before
    lo, hi = torch.minimum(rows, cols), torch.maximum(rows, cols)
    pairs, of = torch.unique(lo * m + hi, return_inverse=True)
    w = torch.exp(torch.randn(pairs.numel(), generator=g, device="cuda", dtype=torch.float64))[of]
    rp = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=m), 0)
    # degrees summed on the host, in the order of the entries (a GPU scan rounds differently from run to run)
    deg = torch.from_numpy(np.add.reduceat(w.cpu().numpy(), rp[:-1].cpu().numpy())).cuda()
    s = deg.rsqrt()
    w = w * (s[lo] * s[hi])
    return m, rp, cols, w.float()


def _chung_lu_sizes(case):
    """(vertices, edges drawn) of each graph: sizes spread evenly over the logarithm of [1000, nmax], not
    in order of size, average degree 8..32."""
    count = case["graphs"]
    sizes = []
    for i in range(count):
        n = int(1000.0 * (case["nmax"] / 1000.0) ** (((i * 0.7548776662466927) % 1.0)))
        sizes.append((n, int(n * (8 + 24 * ((i * 0.5698402909980532) % 1.0)))))
    return sizes


def _chung_lu(case, g):
    """Directed Chung-Lu graphs, exponent 2.1: sources by weight (i + 1)^(-1/1.1), targets by the same
    weights under a permutation."""
    out = []
    for n, m in _chung_lu_sizes(case):
        cum = torch.from_numpy(np.cumsum(np.arange(1, n + 1) ** (-1.0 / 1.1))).cuda()
        u = torch.rand(2, m, generator=g, device="cuda", dtype=torch.float64) * cum[-1]
        ends = torch.searchsorted(cum, u, right=True).clamp_(max=n - 1)
        perm = torch.randperm(n, generator=g, device="cuda")
        rp, _, cols = _coo_to_csr(n, n, ends[0], perm[ends[1]])
        out.append((n, rp, cols))
    return out


def _widths(case):
    return [case["k"] or (1, 8, 33)[i % 3] for i in range(case["graphs"])]


def _uniform(shape, g, dtype="f32"):
    return (torch.rand(shape, generator=g, device="cuda") * 2 - 1).to(DTYPES[dtype])


def _values(case, values):
    """Stored values as the library takes them: float32 numpy, or 16-bit of X's own type."""
    if values is None:
        return None
    return values.to(DTYPES[case["x"]]).cpu() if case["values"] == "own" else values.cpu().numpy()


def prepare(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    if kind in ("product", "streaming"):
        n = case["n"]
        rp, cols, values = _rmat(case, g)
        G = _to_host(n, n, rp, cols)
        X = _uniform((n, case["k"]), g, case.get("x", "f32"))
        if kind == "streaming":
            h = spmm.SparseMatrix(n, n, G.row_ptr, G.col_idx, None, streaming=True)
            return {"kind": kind, "h": h, "X": X, "transpose": False}
        h = spmm.SparseMatrix(n, n, G.row_ptr, G.col_idx, _values(case, values), transpose=case["transpose"])
        return {"kind": kind, "h": h, "X": X, "transpose": case["transpose"]}
    if kind == "pagerank":
        n = case["n"]
        rp, cols, _ = _rmat(case, g)
        G = _to_host(n, n, rp, cols)
        return {"kind": kind, "h": spmm.SparseMatrix(n, n, G.row_ptr, G.col_idx, None, transpose=True),
                "iters": case["iters"]}
    if kind in ("eigs", "eigs_filtered"):
        n, rp, cols, w = _symmetric(case)
        G = _to_host(n, n, rp, cols, w)
        V0 = torch.rand((n, 16), generator=g, device="cuda", dtype=torch.float64) * 2 - 1
        return {"kind": kind, "h": spmm.SparseMatrix.from_csr(G), "V0": V0, "case": dict(case)}
    graphs = _chung_lu(case, g)
    if kind == "nmf":
        k = case["k"]
        h = spmm.SparseMatrix.batched([_to_host(n, n, rp, cols) for n, rp, cols in graphs], transpose=True,
                                      weighted=False)
        total = sum(n for n, _, _ in graphs)
        W = torch.rand((total, k), generator=g, device="cuda") + 0.01
        Ht = torch.rand((total, k), generator=g, device="cuda") + 0.01
        return {"kind": kind, "h": h, "W": W, "Ht": Ht, "case": dict(case)}
    hs, Xs, Ys = [], [], []
    for (n, rp, cols), k in zip(graphs, _widths(case)):
        G = _to_host(n, n, rp, cols)
        hs.append(spmm.SparseMatrix(n, n, G.row_ptr, G.col_idx, None))
        Xs.append(_uniform((n, k), g, case["x"]))
        Ys.append(torch.empty((n, k), device="cuda"))
    return {"kind": kind, "hs": hs, "Xs": Xs, "Ys": Ys}


def run(state):
    kind = state["kind"]
    if kind in ("product", "streaming"):
        return state["h"].apply(state["X"], transpose=state["transpose"])
    if kind == "pagerank":
        return state["h"].pagerank(0.85, state["iters"])
    if kind == "eigs":
        c = state["case"]
        evals, residuals, _ = state["h"].eigs(c["nev"], state["V0"], block=16, max_basis=64,
                                              max_restarts=c["restarts"], tol=1e-6)
        return evals, residuals
    if kind == "eigs_filtered":
        c = state["case"]
        vectors = torch.empty((state["V0"].shape[0], c["nev"]), dtype=torch.float64, device="cuda")
        evals, residuals, _ = state["h"].eigs_filtered(c["nev"], state["V0"], degree=c["degree"], lower=-1.0,
                                                       max_iters=c["iters"], tol=1e-6, evecs=vectors)
        return evals, residuals, vectors
    if kind == "nmf":
        c = state["case"]
        W, Ht = state["W"].clone(), state["Ht"].clone()       # the factors are updated in place
        objective = state["h"].nmf(c["k"], c["steps"], W, Ht, ftype=CODES[c["x"]])
        return W, Ht, objective
    spmm.spmm_apply_batched([h.handle for h in state["hs"]], state["Xs"], state["Ys"])
    return state["Ys"]


# ------------------------------------------------------------------ what a pass cannot do without
def _stored(n, m):
    """Expected distinct R-MAT edges among m drawn on n vertices (exact for a power of two)."""
    s = max(1, (n - 1).bit_length())
    a, b, _, d = RMAT
    total = 0.0
    for i in range(s + 1):
        for j in range(s + 1 - i):
            cells = math.comb(s, i) * math.comb(s - i, j) * 2.0 ** j
            total += cells * -math.expm1(-m * a ** i * b ** j * d ** (s - i - j))
    return min(float(m), total)


def work(case):
    kind = case["kind"]
    if kind in ("product", "streaming"):
        n, k = case["n"], case["k"]
        nnz = _stored(n, n * case["deg"])
        v = {"pattern": 0, "f32": 4, "own": 2}[case.get("values", "pattern")]
        return {"bytes": nnz * (4 + v) + 8 * (n + 1) + n * k * (BYTES[case.get("x", "f32")] + 4),
                "flops": 2 * nnz * k}
    if kind == "pagerank":      # per iteration: A^T once, z read, ranks and 1/degree read, ranks and z written
        n, nnz = case["n"], _stored(case["n"], case["n"] * case["deg"])
        return {"bytes": case["iters"] * (4 * nnz + 8 * (n + 1) + 20 * n), "flops": case["iters"] * (2 * nnz + 6 * n)}
    if kind in ("eigs", "eigs_filtered"):
        n = case["n"] * 0.55                          # vertices of the largest component
        nnz = 15.0 * case["n"]
        product = nnz * 8 + 8 * n + n * 16 * 8        # one block product, 16 float32 columns
        if kind == "eigs":
            # expansions of the basis (FP64 block Gram-Schmidt twice, CholQR twice), projections, Ritz vectors
            flops, blocks, byte = 0.0, 0, 0.0
            for cycle in range(case["restarts"] + 1):
                first = 16 if cycle == 0 else case["nev"] + 16
                cur = first
                while cur + 16 <= 64:
                    flops += n * (2 * 4 * cur * 16 + 2 * 4 * 16 * 16)
                    byte += n * 8 * (2 * (2 * cur + 32) + 4 * 16)
                    cur, blocks = cur + 16, blocks + 1
                flops += n * (2 * cur * cur + 4 * cur * (case["nev"] + 16))
                byte += n * 8 * (2 * cur + 2 * (case["nev"] + 16))
            return {"bytes": byte + blocks * product, "flops": flops + blocks * 2 * nnz * 16}
        products = case["iters"] * (case["degree"] + 1) + 1
        dense = (case["iters"] + 1) * n * (2 * 3 * 16 * 16 + 4 * 16 * 16)
        return {"bytes": products * product + (case["iters"] + 1) * n * 16 * 8 * 6,
                "flops": products * 2 * nnz * 16 + dense}
    sizes = _chung_lu_sizes(case)       # few of a Chung-Lu graph's drawn edges are merged: about 15%
    n, nnz = sum(v for v, _ in sizes), 0.85 * sum(m for _, m in sizes)
    if kind == "nmf":           # per step: both products, both factors and both numerators read, the factors written
        k, steps = case["k"], case["steps"]
        per = 2 * (4 * nnz + 8 * n + 2 * 4 * n * k) + 2 * 3 * 4 * n * k
        return {"bytes": steps * per, "flops": steps * (4 * nnz * k + 2 * 4 * n * k * k)}
    rows = sum(v * k for (v, _), k in zip(sizes, _widths(case)))
    flops = 2 * 0.85 * sum(m * k for (_, m), k in zip(sizes, _widths(case)))
    return {"bytes": 4 * nnz + 8 * n + rows * (BYTES[case["x"]] + 4), "flops": flops}


# ------------------------------------------------------------------ the same in 64 bits, plain torch
def _csr64(n_rows, n_cols, rp, cols, values=None):
    v = torch.ones(cols.numel(), dtype=torch.float64, device="cuda") if values is None else values.double()
    return torch.sparse_csr_tensor(rp, cols, v, size=(n_rows, n_cols))


def _transposed(n_rows, n_cols, rp, cols, values=None):
    rows = torch.repeat_interleave(torch.arange(n_rows, device="cuda"), rp[1:] - rp[:-1])
    order = torch.argsort(cols, stable=True)
    tp = torch.zeros(n_cols + 1, dtype=torch.int64, device="cuda")
    tp[1:] = torch.cumsum(torch.bincount(cols, minlength=n_cols), 0)
    return _csr64(n_cols, n_rows, tp, rows[order], None if values is None else values[order])


def _filtered64(S, n, nev, lower=-1.0, degree=24, most=80):
    """Top eigenvalues of a symmetric S by Chebyshev-filtered subspace iteration."""
    U = torch.linalg.qr(torch.randn((n, 40), generator=_generator(1), device="cuda", dtype=torch.float64))[0]
    last = None
    for _ in range(most):
        SU = S @ U
        theta, Y = torch.linalg.eigh(U.T @ SU)
        U = U @ Y
        top = theta.flip(0)[:nev]
        if last is not None and float((top - last).abs().max()) < 1e-14:
            return top
        last = top
        lo, hi = lower, float(theta[0])
        e, c = (hi - lo) / 2, (hi + lo) / 2
        s1 = e / (float(theta[-1]) - c)
        s, Yp = s1, U
        Yc = (S @ U - c * U) * (s1 / e)
        for _j in range(degree - 1):
            sn = 1.0 / (2.0 / s1 - s)
            Yp, Yc = Yc, (S @ Yc - c * Yc) * (2 * sn / e) - s * sn * Yp
            s = sn
        U = torch.linalg.qr(Yc)[0]
    return last


def exact(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    if kind in ("product", "streaming"):
        n = case["n"]
        rp, cols, values = _rmat(case, g)
        X = _uniform((n, case["k"]), g, case.get("x", "f32")).double()
        if values is not None and case["values"] == "own":
            values = values.to(DTYPES[case["x"]])
        A = (_transposed if case.get("transpose") else _csr64)(n, n, rp, cols, values)
        return A @ X
    if kind == "pagerank":
        n = case["n"]
        rp, cols, _ = _rmat(case, g)
        deg = (rp[1:] - rp[:-1]).double()
        dangling = deg == 0
        inv = torch.where(dangling, 0.0, 1.0 / deg.clamp(min=1))
        At = _transposed(n, n, rp, cols)
        x = torch.full((n, 1), 1.0 / n, dtype=torch.float64, device="cuda")
        residuals = []
        for _ in range(case["iters"]):
            y = At @ (x * inv[:, None])
            new = 0.15 / n + 0.85 * (x[dangling].sum() / n + y)
            residuals.append((new - x).abs().sum())
            x = new
        return x[:, 0], torch.stack(residuals).cpu().numpy()
    if kind == "eigs":
        # one restart leaves Ritz values of the method's own, not eigenvalues
        return None
    if kind == "eigs_filtered":
        n, rp, cols, w = _symmetric(case)
        return _filtered64(_csr64(n, n, rp, cols, w), n, case["nev"]).cpu().numpy(), None, None
    graphs = _chung_lu(case, g)
    if kind == "nmf":
        k = case["k"]
        total = sum(n for n, _, _ in graphs)
        W = (torch.rand((total, k), generator=g, device="cuda") + 0.01).double()
        Ht = (torch.rand((total, k), generator=g, device="cuda") + 0.01).double()
        objective, at = np.zeros((case["graphs"], case["steps"] + 1)), 0
        for i, (n, rp, cols) in enumerate(graphs):
            A, At = _csr64(n, n, rp, cols), _transposed(n, n, rp, cols)
            w, h = W[at:at + n], Ht[at:at + n]
            for t in range(case["steps"] + 1):
                if t:
                    h = h * ((At @ w) / (h @ (w.T @ w) + 1e-12))
                    w = w * ((A @ h) / (w @ (h.T @ h) + 1e-12))
                objective[i, t] = float(cols.numel() - 2 * (w * (A @ h)).sum() + ((w.T @ w) * (h.T @ h)).sum())
            W[at:at + n], Ht[at:at + n] = w, h
            at += n
        return W, Ht, objective
    return [_csr64(n, n, rp, cols) @ _uniform((n, k), g, case["x"]).double()
            for (n, rp, cols), k in zip(graphs, _widths(case))]
