"""The device's inverse Cholesky factor: correctly rounded square roots and divisions,
both widths of the kernel, breakdown."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def chol_inv(G):
    import torch
    from paper_1602_02864_gb300 import probe
    Gg = torch.from_numpy(np.ascontiguousarray(G)).cuda()
    R, flag = torch.empty_like(Gg), torch.zeros(1, dtype=torch.int32, device="cuda")
    probe.spmm_probe_chol_inv(Gg, R, flag)
    return R.cpu().numpy(), int(flag.item())


def test_pivots_are_correctly_rounded():
    """1 x 1: the rounded reciprocal of the rounded square root, subnormal pivots included."""
    rng = np.random.default_rng(0)
    pivots = np.concatenate([np.arange(1, 120, dtype=np.float64) ** 2, rng.random(120) * 4,
                             rng.random(40) * 2.0 ** rng.integers(-1000, 1000, 40), [2.0 ** -1060, 3e-310, 1.7e308]])
    for d in pivots:
        R, flag = chol_inv(np.array([[d]]))
        assert flag == 0 and R[0, 0] == 1.0 / np.sqrt(d), d


@pytest.mark.parametrize("b", [1, 2, 15, 16, 17, 24, 31, 32])
def test_inverse_factor(b):
    """R^-T G R^-1 = I.  The factor's backward error is at most (b + 1) 2^-53 |R^T||R| and the
    inverse's residual |R^-1 R - I| at most b 2^-53 |R^-1||R|; three such terms, each at most
    b times the condition number of G, bound the difference."""
    rng = np.random.default_rng(b)
    M = rng.standard_normal((4 * b + 8, b))
    G = M.T @ M
    R, flag = chol_inv(G)
    assert flag == 0 and np.all(np.tril(R, -1) == 0.0)
    tol = 3 * (b + 1) * b * np.linalg.cond(G) * 2.0 ** -53
    assert np.abs(R.T @ G @ R - np.eye(b)).max() <= tol


@pytest.mark.parametrize("b", [3, 16, 20, 32])
def test_breakdown_leaves_the_identity(b):
    M = np.random.default_rng(b).standard_normal((50, b))
    M[:, b - 1] = M[:, 0]
    G = M.T @ M
    G[b - 1] = G[0]
    G[:, b - 1] = G[:, 0]
    G[b - 1, b - 1] = -1.0
    R, flag = chol_inv(G)
    assert flag == 1 and np.array_equal(R, np.eye(b))
