"""The Householder panel reduction over the range of float64: matrices far from
1, whose columns are brought near it by a power of two; a small first column in
front of a large trailing matrix; columns that leave and enter the range that
needs no scaling inside a panel. Bars: the backward error of an n-step
orthogonal reduction, n eps ||A||, on the eigenvalues of T and on
Q^T A Q - T (largest entry) with Q formed from the stored reflectors."""
import numpy as np
import pytest

from paper_1703_00387_gb300 import binding as B

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    c.close()


def _check(ctx, S, unit):
    """S = unit x a matrix whose squares are in range (unit: a power of two)."""
    import torch
    n = S.shape[0]
    A = torch.from_numpy(S.copy()).cuda()
    d, e, tau = (torch.full((n,), float("nan"), dtype=torch.float64, device="cuda:0") for _ in range(3))
    B.osmps_sytrd(ctx, A, d, e, tau)
    A, tau = A.cpu().numpy(), tau.cpu().numpy()
    d, e = d.cpu().numpy() / unit, e.cpu().numpy()[:n - 1] / unit
    assert np.isfinite(d).all() and np.isfinite(e).all() and np.isfinite(tau[:n - 1]).all()
    T = np.diag(d) + np.diag(e, 1) + np.diag(e, -1)
    S1 = S / unit
    w = np.linalg.eigvalsh(S1)
    bar = n * EPS * np.abs(w).max()
    assert np.abs(np.linalg.eigvalsh(T) - w).max() <= bar
    Q = np.eye(n)
    for j in range(n - 1):  # H(0) H(1) ... H(n - 2)
        v = np.zeros(n)
        v[j + 1], v[j + 2:] = 1.0, A[j, j + 2:]
        Q -= np.outer(Q @ v, tau[j] * v)
    assert np.abs(Q.T @ S1 @ Q - T).max() <= bar


def _random(n, seed):
    M = np.random.default_rng(seed).standard_normal((n, n))
    return M + M.T


@pytest.mark.parametrize("p", [-500, -330, -130, 100, 130, 330, 500, 960, 1010])
@pytest.mark.parametrize("n", [33, 300, 600])  # sums taken in one and in two exchanges
def test_scaled_matrices(ctx, n, p):
    _check(ctx, _random(n, n) * 2.0 ** p, 2.0 ** p)


@pytest.mark.parametrize("n", [5, 70, 300, 600])
@pytest.mark.parametrize("first,rest", [(95, 850), (0, 1000), (-100, 1000), (-9, 1010), (100, 1010), (95, 700)])
def test_small_column_before_a_large_matrix(ctx, n, first, rest):
    p = np.where(np.minimum.outer(np.arange(n), np.arange(n)) == 0, float(first), float(rest))
    _check(ctx, _random(n, n + 1) * 2.0 ** p, 2.0 ** rest)


@pytest.mark.parametrize("n", [70, 300])
def test_columns_cross_the_scaling_limits(ctx, n):
    p = 300.0 - 40.0 * np.minimum(np.minimum.outer(np.arange(n), np.arange(n)), 20)
    _check(ctx, _random(n, n + 2) * 2.0 ** p, 2.0 ** 300)
