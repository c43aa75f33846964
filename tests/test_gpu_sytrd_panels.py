"""The Householder panel reduction where its launches change: one row, edges of
32-column panels and of the rows per block, the block counts whose sums take
one or two exchanges (trailing sizes 256, 544), rows kept in shared memory or
read from L2 (from about 1650 trailing rows on), odd sizes and addresses there;
columns with nothing below the subdiagonal. Bar: the backward error of an
n-step orthogonal reduction, n eps ||A||, on the eigenvalues of T."""
import numpy as np
import pytest

from paper_1703_00387_gb300 import binding as B

pytestmark = pytest.mark.gpu


def _reduce(ctx, S, offset=0):
    import torch
    n = S.shape[0]
    buf = torch.empty(n * n + 1, dtype=torch.float64, device="cuda:0")
    A = buf[offset:offset + n * n].view(n, n)
    A.copy_(torch.from_numpy(S))
    d, tau = (torch.full((n,), float("nan"), dtype=torch.float64, device="cuda:0") for _ in range(2))
    e = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda:0")
    B.osmps_sytrd(ctx, A, d, e, tau)
    d, e = d.cpu().numpy(), e.cpu().numpy()[:n - 1]
    return np.diag(d) + np.diag(e, 1) + np.diag(e, -1)


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n,offset", [(2, 0), (31, 0), (32, 1), (33, 0), (65, 0), (257, 1), (289, 0), (545, 0),
                                      (577, 1), (1800, 0), (1801, 0), (1800, 1)])
def test_panel_sizes(ctx, n, offset):
    rng = np.random.default_rng(n)
    M = rng.standard_normal((n, n)) * np.exp(-np.arange(n) / (0.2 * n))  # graded columns
    S = M @ M.T if n < 600 else M + M.T
    S = 0.5 * (S + S.T)
    w = np.linalg.eigvalsh(S)
    got = np.linalg.eigvalsh(_reduce(ctx, S, offset))
    assert np.abs(got - w).max() <= n * np.finfo(float).eps * np.abs(w).max()


@pytest.mark.parametrize("kind", ["identity", "zero", "tridiagonal", "blocks", "tiny"])
def test_columns_without_a_reflector(ctx, kind):
    n = 70
    rng = np.random.default_rng(3)
    S = {"identity": np.eye(n), "zero": np.zeros((n, n)),
         "tridiagonal": np.diag(rng.standard_normal(n)) + np.diag(np.ones(n - 1), 1) + np.diag(np.ones(n - 1), -1),
         "blocks": np.kron(np.eye(2), np.ones((35, 35))), "tiny": 1e-150 * np.ones((n, n))}[kind]
    w = np.linalg.eigvalsh(S)
    got = np.linalg.eigvalsh(_reduce(ctx, S))
    assert np.abs(got - w).max() <= n * np.finfo(float).eps * max(np.abs(w).max(), 1e-300)
