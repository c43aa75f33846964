"""The float64 DMMA product at the edges of its 16x16 and 8x8 tiles and of the
K groups its four warps take in turn (groups of 4, rounds of 16), through theta
formation (row-major operands) and the float64 environment updates (transposed
and batched operands). Bar per entry: the rounding of a K-term sum,
(2 K + 4) eps |A| |B| with the reference's own; for the update, two sums and a W-step, applied norm-wise."""
import numpy as np
import pytest

from paper_1703_00387_gb300 import binding as B
from paper_1703_00387_gb300 import inputs

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("K", [1, 3, 4, 15, 16, 17, 65, 128])
@pytest.mark.parametrize("M,N", [(1, 1), (7, 9), (16, 8), (17, 15), (129, 33), (400, 410), (1030, 515)])
def test_theta_form_tile_edges(ctx, M, N, K):
    import torch
    rng = np.random.default_rng(M + 3 * N + 7 * K)
    a, b = rng.standard_normal((M, 1, K)), rng.standard_normal((K, 1, N))
    out = torch.full((M, 1, 1, N), float("nan"), dtype=torch.float64, device="cuda:0")
    B.osmps_theta_form(ctx, torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), out)
    got = out.cpu().numpy().reshape(M, N)
    ref = a[:, 0, :] @ b[:, 0, :]
    bar = (2 * K + 4) * EPS * (np.abs(a[:, 0, :]) @ np.abs(b[:, 0, :]))
    assert np.all(np.abs(got - ref) <= bar)


@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("chi_l,d,chi_r,w_in,w_out", [(1, 2, 3, 1, 5), (15, 2, 17, 3, 4), (33, 3, 31, 5, 5),
                                                      (130, 2, 100, 5, 5)])
def test_env_update_fp64_edges(ctx, side, chi_l, d, chi_r, w_in, w_out):
    import torch

    from oracle import dmrg as odmrg
    env, A, W = inputs.random_env_operands(chi_l, d, chi_r, w_in, w_out, side, seed=chi_l + side)
    n = chi_r if side == 0 else chi_l
    out = torch.full((n, w_out, n), float("nan"), dtype=torch.float64, device="cuda:0")
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (env, A, W)]
    B.osmps_env_update(ctx, side, *t, out, precision="fp64")
    ref = odmrg.env_left(env, A, W) if side == 0 else odmrg.env_right(env, A, W)
    err = np.linalg.norm(out.cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err <= 4 * (chi_l + chi_r + d * max(w_in, w_out)) * EPS
