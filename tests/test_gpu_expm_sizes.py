"""The propagator at the vector length where the orthogonalisation changes its
form (2^18 entries of the embedded vector): against the oracle's Krylov space,
and projected twice in every step on both sides of it. Below it two projections
and the norm are seven launches, beyond it nine (twice three and two for the
norm, one for alpha and beta); deciding whether to project again would add a norm
and the decision.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import tdvp as T
from paper_1703_00387_gb300 import binding as B
from paper_1703_00387_gb300 import hamiltonians

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    c.close()


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _operator(chi_l, chi_r):
    W = hamiltonians.ising(4, 1.0, 1.0)
    rng = np.random.default_rng(chi_l)

    def env(chi):
        E = rng.standard_normal((chi, 3, chi)) + 1j * rng.standard_normal((chi, 3, chi))
        return (E + E.conj().transpose(2, 1, 0)) / np.sqrt(8 * chi)

    theta = rng.standard_normal((chi_l, 2, 2, chi_r)) + 1j * rng.standard_normal((chi_l, 2, 2, chi_r))
    return env(chi_l), W[1], W[2], env(chi_r), theta


SIZES = [(128, 128), (130, 130)]  # 2^18 and 2^18 + 8256 entries


@pytest.mark.parametrize("chi_l,chi_r", SIZES)
def test_matches_oracle(ctx, chi_l, chi_r):
    L, W1, W2, R, theta = _operator(chi_l, chi_r)
    ref, m_ref, _ = T.krylov_expm(lambda x: T.heff2_apply(L, W1, W2, R, x), theta, 0.2, max_iter=40, tol=1e-12)
    th = dev(theta)
    m, _, ok = B.osmps_heff_expm(ctx, dev(L), dev(W1), dev(W2), dev(R), th, 0.2, max_iter=40, tol=1e-12,
                                 precision="fp64")
    assert ok and abs(m - m_ref) <= 1 and m >= 8
    assert np.linalg.norm(th.cpu().numpy() - ref) <= 1e-11 * np.linalg.norm(ref)


def test_two_projections_in_every_step(ctx):
    per_step = []
    for chi_l, chi_r in SIZES:
        L, W1, W2, R, theta = _operator(chi_l, chi_r)
        ops = [dev(x) for x in (L, W1, W2, R)]
        counts = []
        for cap in (2, 2, 6):  # the first run sizes the workspaces
            th = dev(theta)
            n0 = B.osmps_kernel_launches()
            m, _, ok = B.osmps_heff_expm(ctx, *ops, th, 3.0, max_iter=cap, tol=0.0, precision="fp64")
            counts.append(B.osmps_kernel_launches() - n0)
            assert m == cap and not ok
        per_step.append((counts[2] - counts[1]) / 4)
    assert per_step[1] <= per_step[0] + 2
