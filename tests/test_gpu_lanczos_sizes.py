"""Lanczos at the vector lengths where the orthogonalisation changes its form:
one element or a pair per thread (2^15), partial sums added in the update or
apart (2^16), two passes always or on demand (2^18). Six steps (each solve of T
beside the next product, the last one alone) against the oracle's Krylov space
of the same size; the Ritz value is good to a few eps ||H|| (bar 1e-12 ||H||,
||H|| bounded by the first residual and energy), the vector to 1e-10."""
import numpy as np
import pytest

from oracle import dmrg as od
from paper_1703_00387_gb300 import binding as B
from paper_1703_00387_gb300 import hamiltonians, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["host", "graph"])
@pytest.mark.parametrize("chi_l,chi_r", [(91, 90), (92, 90), (127, 129), (129, 128), (256, 256), (257, 256)])
def test_lanczos_vector_lengths(chi_l, chi_r, mode):
    import torch
    W = hamiltonians.ising(4, 1.0, 1.0)
    L, R = (inputs.random_symmetric_env(c, 3, seed=c) / np.sqrt(c) for c in (chi_l, chi_r))
    theta = np.random.default_rng(chi_l).standard_normal((chi_l, 2, 2, chi_r))
    mv = lambda x: od.heff_apply(L, W[1], W[2], R, x)  # noqa: E731
    e_ref, v_ref, m_ref, _ = od.lanczos_ground(mv, theta, 6, 0.0)
    assert m_ref == 6
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (L, W[1], W[2], R, theta)]
    ctx = B.Context(0)
    ctx.set_lanczos_mode(mode)
    e, it, res, ok = B.osmps_lanczos_ground(ctx, *t, max_iter=6, tol=0.0, precision="fp64")
    assert it == 6 and not ok
    x = theta / np.linalg.norm(theta)
    scale = np.linalg.norm(mv(x)) + abs(e_ref)
    assert abs(e - e_ref) <= 1e-12 * scale
    v, r = t[4].cpu().numpy().ravel(), np.asarray(v_ref).ravel()
    assert abs(np.linalg.norm(v) - 1) <= 1e-13
    assert np.linalg.norm(v - r * np.sign(v @ r) / np.linalg.norm(r)) <= 1e-10
    ctx.close()
