"""Lanczos where the tridiagonal solve stops running beside the next product
(2^20 entries): six steps just below, at and above, host loop and step graph,
against the oracle's Krylov space of the same size, and a solve that converges
(its last product beside the solve is discarded). Bars as for the shorter
vectors: 1e-12 ||H|| on the Ritz value, ||H|| bounded by the first residual and
energy, 1e-10 on the vector."""
import numpy as np
import pytest

from oracle import dmrg as od
from paper_1703_00387_gb300 import binding as B
from paper_1703_00387_gb300 import hamiltonians, inputs

pytestmark = pytest.mark.gpu
SIZES = [(512, 511), (512, 512), (513, 512)]  # 2^20 - 2048, 2^20, 2^20 + 2048


def _problem(chi_l, chi_r):
    W = hamiltonians.ising(4, 1.0, 1.0)
    L, R = (inputs.random_symmetric_env(c, 3, seed=c) / np.sqrt(c) for c in (chi_l, chi_r))
    theta = np.random.default_rng(chi_l).standard_normal((chi_l, 2, 2, chi_r))
    return L, W[1], W[2], R, theta


@pytest.mark.parametrize("chi_l,chi_r", SIZES)
def test_six_steps(chi_l, chi_r):
    import torch
    ops = _problem(chi_l, chi_r)
    mv = lambda x: od.heff_apply(*ops[:4], x)  # noqa: E731
    e_ref, v_ref, m_ref, _ = od.lanczos_ground(mv, ops[4], 6, 0.0)
    assert m_ref == 6
    scale = np.linalg.norm(mv(ops[4] / np.linalg.norm(ops[4]))) + abs(e_ref)
    r = np.asarray(v_ref).ravel()
    for mode in ("host", "graph"):
        t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in ops]
        ctx = B.Context(0)
        ctx.set_lanczos_mode(mode)
        e, it, _, ok = B.osmps_lanczos_ground(ctx, *t, max_iter=6, tol=0.0, precision="fp64")
        assert it == 6 and not ok
        assert abs(e - e_ref) <= 1e-12 * scale
        v = t[4].cpu().numpy().ravel()
        assert abs(np.linalg.norm(v) - 1) <= 1e-13
        assert np.linalg.norm(v - r * np.sign(v @ r) / np.linalg.norm(r)) <= 1e-10
        ctx.close()


@pytest.mark.parametrize("chi_l,chi_r", SIZES)
def test_converged_solve_is_the_same_in_both_drivers(chi_l, chi_r):
    import torch
    ops = _problem(chi_l, chi_r)
    out = []
    tol = 0.0  # then the residual of ten steps, which the first step's is far above
    for mode in ("host", "host", "graph"):
        t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in ops]
        ctx = B.Context(0)
        ctx.set_lanczos_mode(mode)
        e, it, res, ok = B.osmps_lanczos_ground(ctx, *t, max_iter=10 if tol == 0.0 else 40, tol=tol,
                                                precision="fp64")
        ctx.close()
        if tol == 0.0:
            assert it == 10 and not ok and res > 0.0
            tol = res
            continue
        assert ok and 1 < it <= 10 and res <= tol
        out.append((e, it, res, t[4].clone()))
    assert out[0][:3] == out[1][:3] and torch.equal(out[0][3], out[1][3])
