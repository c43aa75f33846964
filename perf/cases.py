"""The calls that a variational search, a quench or a gradient run spends its
time in, with the sizes they meet: what is timed when a kernel or the host
path under it changes.

Most cases are one call of the C ABI through ``binding`` (one product, one
environment update, one local eigenproblem, one split); two are whole calls:
the small ground-state job, from host tensors to the final state, and the
two-site update (theta, Lanczos, split) at the benchmark's bond dimension.

Inputs are drawn on the GPU from the seed alone. Environments are built from
random canonical site tensors and the model's MPO by plain torch contractions,
from the chain's end inwards, so they carry the identity channel, the
Hermitian structure and the scale that a sweep's environments carry.

The sign of a Ritz vector is free and is kept on the start vector's side.
Site tensors after a split are fixed up to a sign per kept state (and, inside
a nearly degenerate tail, a rotation), so what is returned of a split is the
spectrum and the two-site tensor that the two sites form again
(``osmps_theta_form``, which is also the next call of a sweep that turns
round); of a whole sweep it is the energies and the state vector.
"""
import math

import numpy as np
import torch

from paper_1703_00387_gb300 import binding as B
from paper_1703_00387_gb300 import hamiltonians
from paper_1703_00387_gb300 import inputs
from paper_1703_00387_gb300 import u1

DEV = "cuda:0"
_CTX = None


def _context():
    """The one context (workspace, graphs, tile widths) a program keeps."""
    global _CTX
    if _CTX is None:
        _CTX = B.Context(0)
    return _CTX


def listed():
    return [
        # The smallest call: one float64 product at the bond dimension of the
        # small Ising run (chi = 32, w = 3). Launches and latency only.
        dict(name="heff_fp64_tfi_chi32", kind="heff", model="ising", chi_l=32, chi_r=32, precision="fp64"),
        # The benchmark's product: spin-1/2 XXZ at chi = 1024 in split bf16,
        # operands converted in the call as a caller without a solver pays.
        dict(name="heff_bf16x3_xxz_chi1024", kind="heff", model="xxz", chi_l=1024, chi_r=1024, precision="bf16x3"),
        # Odd bond dimensions, d = 3, w = 14 (AKLT chain), split tf32: neither
        # the fused W-step nor any tile or vector width divides the sizes.
        dict(name="heff_tf32x3_aklt_301x257", kind="heff", model="aklt", chi_l=301, chi_r=257, precision="tf32x3"),
        # Environment growth of a left-to-right half sweep at the benchmark's size.
        dict(name="env_left_bf16x3_xxz_chi1024", kind="env", model="xxz", side=0, chi_l=1024, chi_r=1024,
             precision="bf16x3"),
        # Right-to-left growth in a refinement sweep, ragged bonds.
        dict(name="env_right_fp64emu_xxz_381x500", kind="env", model="xxz", side=1, chi_l=381, chi_r=500,
             precision="fp64emu"),
        # The local eigenproblem of a refinement sweep: float64-accurate
        # products, one Krylov space of the benchmark's 20 vectors.
        dict(name="lanczos_fp64emu_xxz_chi512", kind="lanczos", model="xxz", chi_l=512, chi_r=512, max_iter=20,
             precision="fp64emu"),
        # The local eigenproblem of a small chain run: launch- and
        # latency-bound steps (the recorded step graph).
        dict(name="lanczos_bf16x3_xxz_chi64", kind="lanczos", model="xxz", chi_l=64, chi_r=64, max_iter=20,
             precision="bf16x3"),
        # Truncating split of a converged two-site tensor (steep spectrum, cut
        # by the local tolerance), ragged sides, at the batch runs' sizes.
        dict(name="split_decay_150x170", kind="split", chi_l=150, d=2, chi_r=170, chi_max=256, eps_local=1e-10,
             decay=1.0, move_right=1, precision="bf16x3"),
        # The benchmark's two-site update: theta, 20 Lanczos steps in bf16x3,
        # the float64 split to chi_max = 1024.
        dict(name="update_bf16x3_xxz_chi1024", kind="update", model="xxz", chi=1024, max_iter=20,
             precision="bf16x3"),
        # U(1) block-sparse local eigenproblem: Bose-Hubbard, n <= 4, chi = 512
        # in 13 sectors, the middle of a 64-site chain at unit filling.
        dict(name="u1_lanczos_bh_chi512", kind="u1", chi=512, nmax=4, width=8.0, max_iter=20, precision="bf16x3"),
        # Krylov propagator of one TDVP pair, complex tensors.
        dict(name="expm_bf16x3_xxz_chi128", kind="expm", model="xxz", chi_l=128, chi_r=128, tau=0.025,
             precision="bf16x3"),
        # The small ground-state job: Ising L = 12, chi_max = 32, 4 float64
        # sweeps, host tensors in, final state out.
        dict(name="sweep_fp64_tfi_L12_chi32", kind="sweep", L=12, chi=32, n_sweeps=4, g=1.0, precision="fp64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["heff", "heff", "env", "env", "lanczos", "lanczos", "split", "split", "split", "update",
                       "u1", "expm", "sweep"])
    if kind in ("heff", "env", "lanczos"):
        model = rng.choice(["ising", "xxz", "xxz", "aklt"])
        precision = rng.choice(["fp64", "bf16x3", "bf16x3", "tf32x3", "fp64emu"])
        top = {"fp64": 300, "fp64emu": 512, "tf32x3": 768, "bf16x3": 1024}[precision]
        if model == "aklt":
            top = min(top, 400)
        if kind == "lanczos":
            top = min(top, 640 if precision == "bf16x3" else 256)
        chi_l = _log(rng, 16, top)
        chi_r = max(16, min(top, int(round(chi_l * rng.uniform(0.7, 1.4)))))
        c = dict(kind=kind, model=model, chi_l=chi_l, chi_r=chi_r, precision=precision)
        if kind == "env":
            c["side"] = rng.randrange(2)
        if kind == "lanczos":
            c["max_iter"] = rng.randint(8, 20)
        return c
    if kind == "split":
        chi_l = _log(rng, 12, 700)
        chi_r = max(12, min(700, int(round(chi_l * rng.uniform(0.7, 1.4)))))
        decay = rng.choice([0.0, 0.5, 1.0])
        return dict(kind="split", chi_l=chi_l, d=rng.choice([2, 2, 3]) if chi_l < 400 else 2, chi_r=chi_r,
                    chi_max=max(8, min(chi_l, chi_r)), eps_local=rng.choice([0.0, 1e-10]) if decay else 0.0,
                    decay=decay, move_right=rng.randrange(2), precision=rng.choice(["fp64", "bf16x3"]))
    if kind == "update":
        return dict(kind="update", model=rng.choice(["ising", "xxz"]), chi=_log(rng, 48, 768),
                    max_iter=rng.randint(8, 20), precision=rng.choice(["bf16x3", "tf32x3"]))
    if kind == "u1":
        return dict(kind="u1", chi=_log(rng, 64, 512), nmax=rng.choice([2, 3, 4]), width=rng.uniform(4.0, 10.0),
                    max_iter=rng.randint(8, 20), precision=rng.choice(["bf16x3", "tf32x3"]))
    if kind == "expm":
        chi_l = _log(rng, 16, 128)
        return dict(kind="expm", model="xxz", chi_l=chi_l, chi_r=max(16, min(128, int(chi_l * rng.uniform(0.8, 1.25)))),
                    tau=rng.choice([0.025, -0.025, 0.05]), precision=rng.choice(["bf16x3", "fp64emu"]))
    L = rng.randint(8, 12)
    return dict(kind="sweep", L=L, chi=rng.randint(8, 32), n_sweeps=rng.randint(3, 4), g=round(rng.uniform(0.5, 1.5), 3),
                precision="fp64")


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1009 + salt)
    return g


def _normal(g, *shape, dtype=torch.float64):
    return torch.randn(*shape, generator=g, dtype=dtype, device=DEV)


def _model(name):
    """(d, w, the MPO's first, bulk and last site tensors) of a uniform chain."""
    W = {"ising": lambda: hamiltonians.ising(4, 1.0, 1.0), "xxz": lambda: hamiltonians.xxz(4, 1.0, 1.0, 0.0),
         "aklt": lambda: hamiltonians.aklt(4)}[name]()
    first, bulk, last = (torch.from_numpy(np.ascontiguousarray(W[i])).to(DEV) for i in (0, 1, 3))
    return bulk.shape[1], bulk.shape[0], first, bulk, last


def _isometry(g, rows, cols, dtype):
    """rows x cols with orthonormal columns (rows >= cols)."""
    return torch.linalg.qr(_normal(g, rows, cols, dtype=dtype))[0].contiguous()


def _left_site(g, a, d, b, dtype):
    return _isometry(g, a * d, b, dtype).reshape(a, d, b)


def _right_site(g, a, d, b, dtype):
    return _isometry(g, d * b, a, dtype).mT.reshape(a, d, b).contiguous()


def _grow_left(E, A, W):
    a, d, b = A.shape
    w, w2 = W.shape[0], W.shape[3]
    W = W.to(A.dtype)
    X = (E.reshape(-1, a) @ A.reshape(a, d * b)).reshape(a, w, d, b)
    Y = torch.einsum("awsb,wtsv->atvb", X, W).reshape(a * d, w2 * b)
    return (A.reshape(a * d, b).mH @ Y).reshape(b, w2, b)


def _grow_right(E, A, W):
    a, d, b = A.shape
    w, w2 = W.shape[0], W.shape[3]
    W = W.to(A.dtype)
    X = torch.einsum("asb,cvb->asvc", A, E)
    Y = torch.einsum("asvc,wtsv->awtc", X, W).reshape(a, w, d * b)
    return torch.einsum("ek,awk->ewa", A.conj().reshape(a, d * b), Y)


def _dims(chi, d):
    out = [1]
    while out[-1] < chi:
        out.append(min(out[-1] * d, chi))
    return out


def _left_env(g, chi, model, dtype=torch.float64):
    d, w, first, bulk, _ = _model(model)
    E = torch.ones(1, 1, 1, dtype=dtype, device=DEV)
    dims = _dims(chi, d)
    for i in range(len(dims) - 1):
        E = _grow_left(E, _left_site(g, dims[i], d, dims[i + 1], dtype), first if i == 0 else bulk)
    return E.contiguous()


def _right_env(g, chi, model, dtype=torch.float64):
    d, w, _, bulk, last = _model(model)
    E = torch.ones(1, 1, 1, dtype=dtype, device=DEV)
    dims = _dims(chi, d)
    for i in range(len(dims) - 1):
        E = _grow_right(E, _right_site(g, dims[i + 1], d, dims[i], dtype), last if i == 0 else bulk)
    return E.contiguous()


def _unit(x):
    return (x / torch.linalg.vector_norm(x)).contiguous()


def _u1_masks(case):
    """Charges and allowed entries of the middle pair of the Bose-Hubbard chain."""
    left = inputs.u1_sector_profile(31.0, total=case["chi"], width=case["width"])
    right = inputs.u1_sector_profile(33.0, total=case["chi"], width=case["width"])
    qa, qc = (torch.from_numpy(np.repeat(np.asarray(q), np.asarray(c))).to(DEV) for q, c in (left, right))
    d = case["nmax"] + 1
    s = torch.arange(d, device=DEV)
    qw = torch.tensor([0, 1, -1, 0], device=DEV)  # done, -J b^dag, -J b, start
    m_theta = (qa[:, None, None, None] + s[None, :, None, None] + s[None, None, :, None]) == qc[None, None, None, :]
    m_L = qa[:, None, None] == qa[None, None, :] + qw[None, :, None]
    m_R = qc[:, None, None] == qc[None, None, :] + qw[None, :, None]
    return left, right, m_theta, m_L, m_R


def _u1_dense(case, seed):
    left, right, m_theta, m_L, m_R = _u1_masks(case)
    g = _gen(seed, 7)
    chi = case["chi"]

    def env(mask, unit):
        E = torch.zeros(mask.shape, dtype=torch.float64, device=DEV)
        h = _normal(g, chi, chi) / math.sqrt(chi)
        E[:, 3 - unit, :] = h + h.mT
        E[:, 1, :] = _normal(g, chi, chi) / math.sqrt(chi)
        E[:, unit, :] = torch.eye(chi, dtype=torch.float64, device=DEV)
        E = torch.where(mask, E, torch.zeros((), dtype=torch.float64, device=DEV))
        E[:, 2, :] = E[:, 1, :].mT
        return E.contiguous()

    L, R = env(m_L, 3), env(m_R, 0)
    theta = _unit(torch.where(m_theta, _normal(g, *m_theta.shape), torch.zeros((), dtype=torch.float64, device=DEV)))
    W = hamiltonians.bose_hubbard(4, 1.0, 4.0, case["nmax"])
    W1, W2 = (torch.from_numpy(np.ascontiguousarray(W[i])).to(DEV) for i in (1, 2))
    return left, right, m_theta, m_L, m_R, L, W1, W2, R, theta


def _split_theta(case, seed):
    """A two-site tensor whose singular values fall off as exp(-decay * 2 ln^2(1 + i))
    or so: a Gaussian matrix with graded rows and columns."""
    g = _gen(seed, 5)
    rows, cols = case["chi_l"] * case["d"], case["d"] * case["chi_r"]
    M = _normal(g, rows, cols)
    if case["decay"]:
        for n, shape in ((rows, (rows, 1)), (cols, (1, cols))):
            i = torch.arange(n, dtype=torch.float64, device=DEV)
            f = torch.exp(-case["decay"] * 0.25 * torch.log1p(i) ** 2)
            M = M * f[torch.randperm(n, generator=g, device=DEV)].reshape(shape)
    return _unit(M.reshape(case["chi_l"], case["d"], case["d"], case["chi_r"]))


def prepare(case, seed):
    ctx = _context()
    kind = case["kind"]
    s = dict(case=case, ctx=ctx, kind=kind)
    if kind in ("heff", "lanczos", "expm"):
        dtype = torch.complex128 if kind == "expm" else torch.float64
        g = _gen(seed, 1)
        d, w, _, bulk, _ = _model(case["model"])
        s["L"] = _left_env(g, case["chi_l"], case["model"], dtype)
        s["R"] = _right_env(g, case["chi_r"], case["model"], dtype)
        s["W1"], s["W2"] = bulk.contiguous(), bulk.clone()
        s["start"] = _unit(_normal(g, case["chi_l"], d, d, case["chi_r"], dtype=dtype))
        s["theta"] = torch.empty_like(s["start"])
    elif kind == "env":
        g = _gen(seed, 2)
        d, w, _, bulk, _ = _model(case["model"])
        a, b = case["chi_l"], case["chi_r"]
        s["W"] = bulk.contiguous()
        if case["side"] == 0:
            s["env"] = _left_env(g, a, case["model"])
            s["A"] = _left_site(g, a, d, b, torch.float64) if a * d >= b else _unit(_normal(g, a, d, b))
            s["out"] = torch.empty(b, w, b, dtype=torch.float64, device=DEV)
        else:
            s["env"] = _right_env(g, b, case["model"])
            s["A"] = _right_site(g, a, d, b, torch.float64) if d * b >= a else _unit(_normal(g, a, d, b))
            s["out"] = torch.empty(a, w, a, dtype=torch.float64, device=DEV)
    elif kind == "split":
        s["theta"] = _split_theta(case, seed)
    elif kind == "update":
        g = _gen(seed, 3)
        d, w, _, bulk, _ = _model(case["model"])
        chi = case["chi"]
        s["L"] = _left_env(g, chi, case["model"])
        s["R"] = _right_env(g, chi, case["model"])
        s["W1"], s["W2"] = bulk.contiguous(), bulk.clone()
        s["A1"], s["A2"] = _left_site(g, chi, d, chi, torch.float64), _unit(_normal(g, chi, d, chi))
        s["start"], s["theta"] = (torch.empty(chi, d, d, chi, dtype=torch.float64, device=DEV) for _ in range(2))
    elif kind == "u1":
        left, right, m_theta, m_L, m_R, L, W1, W2, R, theta = _u1_dense(case, seed)
        W = hamiltonians.bose_hubbard(4, 1.0, 4.0, case["nmax"])
        q = u1.channel_charges(W)
        d = case["nmax"] + 1
        s["plan"] = B.U1Heff(ctx, left[0], left[1], right[0], right[1], d, d, 4, 4, 4, q[1], q[3])
        s["W1"], s["W2"] = W1, W2
        s["L"], s["R"], s["start"] = L[m_L].contiguous(), R[m_R].contiguous(), theta[m_theta].contiguous()
        s["theta"] = torch.empty_like(s["start"])
    elif kind == "sweep":
        s["mpo"] = B.MPO(ctx, hamiltonians.ising(case["L"], 1.0, case["g"]))
        s["tensors"] = inputs.random_mps(case["L"], 2, case["chi"], seed=int(seed))
        s["params"] = B.sweep_params(case["chi"], n_sweeps=case["n_sweeps"], precision=case["precision"],
                                     lanczos_tol=1e-12)
    if kind in ("split", "update"):
        if kind == "update":
            chi_l = chi_r = chi_max = case["chi"]
            d = s["W1"].shape[1]
        else:
            chi_l, d, chi_r, chi_max = case["chi_l"], case["d"], case["chi_r"], case["chi_max"]
        cap = min(chi_max, chi_l * d, d * chi_r)
        s["B1"] = torch.empty(chi_l * d * cap, dtype=torch.float64, device=DEV)
        s["B2"] = torch.empty(cap * d * chi_r, dtype=torch.float64, device=DEV)
        s["again"] = torch.empty(chi_l, d, d, chi_r, dtype=torch.float64, device=DEV)
        s["cap"] = cap
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _split(s, theta, move_right, chi_max, eps_local, precision):
    chi_l, d, _, chi_r = theta.shape
    keep, discarded, entropy, lam2 = B.osmps_split(s["ctx"], theta, s["B1"], s["B2"], move_right, chi_max, eps_local,
                                                   precision=precision)
    A1 = s["B1"][:chi_l * d * keep].view(chi_l, d, keep)
    A2 = s["B2"][:keep * d * chi_r].view(keep, d, chi_r)
    B.osmps_theta_form(s["ctx"], A1, A2, s["again"])
    return dict(keep=keep, numbers=np.array([entropy, 1.0 - discarded]), lam2=lam2, theta=s["again"])


def _vector(tensors):
    """The state vector; its sign is free, and the Ising ground state can be
    taken positive."""
    v = np.ones((1, 1))
    for A in tensors:
        v = (v @ A.reshape(A.shape[0], -1)).reshape(-1, A.shape[2])
    return v.reshape(-1) * np.sign(v.sum())


def _same_side(theta, start):
    """An eigenvector's sign is free: keep it on the start vector's side, as a
    program that follows a state does."""
    return theta.mul_(torch.sign(torch.dot(theta.reshape(-1), start.reshape(-1))))


def run(s):
    case, ctx, kind = s["case"], s["ctx"], s["kind"]
    if kind == "heff":
        B.osmps_heff_apply(ctx, s["L"], s["W1"], s["W2"], s["R"], s["start"], s["theta"], precision=case["precision"])
        return s["theta"]
    if kind == "env":
        return B.osmps_env_update(ctx, case["side"], s["env"], s["A"], s["W"], s["out"], precision=case["precision"])
    if kind == "lanczos":
        s["theta"].copy_(s["start"])
        e, _, _, _ = B.osmps_lanczos_ground(ctx, s["L"], s["W1"], s["W2"], s["R"], s["theta"],
                                            max_iter=case["max_iter"], tol=1e-10, precision=case["precision"])
        return dict(energy=np.array([e]), theta=_same_side(s["theta"], s["start"]))
    if kind == "split":
        return _split(s, s["theta"], case["move_right"], case["chi_max"], case["eps_local"], case["precision"])
    if kind == "update":
        B.osmps_theta_form(ctx, s["A1"], s["A2"], s["start"])
        s["theta"].copy_(s["start"])
        e, _, _, _ = B.osmps_lanczos_ground(ctx, s["L"], s["W1"], s["W2"], s["R"], s["theta"],
                                            max_iter=case["max_iter"], tol=1e-10, precision=case["precision"])
        out = _split(s, _same_side(s["theta"], s["start"]), 1, case["chi"], 0.0, case["precision"])
        out["energy"], out["ritz"] = np.array([e]), s["theta"]
        return out
    if kind == "u1":
        s["theta"].copy_(s["start"])
        e, _, _, _ = B.osmps_lanczos_ground_u1(ctx, s["plan"], s["L"], s["W1"], s["W2"], s["R"], s["theta"],
                                               max_iter=case["max_iter"], tol=1e-10, precision=case["precision"])
        return dict(energy=np.array([e]), theta=_same_side(s["theta"], s["start"]))
    if kind == "expm":
        s["theta"].copy_(s["start"])
        B.osmps_heff_expm(ctx, s["L"], s["W1"], s["W2"], s["R"], s["theta"], case["tau"], max_iter=40, tol=1e-12,
                          precision=case["precision"])
        return s["theta"]
    mps = B.MPS(ctx, s["tensors"], case["chi"])
    st = B.osmps_sweep(ctx, mps, s["mpo"], s["params"])
    tensors = mps.tensors()
    mps.close()
    return dict(energy=np.array([st["energy"]]), entropy=np.array([st["entropy_center"]]), steps=st["step_energies"],
                state=_vector(tensors))


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _heff_work(chi_l, chi_r, d, w):
    n = chi_l * d * d * chi_r
    flops = 2.0 * n * w * (chi_l + chi_r) + 4.0 * n * d * w * w
    return 8.0 * (w * (chi_l ** 2 + chi_r ** 2) + 2 * n), flops, n


def _split_work(rows, cols, keep):
    n = min(rows, cols)
    return 8.0 * (2 * rows * cols + keep * (rows + cols)), 2.0 * rows * cols * n + 4.0 / 3 * n ** 3 \
        + 2.0 * n * n * keep + 4.0 * rows * cols * keep


def work(case):
    kind = case["kind"]
    dw = {"ising": (2, 3), "xxz": (2, 5), "aklt": (3, 14)}
    if kind in ("heff", "lanczos"):
        d, w = dw[case["model"]]
        b, f, _ = _heff_work(case["chi_l"], case["chi_r"], d, w)
        return dict(bytes=b, flops=f * case.get("max_iter", 1))
    if kind == "env":
        d, w = dw[case["model"]]
        a, b = case["chi_l"], case["chi_r"]
        return dict(bytes=8.0 * (w * (a * a + b * b) + a * d * b), flops=2.0 * a * b * d * w * (a + b))
    if kind == "split":
        rows, cols = case["chi_l"] * case["d"], case["d"] * case["chi_r"]
        b, f = _split_work(rows, cols, min(case["chi_max"], rows, cols))
        return dict(bytes=b, flops=f)
    if kind == "update":
        d, w = dw[case["model"]]
        chi = case["chi"]
        b, f, n = _heff_work(chi, chi, d, w)
        b2, f2 = _split_work(chi * d, d * chi, chi)
        return dict(bytes=b + b2, flops=f * case["max_iter"] + f2 + 2.0 * n * chi)
    if kind == "u1":
        d, chi = case["nmax"] + 1, case["chi"]
        sizes = inputs.u1_sector_profile(31.0, total=chi, width=case["width"])[1].astype(float)
        share = float((sizes ** 2).sum()) / chi ** 2  # of a dense bond matrix
        b, f, _ = _heff_work(chi, chi, d, 4)
        return dict(bytes=b * share, flops=f * share * share * case["max_iter"])
    if kind == "expm":
        d, w = dw[case["model"]]
        b, f, _ = _heff_work(case["chi_l"], case["chi_r"], d, w)
        return dict(bytes=2 * b, flops=4 * f * 6)  # complex; about six Krylov vectors
    n, f = 2 * (case["L"] - 1) * case["n_sweeps"], 0.0
    for k in range(1, case["L"]):
        a, b = (min(2 ** (k - 1), 2 ** (case["L"] - k + 1), case["chi"]), min(2 ** (k + 1), 2 ** (case["L"] - k - 1), case["chi"]))
        f += 2 * case["n_sweeps"] * 8 * _heff_work(a, max(b, 1), 2, 3)[1]
    return dict(bytes=8.0 * n * 4 * case["chi"] ** 2, flops=f)


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch and numpy
# ---------------------------------------------------------------------------
def _apply(L, W1, W2, R, x):
    a, d1, d2, c = x.shape
    W1, W2 = W1.to(x.dtype), W2.to(x.dtype)
    T = (L.reshape(-1, L.shape[2]) @ x.reshape(a, -1)).reshape(L.shape[0], L.shape[1], d1, d2, c)
    T = torch.einsum("awspc,wtsv->atvpc", T, W1)
    T = torch.einsum("atvpc,vupx->atuxc", T, W2).reshape(a * d1 * d2, -1)
    return (T @ R.reshape(R.shape[0], -1).mT).reshape(a, d1, d2, c)


def _krylov(apply, x, m):
    """Krylov basis of m vectors and the projected (tridiagonal) matrix."""
    V, T = [x / torch.linalg.vector_norm(x)], np.zeros((m, m))
    for j in range(m):
        w = apply(V[j])
        Q = torch.stack([v.reshape(-1) for v in V])
        for _ in range(2):
            c = Q.conj() @ w.reshape(-1)
            w = w - (c @ Q).reshape(w.shape)
            T[j, j] += c[j].real.item()
        beta = torch.linalg.vector_norm(w).item()
        if j + 1 < m:
            T[j, j + 1] = T[j + 1, j] = beta
            V.append(w / beta)
    return torch.stack([v.reshape(-1) for v in V]), T, beta


def _ground(apply, x, m):
    Q, T, _ = _krylov(apply, x, m)
    e, z = np.linalg.eigh(T)
    z = z[:, 0] * np.sign(z[0, 0])  # on the start vector's side, as run() leaves it
    y = torch.from_numpy(z).to(Q) @ Q
    return e[0], (y / torch.linalg.vector_norm(y)).reshape(x.shape)


def _truncated(theta, chi_max, eps_local):
    a, d1, d2, c = theta.shape
    U, S, V = torch.linalg.svd(theta.reshape(a * d1, d2 * c), full_matrices=False)
    p = (S ** 2 / (S ** 2).sum()).cpu().numpy()
    keep = 1
    while keep < min(chi_max, len(p)) and p[keep:].sum() > eps_local:
        keep += 1
    kept = p[:keep].sum()
    M = (U[:, :keep] * S[:keep]) @ V[:keep]
    lam2 = np.zeros(min(a * d1, d2 * c))
    nev = min(chi_max, len(p))
    lam2[:nev] = p[:nev]
    q = p[:keep] / kept
    q = q[q > 0]
    return dict(keep=None, numbers=np.array([float(-(q * np.log(q)).sum()), float(kept)]), lam2=lam2,
                theta=(M / torch.linalg.vector_norm(M)).reshape(theta.shape))


def exact(case, seed):
    kind = case["kind"]
    if kind == "u1":
        left, right, m_theta, m_L, m_R, L, W1, W2, R, theta = _u1_dense(case, seed)
        e, y = _ground(lambda x: _apply(L, W1, W2, R, x), theta, case["max_iter"])
        return dict(energy=np.array([e]), theta=y[m_theta])
    if kind == "sweep":
        W = hamiltonians.ising(case["L"], 1.0, case["g"])
        if case["chi"] < 24 or case["n_sweeps"] < 4:
            return None  # truncated or not yet converged: not the exact ground state
        H = W[0][0]  # (t, s, w)
        for k in range(1, case["L"]):
            H = np.einsum("tsw,wpqv->tpsqv", H, W[k]).reshape(H.shape[0] * 2, H.shape[1] * 2, -1)
        e = torch.linalg.eigvalsh(torch.from_numpy(np.ascontiguousarray(H[:, :, 0])).to(DEV))[0].item()
        return dict(energy=np.array([e]), entropy=None, steps=None, state=None)
    s = prepare(case, seed)
    if kind == "heff":
        return _apply(s["L"], s["W1"], s["W2"], s["R"], s["start"])
    if kind == "env":
        return (_grow_left if case["side"] == 0 else _grow_right)(s["env"], s["A"], s["W"])
    if kind == "split":
        return _truncated(s["theta"], case["chi_max"], case["eps_local"])
    op = lambda x: _apply(s["L"], s["W1"], s["W2"], s["R"], x)  # noqa: E731
    if kind == "lanczos":
        e, y = _ground(op, s["start"], case["max_iter"])
        return dict(energy=np.array([e]), theta=y)
    if kind == "update":
        a, d, m = s["A1"].shape
        x = (s["A1"].reshape(a * d, m) @ s["A2"].reshape(m, -1)).reshape(a, d, d, m)
        e, y = _ground(op, x, case["max_iter"])
        out = _truncated(y, case["chi"], 0.0)
        out["energy"], out["ritz"] = np.array([e]), y
        return out
    if kind == "expm":
        Q, T, _ = _krylov(op, s["start"], 14)
        lam, z = np.linalg.eigh(T)
        u = (z * np.exp(-1j * case["tau"] * lam)) @ z[0]
        return (torch.from_numpy(u).to(Q) @ Q).reshape(s["start"].shape)
    return None
