"""The work a Newton time step has this library do, as measurable cases.

One Newton correction assembles the residual and the Jacobian on the device
(``FSIAssembler``), hands the new values to the solver context and rebuilds the
preconditioner (``update_values``, ``precond_build``), and solves (``solve``).  The
learned stage adds its correction (``learned_apply``) and its training step
(``Trainer``).  Each case is one of these calls on a seeded system of the input
generator; inputs are made on the host or the device from the seed alone and are
resident on the GPU before the call.

Case fields: ``kind``; ``dim`` and ``nx, ny[, nz]`` cells of the box
[0,2]x[0,1][x[0,1]] (solid: the lowest quarter); ``pressure`` ("q1" or "p1disc");
``theta`` of the time scheme; ``precision`` of the preconditioner ("fp32" FP32-AMG or
"fp64"); ``learned``: whether the learned correction stage runs inside the solve;
``state``: the seed of a fixed linearisation state, with only the right-hand side new
(a quasi-Newton iteration keeps its Jacobian over several corrections).
"""
from __future__ import annotations

import functools
import math
import os
import struct

import numpy as np
import torch

import fsigen
import paper_1801_05648_gb300 as P

_WEIGHTS_2D = os.path.join(os.path.dirname(P.LIB_PATH), "weights", "mlp_fsi2d_256x128.bin")
_RTOL = 1e-8      # relative residual of every solve
_LR = 1e-4        # learning rate of the training step


# ------------------------------------------------------------------ the cases
def _case(kind, cells, pressure="q1", theta=1.0, precision="fp32", learned=False):
    c = {"kind": kind, "dim": len(cells), "nx": cells[0], "ny": cells[1], "nz": cells[2] if len(cells) == 3 else 1}
    if kind in ("jacobian", "residual", "rebuild", "solve"):
        c.update(pressure=pressure, theta=theta)
    if kind in ("rebuild", "solve"):
        c["precision"] = precision
    if kind == "solve":
        c["learned"] = learned
    return c


def listed():
    return [
        # the smallest solve: a coarse mesh in a parameter study, where launches and latency are all
        {"name": "solve_2d_16x16", **_case("solve", (16, 16))},
        # the ordinary 2D solve: the 256x128 channel, default FP32-AMG form
        {"name": "solve_2d_256x128", **_case("solve", (256, 128))},
        # the largest: 8.9 million unknowns, one Jacobian of 6 GB
        {"name": "solve_2d_1024x512", **_case("solve", (1024, 512)), "state": 0},
        # a ragged 3D mesh of the elastic obstacle in the all-FP64 form
        {"name": "solve_3d_21x11x10_fp64", **_case("solve", (21, 11, 10), precision="fp64")},
        # what every re-assembled Newton Jacobian costs before its solve: new values into the
        # context, the Schur operators and four AMG hierarchies, and the first P^-1 application
        {"name": "rebuild_2d_256x128", **_case("rebuild", (256, 128))},
        {"name": "rebuild_3d", **_case("rebuild", (32, 16, 16))},
        # the same for a small ragged mesh with the discontinuous pressure element, FP64
        {"name": "rebuild_2d_37x19_p1disc", **_case("rebuild", (37, 19), pressure="p1disc", precision="fp64")},
        # Jacobian assembly of the 2D channel, and of the 3D obstacle under Crank-Nicolson
        {"name": "jacobian_2d_256x128", **_case("jacobian", (256, 128))},
        {"name": "jacobian_3d_theta", **_case("jacobian", (32, 16, 16), theta=0.5)},
        # residual: evaluated once per Newton iterate, more often than the Jacobian
        {"name": "residual_2d_p1disc", **_case("residual", (256, 128), pressure="p1disc")},
        # learned stage: one correction of a residual, and one training step of the MLP
        {"name": "learned_2d_256x128", **_case("learned", (256, 128))},
        {"name": "train_2d_256x128", **_case("train", (256, 128))},
    ]


def draw(rng):
    kind = rng.choice(("solve", "solve", "rebuild", "rebuild", "jacobian", "residual", "learned", "train"))
    dim = rng.choice((2, 2, 3))

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if dim == 2:
        top = 512 if kind in ("jacobian", "residual") else 320
        nx = log_int(14, top)
        cells = (nx, max(7, min(top // 2, nx // 2 + rng.randint(-2, 3))))
    else:
        nx = log_int(6, 32 if kind in ("jacobian", "residual", "learned") else 24)
        cells = (nx, max(4, min(16, nx // 2 + rng.randint(-1, 1))), max(4, min(16, nx // 2 + rng.randint(-1, 1))))
    pressure = "p1disc" if kind in ("jacobian", "residual", "rebuild") and rng.random() < 0.3 else "q1"
    theta = 0.5 if rng.random() < 0.3 else 1.0
    precision = "fp64" if rng.random() < 0.35 else "fp32"
    learned = kind == "solve" and dim == 2 and precision == "fp32" and rng.random() < 0.3
    return _case(kind, cells, pressure, theta, precision, learned)


# ------------------------------------------------------------------ inputs
def _config(case):
    cells = (case["nx"], case["ny"], case["nz"])[: case["dim"]]
    return fsigen.FSIConfig("case", case["dim"], cells, theta=case.get("theta", 1.0),
                            pressure=case.get("pressure", "q1"))


def _state(cfg):
    """The seeded linearisation state, displacements and velocities of 0.2% to 0.6% of the box
    height: what a time step of the flow meets (some larger states compress the solid past the
    stability limit of its material law, and no hierarchy is built for those)."""
    amplitude = 2e-3 + 4e-3 * float(np.random.default_rng(cfg.state_seed).random())
    return fsigen.get_problem(cfg).seeded_state(cfg.state_seed, amplitude)


def _weights(dim, seed):
    """(sigma_in, sigma_out, bfloat16 words): the trained 2D weights; seeded random ones in 3D."""
    if dim == 2:
        with open(_WEIGHTS_2D, "rb") as f:
            raw = f.read()
        scales = struct.unpack("<10f", raw[24:64])
        return np.array(scales[:5], np.float32), np.array(scales[5:], np.float32), np.frombuffer(raw[64:], np.uint16)
    w = np.random.default_rng(seed + 17).normal(0.0, 0.1, P.mlp_params(3)).astype(np.float32)
    bits = torch.from_numpy(w).bfloat16().view(torch.int16).numpy().view(np.uint16)
    return np.full(5, 0.5, np.float32), np.full(5, 0.1, np.float32), bits


def _class_residual(pb, seed, sigma_in):
    """A residual vector as the learned stage meets it: class-scaled noise, zero on fixed rows."""
    r = np.random.default_rng(seed).standard_normal(pb.n)
    for k in range(5):
        r[pb.offsets[k]:pb.offsets[k + 1]] *= sigma_in[k]
    r[pb.fixed] = 0.0
    return r


def _dev(a):
    return torch.tensor(a, device="cuda")


@functools.lru_cache(maxsize=2)
def _context(cfg, precision=None):
    """The solver context that a program keeps for a mesh: the pattern alone, as a Newton loop
    sets it up, or with ``precision`` a Jacobian and its preconditioner kept for many right-hand sides."""
    pb = fsigen.get_problem(cfg)
    prm = P.default_params(cfg.dim, flags=P.FSI_USE_GRAPHS, dt_theta=cfg.dt * cfg.theta)
    vals = _jacobian(cfg) if precision else None
    S = P.FSISolver(pb.dim, pb.rowptr, pb.colind, vals, pb.offsets, pb.solid_node_coords(), prm)
    if precision:
        S.precond_build(precision)
    return S


@functools.lru_cache(maxsize=1)
def _jacobian(cfg):
    """Host values of the Jacobian at the configuration's seeded state (previous step = state)."""
    pb = fsigen.get_problem(cfg)
    U = _state(cfg)
    return pb.jacobian(U, U)


def _times(pb, vals, x):
    """A x on the GPU from the host CSR, each row summed in storage order."""
    prod = torch.from_numpy(vals).cuda() * _dev(x)[torch.from_numpy(pb.colind).cuda()]
    return torch.segment_reduce(prod, "sum", lengths=torch.from_numpy(np.diff(pb.rowptr)).cuda(), unsafe=True)


def prepare(case, seed):
    cfg = _config(case).with_(state_seed=case.get("state", seed))
    pb = fsigen.get_problem(cfg)
    kind = case["kind"]
    if kind in ("jacobian", "residual"):
        U = _state(cfg)
        Uold = 0.9 * U if case["theta"] != 1.0 else U     # a moving mesh where the previous level counts
        st = {"asm": P.FSIAssembler.from_problem(pb), "U": _dev(U), "Uold": _dev(Uold)}
        st["out"] = torch.empty(pb.nnz if kind == "jacobian" else pb.n, dtype=torch.float64, device="cuda")
    elif kind == "solve":
        make = _context if "state" in case else _context.__wrapped__
        S = make(cfg, case["precision"])
        if case["learned"]:
            S.learned_setup(*pb.node_map())
            S.learned_set_weights(*_weights(case["dim"], seed))
            S.set_flags(P.FSI_USE_GRAPHS | P.FSI_LEARNED)
        b = _times(pb, _jacobian(cfg), pb.rhs(seed + 1))
        st = {"S": S, "b": b, "x": torch.zeros_like(b)}
    elif kind == "rebuild":
        r = _dev(pb.rhs(seed + 1))
        st = {"S": _context(_config(case)), "vals": _dev(_jacobian(cfg)), "r": r, "z": torch.empty_like(r),
              "precision": case["precision"]}
    else:
        sig_in, sig_out, bits = _weights(case["dim"], seed)
        r = _dev(_class_residual(pb, seed, sig_in))
        if kind == "learned":
            S = _context(_config(case))
            S.learned_setup(*pb.node_map())
            S.learned_set_weights(sig_in, sig_out, bits)
            st = {"S": S, "r": r, "c": torch.empty_like(r)}
        else:
            S = _context.__wrapped__(cfg, "fp32")
            S.learned_setup(*pb.node_map())
            T = P.Trainer(dim=case["dim"], sigma_in=sig_in, sigma_out=sig_out)
            T.set_master((bits.astype(np.uint32) << 16).view(np.float32))
            st = {"S": S, "r": r, "T": T}
    st["kind"] = kind
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    kind = st["kind"]
    if kind == "solve":
        s = st["S"].solve(st["b"], st["x"], _RTOL)
        return {"x": st["x"], "iters": s.iters, "relres": s.true_relres}
    if kind == "rebuild":
        S = st["S"]
        S.update_values(st["vals"])
        S.precond_build(st["precision"])
        S.apply_block("precond", st["r"], st["z"])
        return st["z"]
    if kind == "jacobian":
        min_j = st["asm"].jacobian(st["U"], st["Uold"], st["out"])
        return {"vals": st["out"], "min_j": min_j}
    if kind == "residual":
        min_j, r_max = st["asm"].residual(st["U"], st["Uold"], st["out"])
        return {"R": st["out"], "min_j": min_j, "r_max": r_max}
    if kind == "learned":
        st["S"].learned_apply(st["r"], st["c"])
        return st["c"]
    loss = st["T"].step(st["S"], st["r"])
    grad = st["T"].get()[2]
    st["T"].update(st["S"], _LR)
    return {"loss": loss, "grad": grad}


# ------------------------------------------------------------------ work
def _element(case):
    """(unknowns, Jacobian entries, cells, element unknowns, points per cell, Q2 nodes)."""
    pb = fsigen.get_problem(_config(case))
    nq2 = 3 ** case["dim"]
    npr = case["dim"] + 1 if case.get("pressure") == "p1disc" else 2 ** case["dim"]
    cells = case["nx"] * case["ny"] * case["nz"]
    return pb.n, pb.nnz, cells, 2 * nq2 * case["dim"] + npr, nq2, pb.n_q2


def work(case):
    n, nnz, cells, nl, nqp, nodes = _element(case)
    kind, d = case["kind"], case["dim"]
    if kind == "solve":          # matrix, b read; x written; at least one product with the operator
        return {"bytes": 12 * nnz + 8 * n + 16 * n, "flops": 2 * nnz}
    if kind == "rebuild":        # new values, r read; z written; one product with the preconditioner's blocks
        return {"bytes": 12 * nnz + 8 * n + 16 * n, "flops": 2 * nnz}
    if kind == "jacobian":       # state and element map read, values written; per point and column pair an FMA
        return {"bytes": 16 * n + 4 * nl * cells + 12 * nnz, "flops": 2 * cells * nqp * nl * nl}
    if kind == "residual":
        return {"bytes": 24 * n + 4 * nl * cells, "flops": 2 * cells * nqp * nl * 2 * (d + 1)}
    mlp = P.mlp_inputs(d) * 64 + 64 * 64 + 64 * (2 * d + 1)
    if kind == "learned":        # r, node records and patches read, c written
        return {"bytes": 16 * n + nodes * (16 + 4 * 3 ** d), "flops": 2 * nodes * mlp}
    return {"bytes": 16 * n + nodes * (16 + 4 * 3 ** d) + 12 * nnz, "flops": 6 * nodes * mlp + 4 * nnz}


# ------------------------------------------------------------------ 64-bit values
# Plain torch in FP64 from the same mesh tables and vectors.  Solves and rebuilt
# preconditioners have none: at rtol 1e-8 the solution of these systems (condition
# numbers near 1e14) is fixed by the iteration, and P^-1 is defined by its AMG.
def exact(case, seed):
    if case["kind"] in ("solve", "rebuild"):
        return None
    cfg = _config(case).with_(state_seed=seed)
    pb = fsigen.get_problem(cfg)
    if case["kind"] in ("jacobian", "residual"):
        return _exact_assembly(case, cfg, pb, seed)
    return _exact_mlp(case, cfg, pb, seed)


def _tables(dim, h, pressure, face):
    """Gauss points of the reference cell (or of its face x_0 = 1): weights, Q2 basis, its
    gradients in x, pressure basis."""
    g, gw = [0.5 - math.sqrt(0.15), 0.5, 0.5 + math.sqrt(0.15)], [5 / 18, 8 / 18, 5 / 18]
    free = dim - 1 if face else dim
    pts, w = [], []
    for q in range(3 ** free):
        i = [(q // 3 ** k) % 3 for k in range(free)]
        pts.append(([1.0] if face else []) + [g[k] for k in i])
        w.append(math.prod(gw[k] for k in i) * math.prod(h[1:dim] if face else h[:dim]))
    x = np.array(pts)
    b = np.stack([2 * (x - 0.5) * (x - 1), -4 * x * (x - 1), 2 * x * (x - 0.5)])
    db = np.stack([4 * x - 3, 4 - 8 * x, 4 * x - 1])
    N = np.ones((len(pts), 3 ** dim))
    dN = np.ones((len(pts), 3 ** dim, dim))
    for a in range(3 ** dim):
        ia = [(a // 3 ** k) % 3 for k in range(dim)]
        for k in range(dim):
            N[:, a] *= b[ia[k], :, k]
            for j in range(dim):
                dN[:, a, j] *= db[ia[k], :, k] / h[k] if j == k else b[ia[k], :, k]
    if pressure == "p1disc":
        Np = np.concatenate([np.ones((len(pts), 1)), 2 * x - 1], 1)
    else:
        Np = np.ones((len(pts), 2 ** dim))
        for a in range(2 ** dim):
            for k in range(dim):
                Np[:, a] *= x[:, k] if (a >> k) & 1 else 1 - x[:, k]
    return [torch.tensor(t, device="cuda") for t in (np.array(w), N, dN, Np)]


def _element_residual(case, cfg, Ue, Uo, kind, tab):
    """Element residuals [cells, NL] of cells of one kind ("fluid", "solid" or "face": the
    outflow term of fluid cells) and det F at the points."""
    d, nq = case["dim"], 3 ** case["dim"]
    w, N, dN, Np = tab
    eye = torch.eye(d, dtype=torch.float64, device="cuda")
    dtt, dto, th = cfg.dt * cfg.theta, cfg.dt * (1 - cfg.theta), cfg.theta
    mu = cfg.rho_f * cfg.nu_f

    def point(X):
        v, u = X[:, : nq * d].reshape(-1, nq, d), X[:, nq * d: 2 * nq * d].reshape(-1, nq, d)
        Gv, F = torch.einsum("qaj,cai->cqij", dN, v), torch.einsum("qaj,cai->cqij", dN, u) + eye
        J = torch.linalg.det(F)
        return torch.einsum("qa,cai->cqi", N, v), torch.einsum("qa,cai->cqi", N, u), Gv, F, J

    v, u, Gv, F, J = point(Ue)
    vo, uo, Gvo, Fo, Jo = point(Uo)
    Jx, Jox = J[..., None, None], Jo[..., None, None]
    nl = Ue.shape[1]
    zero = torch.zeros_like(Ue[:, 2 * nq * d:])

    def test(f0, f1):
        return (torch.einsum("q,qa,cqi->cai", w, N, f0) + torch.einsum("q,qaj,cqij->cai", w, dN, f1)).reshape(-1, nq * d)

    if kind == "solid":
        def stress(F):
            E = 0.5 * (F.mT @ F - eye)
            tr = E.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None]
            return F @ (2 * cfg.mu_s * E + cfg.lambda_s * tr * eye)
        Rv = test(cfg.rho_s * (v - vo), dtt * stress(F) + dto * stress(Fo))
        k0 = (u - uo) - dtt * v - dto * vo
        Ru = torch.einsum("q,qa,cqi->cai", w, N, k0).reshape(-1, nq * d)
        return torch.cat([Rv, Ru, zero], 1), J
    Fi, Foi = torch.linalg.inv(F), torch.linalg.inv(Fo)
    if kind == "face":
        def out(Gv, Fi, J):
            t = torch.einsum("cqkj,cqk->cqj", Gv, Fi[..., 0, :])
            return J[..., None] * torch.einsum("cqji,cqj->cqi", Fi, t)
        c = -mu * (dtt * out(Gv, Fi, J) + dto * out(Gvo, Foi, Jo))
        Rv = torch.einsum("q,qa,cqi->cai", w, N, c).reshape(-1, nq * d)
        return torch.cat([Rv, torch.zeros_like(Rv), zero], 1), J
    p = torch.einsum("qa,ca->cq", Np, Ue[:, 2 * nq * d:])
    A, Ao = Gv @ Fi, Gvo @ Foi

    def mv(M, x):
        return (M @ x[..., None])[..., 0]
    Jt = (th * J + (1 - th) * Jo)[..., None]
    f0 = cfg.rho_f * (Jt * (v - vo) - J[..., None] * (mv(A, u - uo) - dtt * mv(A, v)) + dto * Jo[..., None] * mv(Ao, vo))
    f1 = mu * (dtt * Jx * ((A + A.mT) @ Fi.mT) + dto * Jox * ((Ao + Ao.mT) @ Foi.mT)) - (J * p)[..., None, None] * Fi.mT
    Rv = test(f0, f1)
    hm = (F - eye) / Jx
    Ru = torch.einsum("q,qaj,cqij->cai", w, dN, hm).reshape(-1, nq * d)
    Rp = torch.einsum("q,qa,cq->ca", w, Np, J * A.diagonal(dim1=-2, dim2=-1).sum(-1))
    return torch.cat([Rv, Ru, Rp], 1)[:, :nl], J


def _exact_assembly(case, cfg, pb, seed):
    d, nq = case["dim"], 3 ** case["dim"]
    h = [cfg.L[k] / cfg.n[k] for k in range(d)]
    U = _state(cfg)
    Ud = _dev(U)
    Uo = _dev(0.9 * U if case["theta"] != 1.0 else U)
    cd, cf = pb.cell_map()
    cd, cf = torch.tensor(cd, device="cuda").long(), torch.tensor(cf.astype(np.int64), device="cuda")
    fixed = torch.tensor(pb.fixed, device="cuda")
    nl = cd.shape[1]
    jac = case["kind"] == "jacobian"
    if jac:
        rowptr = torch.tensor(pb.rowptr, device="cuda")
        rows = torch.repeat_interleave(torch.arange(pb.n, device="cuda"), rowptr.diff())
        key = rows * pb.n + torch.tensor(pb.colind, device="cuda")
        out = torch.where(rows == torch.tensor(pb.colind, device="cuda"), fixed[rows].double(), 0.0)
    else:
        out = torch.zeros(pb.n, dtype=torch.float64, device="cuda")
    min_j = math.inf
    solid = (cf & 1) == 1
    for kind, sel in (("fluid", ~solid), ("face", ~solid & ((cf & 2) == 2)), ("solid", solid)):
        tab = _tables(d, h, case["pressure"], kind == "face")
        for part in torch.nonzero(sel)[:, 0].split(2048):
            dof, fl = cd[part], cf[part]
            keep = ~fixed[dof]                                         # rows of the element that are assembled
            if kind == "solid":
                keep[:, 2 * nq * d:] = False
            else:
                for a in range(nq):                                    # fluid cells: mesh-motion rows only
                    keep[:, nq * d + a * d: nq * d + (a + 1) * d] &= ((fl >> (2 + a)) & 1).bool()[:, None]
            Ue, Uoe = Ud[dof], Uo[dof]

            def f(X):
                return _element_residual(case, cfg, X, Uoe, kind, tab)[0]
            if not jac:
                R, J = _element_residual(case, cfg, Ue, Uoe, kind, tab)
                out.index_add_(0, dof[keep], R[keep])
            else:
                J = _element_residual(case, cfg, Ue, Uoe, kind, tab)[1]
                for k in range(nl):
                    col = dof[:, k]
                    ok = keep & ~fixed[col][:, None]
                    if kind == "solid" and k >= 2 * nq * d:
                        continue
                    t = torch.zeros_like(Ue)
                    t[:, k] = 1.0
                    dR = torch.func.jvp(f, (Ue,), (t,))[1]
                    want, val = (dof * pb.n + col[:, None])[ok], dR[ok]
                    at = torch.searchsorted(key, want).clamp(max=pb.nnz - 1)
                    hit = key[at] == want                              # pairs outside the pattern do not couple
                    out.index_add_(0, at[hit], val[hit])
            if kind != "face":
                min_j = min(min_j, float(J.min()))
    if jac:
        return {"vals": out, "min_j": min_j}
    return {"R": out, "min_j": min_j, "r_max": float(out.abs().max())}


def _exact_mlp(case, cfg, pb, seed):
    d = case["dim"]
    sig_in, sig_out, bits = _weights(d, seed)
    scale_in, scale_out = np.empty(pb.n), np.empty(pb.n)
    for k in range(5):
        scale_in[pb.offsets[k]:pb.offsets[k + 1]] = sig_in[k]
        scale_out[pb.offsets[k]:pb.offsets[k + 1]] = sig_out[k]
    r = _dev(_class_residual(pb, seed, sig_in))
    nd, pt = (torch.tensor(t, device="cuda").long() for t in pb.node_map())
    x = torch.cat([r / _dev(scale_in), torch.zeros(1, dtype=torch.float64, device="cuda")])
    absent = pb.n
    comps = [nd[:, 0] + k for k in range(d)] + [nd[:, 1] + k for k in range(d)]
    comps.append(torch.where(nd[:, 2] >= 0, nd[:, 2], absent))
    dofs = torch.stack(comps, 1)
    pad = torch.cat([dofs, torch.full((1, 2 * d + 1), absent, device="cuda")])
    feat = x[pad[pt]].reshape(len(nd), -1)                              # patch index -1 is the absent node
    rho = feat.square().mean(1).sqrt()
    fl = nd[:, 3]
    par = ((fl >> 4) & 1) + 2 * ((fl >> 5) & 1) + (4 * ((fl >> 7) & 1) if d == 3 else 0)
    flags = torch.stack([(fl >> k) & 1 for k in range(4)], 1).double()
    inv = torch.where(rho > 0, 1 / rho, 0.0)
    f = torch.cat([feat * inv[:, None], torch.nn.functional.one_hot(par, 2 ** d).double(), flags], 1)
    n_in, n_out = f.shape[1], 2 * d + 1
    w = torch.tensor((bits.astype(np.uint32) << 16).view(np.float32), device="cuda").double()
    w.requires_grad_(case["kind"] == "train")
    W1, b1, W2, b2, W3, b3 = torch.split(w, [n_in * 64, 64, 4096, 64, 64 * n_out, n_out])
    g = torch.nn.functional.gelu
    y = g(g(f @ W1.reshape(n_in, 64) + b1) @ W2.reshape(64, 64) + b2) @ W3.reshape(64, n_out) + b3
    free = torch.cat([_dev(~pb.fixed).double() * _dev(scale_out), torch.zeros(1, dtype=torch.float64, device="cuda")])
    c = torch.zeros(pb.n + 1, dtype=torch.float64, device="cuda")
    c = c.index_add(0, dofs.reshape(-1), (y * rho[:, None] * free[dofs]).reshape(-1))[: pb.n]
    if case["kind"] == "learned":
        return c
    A = torch.sparse_csr_tensor(torch.tensor(pb.rowptr), torch.tensor(pb.colind).long(),
                                torch.tensor(_jacobian(cfg)), (pb.n, pb.n)).cuda()
    res = r - (A @ c.detach()[:, None])[:, 0]
    rows = torch.repeat_interleave(torch.arange(pb.n, device="cuda"), A.crow_indices().diff())
    at_res = torch.zeros_like(r).index_add_(0, A.col_indices(), A.values() * res[rows])
    r2 = r.square().sum()
    c.backward(-2 / r2 * at_res)
    return {"loss": float(res.square().sum() / r2), "grad": w.grad}
