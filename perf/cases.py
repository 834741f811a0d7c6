"""Performance cases of the tangent-point surface flow, through the package's public calls.

A program that repels a surface from itself repeats a few calls on a mesh that it keeps: new positions, the
energy and its differential (as a torch loss, or directly), the operators A and L^{2-s} on a few vector
fields, Poisson and preconditioner solves, and the constrained step built from all of them. The kinds below
are those calls; the meshes are the noisy tori, linked tori and icospheres of `synth`, at the sizes of this
repository's benchmark configurations (1,280 to 50,000 faces with exact pair sums, icospheres of 10^5 to
10^6 faces with Barnes-Hut sums) and of the requests that its server takes (2,000 to 200,000 faces).

Pair terms run in FP32 (the default, TP_PREC_FP32), so a program keeps the fields that go in and come out
in float32, as torch parameters and gradients are; the FP64 case keeps float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2107_01664_gb300 as tp
from synth import icosphere, linked_tori, torus

DEV = "cuda:0"
_TOPOLOGY = {}


def listed():
    base = dict(sigma=0.005, p=6.0, theta=0.0, precision="fp32", op="", cols=0, tol=1e-6, seed_shift=0)

    def case(name, kind, mesh, a, b, **kw):
        return {"name": name, "kind": kind, "mesh": mesh, "a": a, "b": b, **base, **kw}

    return [
        # one step of a torch optimiser on the smallest configuration: launches and latency
        case("loss_1k", "loss", "icosphere", 3, 0, sigma=0.01),
        # the same on the ordinary configuration
        case("loss_20k", "loss", "torus", 200, 50),
        # a line-search trial of a served mesh of odd size: new positions, exact energy
        case("energy_70k", "energy", "torus", 345, 101),
        # value and differential of a large smooth surface: tree, interaction lists, far and near sums
        case("diff_bh_328k", "diff", "icosphere", 7, 0, sigma=0.05, theta=0.5),
        # the operator of a Krylov iteration on three right-hand sides at once
        case("apply_A9_20k", "apply", "torus", 200, 50, op="A", cols=9),
        # the preconditioner's operator on one vector field, ragged size, another exponent
        case("apply_L3_8k", "apply", "torus", 97, 41, op="L", cols=3, p=4.5),
        # the operator on one vector field of a large surface, tree and lists kept with the mesh
        case("apply_A3_bh_328k", "apply", "icosphere", 7, 0, sigma=0.05, op="A", cols=3, theta=0.5),
        # the double-precision mode, which runs are checked with
        case("apply_A3_fp64_3k", "apply", "torus", 60, 25, op="A", cols=3, precision="fp64"),
        # new positions and one Laplace solve (Sobolev smoothing of a gradient), two components
        case("poisson_50k", "poisson", "linked", 250, 50, cols=3, sigma=0.002),
        # the same on a large surface, to a tight tolerance
        case("poisson_328k", "poisson", "icosphere", 7, 0, cols=3, sigma=0.05, tol=1e-9),
        # the fractional preconditioner of one gradient
        case("precond_20k", "precond", "torus", 200, 50, cols=3),
        # a whole constrained descent step of the benchmark's configuration
        case("step_20k", "step", "torus", 200, 50, tol=1e-4),
    ]


def draw(rng):
    def loguni(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def grid(nf):   # torus with about nf faces: rows about a third to a fifth of the columns
        b = max(7, round(math.sqrt(nf / 2 / rng.uniform(3.0, 5.0))))
        return max(9, round(nf / 2 / b)), b

    kind = rng.choice(["loss", "loss", "energy", "diff", "diff_bh", "apply", "apply", "apply_bh", "apply64", "poisson",
                       "precond", "step", "step_bh"])
    c = dict(kind=kind.split("_")[0], mesh="torus", sigma=0.005, p=rng.choice([6.0, 6.0, 6.0, 4.5, 3.0]), theta=0.0,
             precision="fp32", op="", cols=0, tol=1e-6, seed_shift=rng.randrange(1000))
    if kind in ("loss", "diff"):
        c["a"], c["b"] = grid(loguni(400, 30000))
    elif kind == "energy":
        c["a"], c["b"] = grid(loguni(1000, 70000))
    elif kind == "diff_bh":
        c["a"], c["b"] = grid(loguni(20000, 200000))
        c.update(theta=rng.choice([0.25, 0.5]), sigma=0.002)
    elif kind == "apply":
        c["a"], c["b"] = grid(loguni(400, 24000))
        c.update(op=rng.choice(["A", "A", "B", "B0", "L"]), cols=rng.choice([1, 3, 3, 4, 9, 9]))
    elif kind == "apply_bh":
        c["a"], c["b"] = grid(loguni(20000, 200000))
        c.update(theta=0.5, sigma=0.002, op=rng.choice(["A", "A", "B", "B0", "L"]), cols=rng.choice([1, 3, 9]))
    elif kind == "apply64":
        c["a"], c["b"] = grid(loguni(400, 4000))
        c.update(kind="apply", precision="fp64", op=rng.choice(["A", "L"]), cols=rng.choice([1, 3, 9]))
    elif kind == "poisson":
        c["a"], c["b"] = grid(loguni(1000, 200000))
        c.update(cols=rng.choice([1, 3, 9]), tol=1e-8)
    elif kind == "precond":
        c["a"], c["b"] = grid(loguni(1000, 20000))
        c.update(cols=rng.choice([3, 9]))
    elif kind == "step":
        c["a"], c["b"] = grid(loguni(1000, 16000))
        c.update(p=6.0, tol=1e-4)
    else:
        c.update(kind="step", mesh="linked", a=rng.randint(60, 220), b=rng.randint(15, 44), theta=0.5, sigma=0.002,
                 p=6.0, tol=1e-4)
    return c


# ---- meshes -----------------------------------------------------------------------------------------------


def _topology(c):
    key = (c["mesh"], c["a"], c["b"])
    if key not in _TOPOLOGY:
        if c["mesh"] == "icosphere":
            V, F = icosphere(c["a"])
        elif c["mesh"] == "linked":
            V, F = linked_tori(c["a"], c["b"], 1.0, 0.25, 1.0)
        else:
            V, F = torus(c["a"], c["b"], 1.0, 0.3)
        _TOPOLOGY[key] = (torch.as_tensor(V, dtype=torch.float64, device=DEV),
                          torch.as_tensor(np.ascontiguousarray(F), dtype=torch.int32, device=DEV))
    return _TOPOLOGY[key]


def _inputs(c, seed):
    """Positions [nv,3] and a field [nv,cols], in the dtype that the program keeps."""
    V, F = _topology(c)
    g = torch.Generator(device=DEV).manual_seed(1000 * seed + c["seed_shift"])
    if c["mesh"] == "icosphere" and c["a"] >= 6:   # a smooth bumpy sphere: low-degree radial bumps
        w = torch.randn(9, generator=g, device=DEV, dtype=torch.float64)
        x, y, z = V.T
        q = torch.stack([x, y, z, x * y, y * z, z * x, x * x - y * y, x * y * z, z * (x * x - y * y)])
        r = w @ q
        V = V * (1.0 + c["sigma"] * r / r.abs().max())[:, None]
    else:
        V = V + c["sigma"] * torch.randn(V.shape, generator=g, device=DEV, dtype=torch.float64)
    dt = torch.float64 if c["precision"] == "fp64" else torch.float32
    v = torch.randn((V.shape[0], max(1, c["cols"])), generator=g, device=DEV, dtype=torch.float64)
    return V.to(dt), F, v.to(dt)


def _params(c):
    kw = dict(p=c["p"], theta=c["theta"], precision=tp.TP_PREC_FP64 if c["precision"] == "fp64" else tp.TP_PREC_FP32,
              cg_tol=c["tol"])
    if c["kind"] == "step":   # the benchmark's step: 1e-5 Krylov solves, a displacement-bounded first trial
        kw.update(krylov_tol=1e-5, krylov_max=60, tau0_disp=0.25)
    return tp.params(**kw)


def prepare(case, seed):
    f, F, v = _inputs(case, seed)
    s = {"case": case, "f": f, "v": v, "p": _params(case), "mesh": tp.Mesh(f, F, device=0)}
    if case["kind"] == "loss":
        s["f"] = f.clone().requires_grad_(True)
    if case["kind"] == "step":
        A0, V0 = tp.tp_mesh_area_volume(s["mesh"])
        s["cons"] = tp.tp_constraints(tp.TP_CONSTRAINT_AREA | tp.TP_CONSTRAINT_VOLUME, A0, V0)
    return s


def run(state):
    kind, mesh, p, f, v = (state["case"]["kind"], state["mesh"], state["p"], state["f"], state["v"])
    if kind == "loss":
        f.grad = None
        E = tp.TangentPointEnergy.apply(f, mesh, p)
        E.backward()
        return E.detach(), f.grad
    if kind == "energy":
        mesh.set_positions(f)
        return tp.tp_energy(mesh, p)
    if kind == "diff":
        mesh.set_positions(f)
        dE, E = tp.tp_differential(mesh, p, like=f)
        return E, dE.to(f.dtype)
    if kind == "apply":
        return tp.fractional_apply(mesh, state["case"]["op"], v, p).to(v.dtype)
    if kind == "poisson":
        mesh.set_positions(f)
        z, _ = tp.cotan_solve(mesh, v, p)
        return z.to(v.dtype)
    if kind == "precond":
        return tp.precond_apply(mesh, v, p).to(v.dtype)
    mesh.set_positions(f)
    rep = tp.precond_step(mesh, state["cons"], p)
    return rep["E_before"], rep["E_after"], mesh.get_positions(like=f).to(f.dtype)


# ---- work -------------------------------------------------------------------------------------------------


def _sizes(c):
    if c["mesh"] == "icosphere":
        return 10 * 4 ** c["a"] + 2, 20 * 4 ** c["a"]
    n = c["a"] * c["b"] * (2 if c["mesh"] == "linked" else 1)
    return n, 2 * n


def work(case):
    """Terms of every ordered pair (exact sums) or of about 1,500 interactions a face (Barnes-Hut), with the
    difference and |d|^2 of a pair counted for both of its orders where both are summed; inputs and results once."""
    nv, nf = _sizes(case)
    k = case["cols"]
    pairs = nf * (nf - 1.0) if case["theta"] == 0.0 else 1500.0 * nf
    energy, diff = 16.0, 50.0
    ops = {"A": 22 + 2 * (2 + 4 * k), "B": 10 + 2 * (1 + 3 * k), "B0": 22 + 2 * (1 + k), "L": 10 + 2 * (1 + k)}
    w = 4 if case["precision"] == "fp32" else 8
    mesh = 12.0 * nf + 3 * w * nv
    lap = 12.0 * (7 * nv) + 2 * w * nv * max(1, k)
    kind = case["kind"]
    if kind == "loss":
        return {"bytes": mesh + 3 * w * nv, "flops": pairs * (energy + diff)}
    if kind == "energy":
        return {"bytes": mesh, "flops": pairs * energy}
    if kind == "diff":
        return {"bytes": mesh + 3 * w * nv, "flops": pairs * diff}
    if kind == "apply":
        return {"bytes": mesh + 2 * w * nv * k, "flops": pairs * ops[case["op"]]}
    if kind == "poisson":   # values of C and a direct solve's factor (about 4 n log2 n entries), once each way
        return {"bytes": mesh + lap + 4.0 * 8 * nv * math.log2(nv), "flops": 16.0 * nv * math.log2(nv) * k}
    if kind == "precond":
        return {"bytes": mesh + 2 * lap, "flops": pairs * ops["L"]}
    k = 9   # about 20 iterations on three right-hand sides, two energies and one differential
    return {"bytes": mesh + 20 * (2 * 8.0 * 9 * nv), "flops": pairs * (2 * energy + diff + 20 * (22 + 4 + 72 + 10 + 20))}


# ---- the same results in 64 bits, in plain torch ----------------------------------------------------------


def _face_geometry(f, F):
    a, b, c = f[F[:, 0]], f[F[:, 1]], f[F[:, 2]]
    n = torch.linalg.cross(b - a, c - a)
    nn = n.norm(dim=1)
    return (a + b + c) / 3.0, n / nn[:, None], 0.5 * nn


def _energy64(f, F, p, grad):
    """E and dE/df by chunks of target faces; the gradient through the faces' X, N and a."""
    X, N, a = _face_geometry(f, F)
    X0, N0, a0 = (t.detach().requires_grad_(grad) for t in (X, N, a))
    E, nf = 0.0, len(a)
    step = max(1, 20_000_000 // nf)
    for i in range(0, nf, step):
        with torch.set_grad_enabled(grad):
            S = slice(i, min(nf, i + step))
            d = X0[S, None, :] - X0[None, :, :]
            r2 = (d * d).sum(-1)
            own = torch.arange(S.start, S.stop, device=f.device)[:, None] == torch.arange(nf, device=f.device)[None, :]
            r2 = torch.where(own, torch.ones_like(r2), r2)
            u = (N0[S, None, :] * d).sum(-1)
            K = ((u * u) / (r2 * r2)) ** (0.5 * p)
            K = torch.where(own, torch.zeros_like(K), K)
            e = (a0[S] * (K @ a0)).sum()
            if grad:
                e.backward()
        E += float(e.detach())
    if not grad:
        return E, None
    leaf = f.detach().requires_grad_(True)
    torch.autograd.backward(_face_geometry(leaf, F), (X0.grad, N0.grad, a0.grad))
    return E, leaf.grad


def _kernel_product64(X, N, a, W, expo, low):
    """(diag(H a / a) - H) W, H_ST = |d|^{-expo}, times the symmetrised k_2 factor for the low-order kernel."""
    nf = len(a)
    out = torch.empty_like(W)
    step = max(1, 20_000_000 // nf)
    for i in range(0, nf, step):
        S = slice(i, min(nf, i + step))
        d = X[S, None, :] - X[None, :, :]
        r2 = (d * d).sum(-1)
        own = torch.arange(S.start, S.stop, device=X.device)[:, None] == torch.arange(nf, device=X.device)[None, :]
        r2 = torch.where(own, torch.ones_like(r2), r2)
        H = r2 ** (-0.5 * expo)
        if low:
            uS, uT = (N[S, None, :] * d).sum(-1), (N[None, :, :] * d).sum(-1)
            H = H * (uS * uS + uT * uT) / (2.0 * r2 * r2)
        H = torch.where(own, torch.zeros_like(H), H)
        out[S] = ((H @ a) / a[S])[:, None] * W[S] - H @ W
    return out


def _hat_gradients(f, F):
    a, b, c = f[F[:, 0]], f[F[:, 1]], f[F[:, 2]]
    _, N, area = _face_geometry(f, F)
    e = torch.stack([c - b, a - c, b - a], 1)
    return torch.linalg.cross(N[:, None, :].expand_as(e), e) / (2.0 * area)[:, None, None]


def _apply64(f, F, v, op, p):
    X, N, a = _face_geometry(f, F)
    s, k = 2.0 - 2.0 / p, v.shape[1]
    G, vF = _hat_gradients(f, F), v[F]            # [nf,3,3], [nf,3,k]
    y = torch.zeros_like(v)
    if op in ("A", "B"):
        W = a[:, None, None] * torch.einsum("sci,sck->sik", G, vF)
        z = a[:, None, None] * _kernel_product64(X, N, a, W.reshape(len(a), 3 * k), 2.0 * s, False).reshape(-1, 3, k)
        for c in range(3):
            y.index_add_(0, F[:, c], 2.0 * torch.einsum("si,sik->sk", G[:, c, :], z))
    if op != "B":
        W = a[:, None] * vF.mean(1)
        expo = 2.0 * (2.0 - s) + 2.0 if op == "L" else 2.0 * s
        z = a[:, None] * _kernel_product64(X, N, a, W, expo, op != "L")
        for c in range(3):
            y.index_add_(0, F[:, c], (2.0 / 3.0) * z)
    return y


def _stiffness(f, F, weight):
    """CSR matrix sum_S w_S a_S grad phi_i . grad phi_j (the cotan matrix for w = 1)."""
    _, _, a = _face_geometry(f, F)
    G = _hat_gradients(f, F)
    blocks = (weight * a)[:, None, None] * torch.einsum("sci,sdi->scd", G, G)
    I = F[:, :, None].expand(-1, 3, 3).reshape(-1)
    J = F[:, None, :].expand(-1, 3, 3).reshape(-1)
    n = f.shape[0]
    return torch.sparse_coo_tensor(torch.stack([I, J]), blocks.reshape(-1), (n, n)).coalesce().to_sparse_csr()


def _mean_zero(x, parts):
    n = x.shape[0] // parts
    return (x.reshape(parts, n, -1) - x.reshape(parts, n, -1).mean(1, keepdim=True)).reshape(x.shape)


def _solve64(C, dinv, b, parts):
    """C^+ b by conjugate gradients, every column to a relative residual of 1e-13 (or as far as 64 bits go)."""
    b = _mean_zero(b, parts)
    x, r = torch.zeros_like(b), b.clone()
    z = dinv[:, None] * r
    q, rz, bb = z.clone(), (r * z).sum(0), b.norm(dim=0)
    for it in range(12000):
        Cq = C @ q
        alpha = rz / (q * Cq).sum(0)
        x += alpha * q
        r -= alpha * Cq
        z = dinv[:, None] * r
        new = (r * z).sum(0)
        q = z + (new / rz) * q
        rz = new
        if it % 50 == 49:
            if bool((r.norm(dim=0) <= 1e-13 * bb).all()):
                break
    return _mean_zero(x, parts)


def exact(case, seed):
    if case["theta"] > 0.0 or case["kind"] == "step":   # tree sums have their own error; a step is many solves
        return None
    f, F, v = _inputs(case, seed)
    f, F, v = f.double(), F.long(), v.double()
    kind, p = case["kind"], case["p"]
    if kind in ("loss", "diff", "energy"):
        E, dE = _energy64(f, F, p, kind != "energy")
        E = torch.tensor(E, dtype=torch.float64)
        return E if kind == "energy" else (E, dE)
    if kind == "apply":
        return _apply64(f, F, v, case["op"], p)
    C = _stiffness(f, F, torch.ones(len(F), dtype=torch.float64, device=f.device))
    n, parts = f.shape[0], 2 if case["mesh"] == "linked" else 1
    rows = torch.repeat_interleave(torch.arange(n, device=f.device), C.crow_indices().diff())
    diag = torch.zeros(n, dtype=torch.float64, device=f.device)
    own = C.col_indices() == rows
    diag[rows[own]] = C.values()[own]
    if kind == "poisson":
        return _solve64(C, 1.0 / diag, v, parts)
    sigma = 2.0 / p                                      # 2 - s
    _, _, a = _face_geometry(f, F)
    G = _stiffness(f, F, 24.0 * a ** (1.0 - sigma))      # the within-face term at its default weight
    z = _solve64(C, 1.0 / diag, v, parts)
    y = _apply64(f, F, z, "L", p) + G @ z
    return _solve64(C, 1.0 / diag, y, parts)
