"""Workloads of the RPY mobility library, each one pass through its public entry points.

A pass is what a simulation does per step: positions go in with
``lm_set_positions`` (or the ``NBody`` class of the paper's interface), then
products, square roots, gradients or a batched run come out, in the default
launch configuration.  Inputs are those of the repository's benchmark
(``paper_2510_02135_gb300.inputs``: spheres uniform in a cube, bead chains,
a layer of rollers above a wall, batches of small suspensions), drawn from
the seed.

``work`` counts one pass's unavoidable work: every input and output once, and
the flops of the far-field pair formulas (FMA = 2) with each unordered pair's
coefficients formed once and applied to both particles.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_02135_gb300 import inputs, lm

# "iters" in a case is the typical number of Lanczos iterations, for work().
# Flops of one pair: (coefficients, once per unordered pair; application, once
# per ordered pair).  Adjoint: one product plus the gradient of the pair term.
_FLOPS = {
    ("open", False): (15, 18), ("open", True): (15, 71),
    ("wall", False): (83, 45), ("wall", True): (113, 185),
    ("adjoint", False): (48, 30), ("adjoint", True): (120, 80),
}


def listed():
    return [
        # One step of a small deterministic simulation: the call's latency.
        {"name": "step_open_n1000", "kind": "step", "n": 1000, "phi": 0.1, "angular": False, "fp64": False},
        # Forces-only product at the largest sizes where a direct sum is the
        # solver of choice (some 50 thousand particles), an odd count.
        {"name": "step_open_n50021", "kind": "step", "n": 50021, "phi": 0.05, "angular": False, "fp64": False},
        # Forces and torques on the polymer melt of the benchmark: the largest product.
        {"name": "melt_6n_n524288", "kind": "melt", "chains": 1024, "beads": 512},
        # Langevin velocities (product and Brownian term) of an ordinary
        # suspension: many small launches per Lanczos iteration.
        {"name": "langevin_open_n4096", "kind": "langevin", "n": 4096, "phi": 0.2, "tol": 1e-3, "iters": 26},
        # Brownian displacements with torque blocks, the benchmark's square root.
        {"name": "sqrt_6n_n32768", "kind": "sqrt", "n": 32768, "phi": 0.2, "angular": True, "fp64": False,
         "tol": 1e-5, "iters": 97},
        # The FP64 reference runs: a square root to tight tolerance on a small
        # system, and products with torques on an ordinary one.
        {"name": "sqrt_fp64_n1024", "kind": "sqrt", "n": 1024, "phi": 0.1, "angular": False, "fp64": True,
         "tol": 1e-8, "iters": 68},
        {"name": "step_fp64_6n_n8001", "kind": "step", "n": 8001, "phi": 0.1, "angular": True, "fp64": True},
        # A differentiable simulation: forward and backward through the product.
        {"name": "grad_open_n65536", "kind": "grad", "n": 65536, "phi": 0.1, "angular": False},
        {"name": "grad_6n_n16384", "kind": "grad", "n": 16384, "phi": 0.1, "angular": True},
        # The paper's bottom-wall benchmark: forces only, above a no-slip wall.
        {"name": "wall_n32768", "kind": "wall", "n": 32768, "rho": 0.1},
        # Active rollers above a wall: steric forces, then the Langevin
        # velocities with torques, Brownian term and thermal drift.
        {"name": "rollers_n32768", "kind": "rollers", "n": 32768, "iters": 10},
        # Brownian dynamics of many small independent suspensions at once.
        {"name": "batch_bd_256", "kind": "batch", "systems": 256, "nmin": 64, "nmax": 4096, "steps": 4, "iters": 38},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over the logarithm of each kind's range."""
    kind = rng.choice(["step", "step", "melt", "langevin", "sqrt", "grad", "wall", "rollers", "batch"])
    phi = round(rng.uniform(0.02, 0.3), 3)
    if kind == "step":
        fp64, angular = rng.random() < 0.3, rng.random() < 0.4
        return {"kind": kind, "n": _log(rng, 1, 20000 if fp64 else 100000), "phi": phi, "angular": angular,
                "fp64": fp64}
    if kind == "melt":
        return {"kind": kind, "chains": _log(rng, 16, 512), "beads": _log(rng, 32, 512)}
    if kind == "langevin":
        return {"kind": kind, "n": _log(rng, 200, 16000), "phi": phi, "tol": 1e-3, "iters": 26}
    if kind == "sqrt":
        fp64 = rng.random() < 0.3
        return {"kind": kind, "n": _log(rng, 100, 1500 if fp64 else 20000), "phi": phi, "angular": rng.random() < 0.5,
                "fp64": fp64, "tol": 1e-8 if fp64 else rng.choice([1e-3, 1e-4]), "iters": 80 if fp64 else 40}
    if kind == "grad":
        angular = rng.random() < 0.5
        return {"kind": kind, "n": _log(rng, 200, 40000 if angular else 80000), "phi": phi, "angular": angular}
    if kind == "wall":
        return {"kind": kind, "n": _log(rng, 500, 65000), "rho": rng.choice([0.1, 0.01, 0.001])}
    if kind == "rollers":
        return {"kind": kind, "n": _log(rng, 500, 32768), "iters": 10}
    return {"kind": kind, "systems": rng.randint(1, 256), "nmin": 16, "nmax": _log(rng, 64, 4096),
            "steps": rng.randint(1, 4), "iters": 38}


def _cuda(x):
    return None if x is None else torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _cube(case, seed):
    """The suspension of a step, sqrt, langevin, grad or wall case, on the host."""
    fp32 = not case.get("fp64", False)
    if case["kind"] == "melt":
        return inputs.polymer_melt(seed, case["chains"], case["beads"])
    if case["kind"] == "wall":
        return inputs.wall_suspension(seed, case["n"], case["rho"])
    return inputs.cube_suspension(seed, case["n"], case["phi"], angular=case.get("angular", False), fp32=fp32)


def _layer(case, seed):
    """Rollers (Sec. 5.1 of the paper): positions, and the torque and weight on each."""
    w = inputs.ROLLERS_N32768
    pos = inputs.roller_monolayer(seed, case["n"], w["a"], w["area_fraction"])
    T = np.zeros_like(pos)
    T[:, 1] = 8.0 * math.pi * w["eta"] * w["a"] ** 3 * w["omega"]
    return pos, T, w["kT"] / ((w["h_g"] - 1.0) * w["a"])


def _batch(case, seed):
    """The batch's sizes and volume fractions belong to the case, the positions to the seed."""
    w = inputs.BATCH_BD_256
    b = inputs.batch_suspensions(w["seed"], case["systems"], case["nmin"], case["nmax"])
    side = [inputs.box_side(int(n), phi) for n, phi in zip(b.sizes, b.phi)]
    u = np.random.default_rng(seed).uniform(-0.5, 0.5, size=b.pos.shape)
    b.pos = (u * np.repeat(side, b.sizes)[:, None]).astype(np.float32)
    return b


def prepare(case, seed):
    """Inputs on the GPU and the solver that a program keeps over its steps."""
    kind = case["kind"]
    st = {"case": case, "seed": seed}
    if kind == "batch":
        b = _batch(case, seed)
        st["pos"] = _cuda(b.pos)
        st["batch"] = lm.lm_batch_create(b.offsets, inputs.BATCH_BD_256["eta"], b.a,
                                         cuda_stream=torch.cuda.current_stream().cuda_stream)
        return st
    if kind == "rollers":
        pos, T, weight = _layer(case, seed)
        w = inputs.ROLLERS_N32768
        st.update(pos=_cuda(pos), T=_cuda(T), weight=weight)
        st["nbody"] = lm.NBody(w["eta"], w["a"], includeAngular=True, periodicityZ="single_wall")
        return st
    s = _cube(case, seed)
    angular = s.T is not None
    precision = lm.LM_FP64 if case.get("fp64") else lm.LM_FP32C
    st.update(pos=_cuda(s.pos), F=_cuda(s.F), T=_cuda(s.T))
    if kind in ("sqrt", "langevin"):
        st["W"] = _cuda(s.W)
    if kind == "grad":
        st.update(G=_cuda(s.G), H=_cuda(s.H))
        for leaf in (st["pos"], st["F"], st["T"]):
            if leaf is not None:
                leaf.requires_grad_()
    st["nbody"] = lm.NBody(1.0, s.a, includeAngular=angular, precision=precision,
                           periodicityZ="single_wall" if kind == "wall" else "open")
    return st


_LANGEVIN = dict(kT=1.0, dt=1e-3)


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        b, w = st["batch"], inputs.BATCH_BD_256
        lm.lm_batch_set_positions(b, st["pos"])
        lm.lm_batch_bd_run(b, w["kT"], w["dt"], w["k_trap"], case["steps"], seed=st["seed"], tol=w["tol"])
        return lm.lm_batch_get_positions(b, like=st["pos"])
    nb = st["nbody"]
    if kind == "grad":
        X, F, T = st["pos"], st["F"], st["T"]
        u, w = lm.mobility(nb.solver, X, F, T)
        if T is None:
            return (u.detach(), *torch.autograd.grad([u], [X, F], [st["G"]]))
        return (u.detach(), w.detach(), *torch.autograd.grad([u, w], [X, F, T], [st["G"], st["H"]]))
    nb.setPositions(st["pos"])
    if kind in ("step", "melt", "wall"):
        return nb.Mdot(st["F"], st["T"])
    if kind == "sqrt":
        return nb.sqrtMdotW(st["W"], tol=case["tol"], max_iter=200)
    if kind == "langevin":
        return lm.lm_langevin_velocities(nb.solver, st["F"], None, W=st["W"], tol=case["tol"], **_LANGEVIN)[:2]
    w = inputs.ROLLERS_N32768
    F = lm.lm_soft_repulsion(nb.solver, 4.0 * w["kT"], 0.1 * w["a"], 2.0 * w["a"], w["a"], like=st["pos"])
    F[:, 2] -= st["weight"]
    v, omega = nb.LangevinVelocities(w["dt"], w["kT"], F, st["T"], seed=st["seed"], tol=w["tol"])
    return F, v, omega


def work(case):
    kind = case["kind"]
    if kind == "batch":
        # expected systems: sizes log-uniform in [nmin, nmax]
        lo, hi = case["nmin"], case["nmax"]
        ln = math.log(hi / lo)
        n1, n2 = (hi - lo) / ln, (hi ** 2 - lo ** 2) / (2.0 * ln)
        n, pairs = case["systems"] * n1, case["systems"] * n2 * (case["iters"] + 1) * case["steps"]
        c, a = _FLOPS["open", False]
        return {"bytes": 24.0 * n, "flops": pairs * (0.5 * c + a)}
    n = case["chains"] * case["beads"] if kind == "melt" else case["n"]
    angular = kind in ("melt", "rollers") or case.get("angular", False)
    size = 8 if case.get("fp64") else 4
    c, a = _FLOPS["wall" if kind in ("wall", "rollers") else "open", angular]
    flops = float(n) * n * (0.5 * c + a)
    vectors = 2 if angular else 1
    bytes_ = 3.0 * n * size * (1 + 2 * vectors)               # positions, [F; T] in, [u; w] out
    if kind == "sqrt":
        flops, bytes_ = flops * case["iters"], 3.0 * n * (size + vectors * (8 + size))
    elif kind == "langevin":
        flops, bytes_ = flops * (1 + case["iters"]), bytes_ + 24.0 * n
    elif kind == "grad":
        c, a = _FLOPS["adjoint", angular]
        flops, bytes_ = flops + float(n) * n * (0.5 * c + a), 3.0 * n * size * (2 + 5 * vectors)
    elif kind == "rollers":
        # two products of the drift sample, the product of the forces, the Lanczos products; steric forces ~20 per pair
        flops, bytes_ = flops * (3 + case["iters"]) + 20.0 * n * n, 3.0 * n * size * 5
    return {"bytes": bytes_, "flops": flops}


# --------------------------------------------------------------------------
# The same in 64 bits with plain torch (radius 1, viscosity 1).
# --------------------------------------------------------------------------
_ROWS = 1 << 26   # pairs evaluated at once


def _blocks(x, y, wall):
    """Displacements d = x_i - x_j and the coefficients (A, B, g, ar, br) of the
    open RPY blocks (far field and overlap), in units of 1/(8 pi eta)."""
    d = x[:, None, :] - y[None, :, :]
    r2 = (d * d).sum(-1)
    near = r2 < 4.0
    r = r2.sqrt()
    q = torch.where(r > 0, 1.0 / r, torch.zeros_like(r))
    q3, q5 = q ** 3, q ** 5
    A = torch.where(near, 4.0 / 3.0 - 0.375 * r, q + (2.0 / 3.0) * q3)
    B = torch.where(near, 0.125 * q, q3 - 2.0 * q5)
    g = torch.where(near, 0.5 - 0.1875 * r, q3)
    ar = torch.where(near, 1.0 - 27.0 / 32.0 * r + 5.0 / 64.0 * r ** 3, -0.5 * q3)
    br = torch.where(near, 9.0 / 32.0 * q - 3.0 / 64.0 * r, 1.5 * q5)
    return d, r, A, B, g, ar, br


def _wall_part(x, y, F):
    """Wall part of u for sources y with forces F: the image system of the
    no-slip plane z = 0 (Swan & Brady 2007)."""
    Rx, Ry = x[:, None, 0] - y[None, :, 0], x[:, None, 1] - y[None, :, 1]
    Rz = x[:, None, 2] + y[None, :, 2]
    u = (Rx * Rx + Ry * Ry + Rz * Rz).rsqrt()
    ex, ey, c, H, al = Rx * u, Ry * u, Rz * u, y[None, :, 2] * u, u * u
    al2, c2 = al * al, c * c
    A = -1 + 2 * H * H - 2 * c * H + al * (2 * c2 - 2 / 3) + al2 * (2 / 3 - 10 / 3 * c2)
    B = -1 - 6 * H * H + 6 * c * H + al * (2 - 10 * c2) + al2 * (70 / 3 * c2 - 10 / 3)
    C = 2 * H + 12 * c * H * H - 12 * c2 * H + al * c * (20 * c2 - 4) + al2 * c * (40 / 3 - 140 / 3 * c2)
    D = 2 * H - 20 / 3 * al2 * c
    E = -4 * H * H - 4 * al * c2 + al2 * (20 * c2 - 8 / 3)
    eF = ex * F[:, 0] + ey * F[:, 1] + c * F[:, 2]
    pe = (B * eF + C * F[:, 2]) * u
    A = A * u
    return torch.stack([A @ F[:, 0] + (pe * ex).sum(1), A @ F[:, 1] + (pe * ey).sum(1),
                        A @ F[:, 2] + (pe * c + (D * eF + E * F[:, 2]) * u).sum(1)], 1)


def _mdot(x, F, T=None, wall=False):
    """[u, w] = M [F; T] (w None without torques)."""
    n = x.shape[0]
    f = torch.ones(n, dtype=x.dtype, device=x.device)
    if wall:
        f, z = x[:, 2].clamp(0.0, 1.0), x[:, 2].clamp(min=1.0)
        x, F = torch.cat([x[:, :2], z[:, None]], 1), F * f[:, None]
    us, ws = [], []
    step = max(1, _ROWS // n)
    for i in range(0, n, step):
        xi = x[i:i + step]
        d, r, A, B, g, ar, br = _blocks(xi, x, wall)
        u = A @ F + (d * (B * (d * F).sum(-1))[:, :, None]).sum(1)
        if wall:
            u = u + _wall_part(xi, x, F)
        if T is not None:
            def cross(V):
                return torch.linalg.cross(V[None].expand_as(d), d)
            u = u + (cross(T) * g[:, :, None]).sum(1)
            ws.append((cross(F) * g[:, :, None]).sum(1) + ar @ T + (d * (br * (d * T).sum(-1))[:, :, None]).sum(1))
        us.append(u * f[i:i + step, None])
    k = 1.0 / (8.0 * math.pi)
    return k * torch.cat(us), (k * torch.cat(ws) if T is not None else None)


def _matrix(x):
    """The dense 3N x 3N mobility (forces only)."""
    n = x.shape[0]
    d, r, A, B, *_ = _blocks(x, x, False)
    M = torch.empty(n, 3, n, 3, dtype=x.dtype, device=x.device)
    for a in range(3):
        for b in range(3):
            M[:, a, :, b] = B * d[:, :, a] * d[:, :, b] + (A if a == b else 0.0)
    return M.reshape(3 * n, 3 * n) / (8.0 * math.pi)


def _lanczos(apply, W, tol, most=200):
    """M^{1/2} W by Lanczos with full reorthogonalisation, stopped as the library
    documents: at the first iterate that changes by less than tol."""
    norm = W.norm()
    V, alpha, beta, z = [W / norm], [], [], None
    for k in range(most):
        w = apply(V[k])
        alpha.append(float(V[k] @ w))
        Q = torch.stack(V)
        for _ in range(2):
            w = w - Q.T @ (Q @ w)
        m = k + 1
        t = np.diag(alpha) + np.diag(beta, 1) + np.diag(beta, -1)
        ev, ec = np.linalg.eigh(t)
        last, z = z, ec @ (np.sqrt(np.maximum(ev, 0.0)) * ec[0])
        if last is not None and np.linalg.norm(z - np.append(last, 0.0)) < tol * np.linalg.norm(z):
            break
        beta.append(float(w.norm()))
        V.append(w / beta[-1])
    return norm * (torch.from_numpy(z).to(W) @ torch.stack(V[:m]))


def _gradient(x, F, T, G, H):
    """dL/dx of L = G.u + H.w: the derivative of each pair term, by autograd on
    the displacement, rows at a time."""
    n = x.shape[0]
    out = torch.zeros_like(x)
    step = max(1, _ROWS // (8 * n))
    for i in range(0, n, step):
        xi = x[i:i + step]
        d, r, A, B, g, ar, br = _blocks(xi, x, False)
        near = r < 2.0
        q = torch.where(r > 0, 1.0 / r, torch.zeros_like(r))
        # derivatives over r, each divided by r
        dA = torch.where(near, -0.375 * q, -q ** 3 - 2.0 * q ** 5)
        dB = torch.where(near, -0.125 * q ** 3, -3.0 * q ** 5 + 10.0 * q ** 7)
        Fi, Gi = F[i:i + step], G[i:i + step]

        def dot(V):
            return (d * V).sum(-1)

        a1, a2, b1, b2 = dot(Gi[:, None]), dot(Fi[:, None]), dot(F[None]), dot(G[None])
        cd = dA * (Gi @ F.T + Fi @ G.T) + dB * (a1 * b1 + a2 * b2)
        s = (B * b1).sum(1)[:, None] * Gi + (B * a1) @ F + (B * b2).sum(1)[:, None] * Fi + (B * a2) @ G
        if T is not None:
            dg = torch.where(near, -0.1875 * q, -3.0 * q ** 5)
            dar = torch.where(near, -27.0 / 32.0 * q + 15.0 / 64.0 * r, 1.5 * q ** 5)
            dbr = torch.where(near, -9.0 / 32.0 * q ** 3 - 3.0 / 64.0 * q, -7.5 * q ** 7)
            Ti, Hi = T[i:i + step], H[i:i + step]
            p = torch.zeros_like(d)
            for v, w in ((Gi, T), (Hi, F), (Ti, G), (Fi, H)):
                p += torch.linalg.cross(v[:, None].expand_as(d), w[None].expand_as(d))
            h1, h2, t1, t2 = dot(Hi[:, None]), dot(Ti[:, None]), dot(T[None]), dot(H[None])
            cd = cd + dar * (Hi @ T.T + Ti @ H.T) + dbr * (h1 * t1 + h2 * t2) + dg * (d * p).sum(-1)
            s = (s + (g * (r > 0))[:, None, :].matmul(p).squeeze(1) + (br * t1).sum(1)[:, None] * Hi + (br * h1) @ T
                 + (br * t2).sum(1)[:, None] * Ti + (br * h2) @ H)
        out[i:i + step] = (cd[:, None, :] @ d).squeeze(1) + s
    return out / (8.0 * math.pi)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "rollers"):
        return None   # their noise is the library's own generator
    n = case["chains"] * case["beads"] if kind == "melt" else case["n"]
    if n * n > 6e9 or (kind in ("sqrt", "langevin") and n > 5000) or (kind == "grad" and case["angular"] and n > 20000):
        return None   # too long in 64 bits
    s = _cube(case, seed)
    x, F, T, W, G, H = (None if v is None else _cuda(v).double() for v in (s.pos, s.F, s.T, s.W, s.G, s.H))
    if kind in ("step", "melt", "wall"):
        return _mdot(x, F, T, wall=kind == "wall")
    if kind == "grad":
        u, w = _mdot(x, F, T)
        dF, dT = _mdot(x, G, H)
        dX = _gradient(x, F, T, G, H)
        return (u, dX, dF) if T is None else (u, w, dX, dF, dT)
    if T is not None:
        def apply(v):
            return torch.stack(_mdot(x, *v.reshape(2, n, 3))).reshape(-1)

        return tuple(_lanczos(apply, W, case["tol"]).reshape(2, n, 3))
    M = _matrix(x)
    y = _lanczos(lambda v: M @ v, W, case["tol"]).reshape(n, 3)
    if kind == "langevin":
        y = _mdot(x, F)[0] + math.sqrt(2.0 * _LANGEVIN["kT"] / _LANGEVIN["dt"]) * y
    return y, None
