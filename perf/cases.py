"""The work that users of libsem3d have it do, as a list of cases to be timed.

Every case goes through the library's public Python entry points (``Plan``,
``Plan.solve``, ``Plan.ch_run``, ``Plan.pcg``, ``solve_batched``) on float64
CUDA tensors, with a plan that a program sets up once and keeps.  The sizes are
those of the workloads in ``paper_2310_00226_gb300/inputs.py`` and ``bench.py``
and of the tests; ``draw`` spreads more of them over the same ranges.

``exact`` recomputes a case in 64-bit torch arithmetic from the 1D matrices of
the method (dense mode products with the eigenvectors numpy finds), without
the library.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2310_00226_gb300 import sem3d

#: Cahn-Hilliard parameters of bench.py (box [0, 2 pi]^3).
CH = {"eps": 0.05, "m": 1.0, "dt": 1e-4, "S": 2.0}


def _solve(name, n, k, prec, sweeps, c=1.0, rhs="smooth", bc="dirichlet", L=(1.0, 1.0, 1.0)):
    d = {"kind": "solve", "nx": n[0], "ny": n[1], "nz": n[2], "k": k, "c": c, "Lx": L[0], "Ly": L[1], "Lz": L[2],
         "bc": bc, "precision": prec, "sweeps": sweeps, "rhs": rhs}
    return dict(d, name=name) if name else d


def listed():
    return [
        # The smallest call: one FP64 solve of the correctness workload (Q^2, 32 elements per axis).
        _solve("fp64_n63", (63, 63, 63), 2, "fp64", 1, c=0.0),
        # FP64 throughout at an ordinary size, for users who want no other arithmetic.
        _solve("fp64_n255", (255, 255, 255), 4, "fp64", 1),
        # The refined split-bf16 solve, the library's fast FP64-accurate path, on a small grid: launches and latency.
        _solve("refined_n63", (63, 63, 63), 4, "bf16x3", 3),
        # The same at an ordinary size.
        _solve("refined_n255", (255, 255, 255), 4, "bf16x3", 3),
        # The same on an uneven box of odd-degree elements, with a rough right-hand side.
        _solve("refined_449x320x383", (449, 320, 383), 3, "bf16x3", 3, c=3.7, rhs="noise", L=(1.5, 1.0, 1.25)),
        # The headline: Q^4, 250 elements per axis, about 1e9 unknowns.
        _solve("refined_n999", (999, 999, 999), 4, "bf16x3", 3),
        # Homogeneous Neumann data (every node is an unknown), the other boundary condition of the paper's Table 1.
        _solve("neumann_321x161x241", (321, 161, 241), 5, "bf16x3", 4, bc="neumann", L=(2.0, 1.0, 1.5)),
        # The paper's single-precision tensor-core arithmetic (Table 10), bare.
        _solve("tf32_n511", (511, 511, 511), 4, "tf32", 0),
        # Many uneven Helmholtz problems at once (the batched workload of inputs.py, a part of it): split-bf16 tier.
        {"name": "batch16_bf16x3", "kind": "batch", "precision": "bf16x3", "sweeps": 3, "problems":
         "63x255x127k2c4.1;383x255x511k4c8.8;383x383x383k3c0.4;511x127x255k2c6.3;383x383x383k6c9.2;255x63x383k4c2.7;"
         "127x127x511k2c7.7;383x383x383k6c5.5;511x511x255k4c1.9;63x63x63k2c3.3;383x255x383k4c0.8;255x511x127k2c9.9;"
         "383x383x383k3c6.1;127x383x63k4c4.6;511x255x511k2c2.2;255x255x255k4c7.0"},
        # The batched workload in the FP32 tier on smaller boxes.
        {"name": "batch8_fp32", "kind": "batch", "precision": "fp32", "sweeps": 2, "problems":
         "63x255x127k2c4.1;255x127x255k4c8.8;191x143x95k6c0.4;127x127x255k2c6.3;239x119x179k3c9.2;255x63x191k4c2.7;"
         "127x255x127k2c7.7;63x63x63k4c5.5"},
        # Cahn-Hilliard time stepping, Q^2, n = 511: nine mode products and two pointwise kernels a step.
        {"name": "ch_n511", "kind": "ch", "nx": 511, "ny": 511, "nz": 511, "k": 2, "steps": 4, "precision": "bf16x3"},
        # Schroedinger problem, preconditioned CG to 1e-10 with the refined split-bf16 solve.
        {"name": "pcg_n383", "kind": "pcg", "nx": 383, "ny": 383, "nz": 383, "k": 4, "amp": 100.0,
         "precision": "bf16x3", "sweeps": 1, "rtol": 1e-10},
    ]


# ------------------------------------------------------------------ draws

def _size(rng, lo, hi, k, bc="dirichlet"):
    """Log-uniform n in [lo, hi] that fits elements of degree k."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    ne = max(2, round(v / k))
    n = ne * k - 1 if bc == "dirichlet" else ne * k + 1
    return n if n <= hi else n - k


def _sizes(rng, lo, hi, k, bc="dirichlet"):
    """Three sizes around one another, as boxes of physical problems have them."""
    mid = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return tuple(_size(rng, max(lo, mid / 1.6), min(hi, mid * 1.6), k, bc) for _ in range(3))


def draw(rng):
    kind = rng.choices(["refined", "fp64", "fp32", "tf32", "neumann", "batch", "ch", "pcg"],
                       [5, 2, 1, 1, 1, 2, 1, 1])[0]
    c = round(rng.uniform(0.0, 10.0), 2)
    L = tuple(round(rng.uniform(0.8, 2.0), 2) for _ in range(3))
    rhs = rng.choice(["smooth", "noise"])
    if kind == "refined":
        k = rng.choice([2, 3, 4, 6])
        return _solve(None, _sizes(rng, 31, 899, k), k, "bf16x3", 3, c, rhs, L=L)
    if kind == "fp64":
        k = rng.choice([2, 3, 4, 5])
        return _solve(None, _sizes(rng, 23, 255, k), k, "fp64", 1, c, rhs, L=L)
    if kind == "fp32":
        k = rng.choice([2, 3, 4])
        return _solve(None, _sizes(rng, 47, 383, k), k, "fp32", 2, c, rhs, L=L)
    if kind == "tf32":
        k = rng.choice([2, 4, 5])
        return _solve(None, _sizes(rng, 63, 767, k), k, "tf32", rng.choice([0, 0, 5]), c, rhs, L=L)
    if kind == "neumann":
        k = rng.choice([4, 5, 6])
        return _solve(None, _sizes(rng, 33, 321, k, "neumann"), k, "bf16x3", 4, max(c, 0.5), rhs, "neumann", L)
    if kind == "batch":
        prec, hi = rng.choice([("bf16x3", 511), ("fp32", 255)])
        probs = []
        for _ in range(rng.randint(2, 12)):
            k = rng.choice([2, 3, 4, 6])
            n = _sizes(rng, 47, hi, k)
            probs.append("%dx%dx%dk%dc%.1f" % (*n, k, rng.uniform(0.0, 10.0)))
        return {"kind": "batch", "precision": prec, "sweeps": 3 if prec == "bf16x3" else 2, "problems": ";".join(probs)}
    if kind == "ch":
        k = rng.choice([2, 4])
        n = _sizes(rng, 95, 511, k)
        return {"kind": "ch", "nx": n[0], "ny": n[1], "nz": n[2], "k": k, "steps": rng.randint(1, 6),
                "precision": "bf16x3"}
    k = rng.choice([2, 4])
    n = _sizes(rng, 63, 383, k)
    return {"kind": "pcg", "nx": n[0], "ny": n[1], "nz": n[2], "k": k, "amp": round(rng.uniform(20.0, 150.0), 1),
            "precision": "bf16x3", "sweeps": rng.choice([0, 1]), "rtol": 1e-10}


def _problems(case):
    out = []
    for text in case["problems"].split(";"):
        n, rest = text.split("k")
        k, c = rest.split("c")
        out.append((tuple(int(v) for v in n.split("x")), int(k), float(c)))
    return out


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _smooth(xyz, bc, seed):
    """Sum of four products of exponentially weighted sines (cosines with
    Neumann data) of a few wavelengths per box, the kind of right-hand side
    the manufactured solutions of inputs.py have."""
    r = np.random.default_rng(seed)
    terms = []
    for x in xyz:
        length = x[-1] + (x[0] if bc == "dirichlet" else 0.0)
        s = x / length
        wave = np.sin if bc == "dirichlet" else np.cos
        terms.append(np.stack([np.exp(r.uniform(-1, 1) * s) * wave(math.pi * r.integers(1, 4) * s) for _ in range(4)]))
    amp = torch.from_numpy(r.uniform(5.0, 40.0, 4)).cuda()
    X, Y, Z = (torch.from_numpy(t).cuda() for t in terms)
    yz = (amp[:, None, None] * Z[:, :, None] * Y[:, None, :]).reshape(4, -1)
    return (yz.T @ X).reshape(len(xyz[2]), len(xyz[1]), len(xyz[0])).contiguous()


def _noise(shape, seed):
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=_gen(seed))


def _n3(case):
    return case["nx"], case["ny"], case["nz"]


def _ch_phi0(case, seed):
    shape = _n3(case)[::-1]
    return torch.rand(shape, dtype=torch.float64, device="cuda", generator=_gen(seed)).sub_(0.5).mul_(0.1)


def _pcg_inputs(case, xyz, seed):
    """V = amp |x - 1/2|^2 on [0,1]^3 and f = 1 plus a small smooth part."""
    X, Y, Z = (torch.from_numpy(np.asarray(x)).cuda() for x in xyz)
    V = case["amp"] * ((Z[:, None, None] - 0.5) ** 2 + (Y[None, :, None] - 0.5) ** 2 + (X[None, None, :] - 0.5) ** 2)
    return V.contiguous(), 1.0 + 0.01 * _smooth(xyz, "dirichlet", seed)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        plans, fs = [], []
        for q, (n, k, c) in enumerate(_problems(case)):
            p = sem3d.Plan(*n, k, (1.0, 1.0, 1.0), c)
            p.set_precision(case["precision"], case["sweeps"])
            plans.append(p)
            fs.append(_noise(p.shape, seed * 1009 + q))
        return {"kind": kind, "plans": plans, "f": fs, "u": [torch.empty_like(f) for f in fs]}
    if kind == "solve":
        p = sem3d.Plan(*_n3(case), case["k"], (case["Lx"], case["Ly"], case["Lz"]), case["c"], case["bc"])
        p.set_precision(case["precision"], case["sweeps"])
        f = _smooth([p.nodes(a) for a in range(3)], case["bc"], seed) if case["rhs"] == "smooth" else _noise(p.shape, seed)
        return {"kind": kind, "plan": p, "f": f, "u": torch.empty_like(f)}
    if kind == "ch":
        p = sem3d.Plan(*_n3(case), case["k"], (2 * math.pi,) * 3, 0.0)
        p.set_precision(case["precision"], 0)
        phi = _ch_phi0(case, seed)
        return {"kind": kind, "plan": p, "phi_nm1": phi, "phi_n": phi.clone(), "steps": case["steps"]}
    p = sem3d.Plan(*_n3(case), case["k"], (1.0, 1.0, 1.0), case["amp"] / 4)
    p.set_precision(case["precision"], case["sweeps"])
    V, f = _pcg_inputs(case, [p.nodes(a) for a in range(3)], seed)
    return {"kind": kind, "plan": p, "V": V, "f": f, "u": torch.empty_like(f), "rtol": case["rtol"]}


def run(state):
    kind = state["kind"]
    if kind == "solve":
        state["plan"].solve(state["f"], state["u"])
        return state["u"]
    if kind == "batch":
        sem3d.solve_batched(state["plans"], state["f"], state["u"])
        return state["u"]
    if kind == "ch":
        # time stepping goes on from where the last call left the fields
        state["plan"].ch_run(state["phi_nm1"], state["phi_n"], state["steps"], CH["eps"], CH["m"], CH["dt"], CH["S"])
        return {"phi_nm1": state["phi_nm1"], "phi_n": state["phi_n"]}
    iterations, _ = state["plan"].pcg(state["V"], state["f"], state["u"], state["rtol"], 200)
    return {"u": state["u"], "iterations": iterations}


# ------------------------------------------------------------------ work

def _products(n, count):
    """Operations of `count` mode products along each axis.  The 1D operators
    of a uniform mesh commute with the reflection of their axis, so a product
    needs n/2 multiply-adds per value (n operations), not n."""
    return count * math.prod(n) * sum(n)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        every = [work({"kind": "solve", "nx": n[0], "ny": n[1], "nz": n[2], "k": k, "sweeps": case["sweeps"]})
                 for n, k, _ in _problems(case)]
        return {key: sum(w[key] for w in every) for key in ("bytes", "flops")}
    n, k = _n3(case), case["k"]
    N = math.prod(n)
    stencil = 2 * 3 * (k + 2) * N
    if kind == "solve":
        s = case["sweeps"]
        return {"bytes": 16 * N, "flops": (1 + s) * _products(n, 2) + s * stencil}
    if kind == "ch":
        return {"bytes": 32 * N, "flops": case["steps"] * (_products(n, 3) + 30 * N)}
    # CG on this potential takes about eight iterations to 1e-10
    s = case["sweeps"]
    return {"bytes": 24 * N, "flops": 8 * ((1 + s) * _products(n, 2) + (1 + s) * stencil + 20 * N)}


# ------------------------------------------------------------------ 64-bit values

def _gll(k):
    P = np.polynomial.legendre.Legendre.basis(k)
    r = np.concatenate(([-1.0], np.sort(P.deriv().roots().real), [1.0]))
    for _ in range(3):  # Newton steps on P_k' (its second derivative from Legendre's equation)
        x = r[1:-1]
        r[1:-1] = x - P.deriv()(x) * (1 - x * x) / (2 * x * P.deriv()(x) - k * (k + 1) * P(x))
    r = 0.5 * (r - r[::-1])
    return r, 2.0 / (k * (k + 1) * P(r) ** 2)


def _axis(n, k, L, bc):
    """Nodes, H = M^-1 S, lumped mass and the eigenbasis (T, T^-1, lambda) of one axis."""
    r, w = _gll(k)
    P = np.polynomial.legendre.Legendre.basis(k)(r)
    D = (P[:, None] / P[None, :]) / (r[:, None] - r[None, :] + np.eye(k + 1))
    np.fill_diagonal(D, 0.0)
    np.fill_diagonal(D, -D.sum(axis=1))
    ne = (n + 1) // k if bc == "dirichlet" else (n - 1) // k
    h = L / ne / 2
    S, M, x = np.zeros((ne * k + 1,) * 2), np.zeros(ne * k + 1), np.zeros(ne * k + 1)
    for e in range(ne):
        s = slice(e * k, e * k + k + 1)
        S[s, s] += (D.T * w) @ D / h
        M[s] += w * h
        x[s] = 2 * h * e + h * (1 + r)
    if bc == "dirichlet":
        S, M, x = S[1:-1, 1:-1], M[1:-1], x[1:-1]
    m = np.sqrt(M)
    S1 = S / m[:, None] / m[None, :]
    lam, Q = np.linalg.eigh((S1 + S1.T) / 2)
    on = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    return {"x": x, "H": on(S / M[:, None]), "M": on(M), "T": on(Q / m[:, None]), "Ti": on(Q.T * m[None, :]), "lam": on(lam)}


def _along(A, U):
    """A[0], A[1], A[2] applied to U (nz, ny, nx) along x, y and z."""
    for a in (0, 1, 2):
        if a == 0:
            U = U @ A[0].T
        elif a == 1:
            U = torch.matmul(A[1], U)
        else:
            U = (A[2] @ U.reshape(U.shape[0], -1)).reshape(U.shape)
    return U


def _apply(ax, U, c):
    """(c + H_x (+) H_y (+) H_z) U."""
    out = U @ ax[0]["H"].T
    out += torch.matmul(ax[1]["H"], U)
    out += (ax[2]["H"] @ U.reshape(U.shape[0], -1)).reshape(U.shape)
    return out.add_(U, alpha=c)


def _lams(ax):
    return ax[2]["lam"][:, None, None] + ax[1]["lam"][None, :, None] + ax[0]["lam"][None, None, :]


def _fast(ax, F, c):
    G = _along([a["Ti"] for a in ax], F)
    return _along([a["T"] for a in ax], G.div_(_lams(ax).add_(c)))


def _direct(n, k, L, c, bc, f, ax=None):
    ax = ax or [_axis(n[a], k, L[a], bc) for a in range(3)]
    u = _fast(ax, f, c)
    if math.prod(n) * sum(n) < 5e11:  # a step of refinement where it is quick
        u += _fast(ax, f - _apply(ax, u, c), c)
    return u


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        if sum(math.prod(n) * sum(n) for n, _, _ in _problems(case)) > 3e12:
            return None
        return [_direct(n, k, (1.0, 1.0, 1.0), c, "dirichlet", _noise(n[::-1], seed * 1009 + q))
                for q, (n, k, c) in enumerate(_problems(case))]
    n, k = _n3(case), case["k"]
    if kind == "solve":
        L, bc = (case["Lx"], case["Ly"], case["Lz"]), case["bc"]
        ax = [_axis(n[a], k, L[a], bc) for a in range(3)]
        f = _smooth([a["x"] for a in ax], bc, seed) if case["rhs"] == "smooth" else _noise(n[::-1], seed)
        return _direct(n, k, L, case["c"], bc, f, ax)
    if kind == "ch":
        ax = [_axis(n[a], k, 2 * math.pi, "dirichlet") for a in range(3)]
        eps, m, dt, S = CH["eps"], CH["m"], CH["dt"], CH["S"]
        lam, Ti, T = _lams(ax), [a["Ti"] for a in ax], [a["T"] for a in ax]
        old = _ch_phi0(case, seed)
        new = old.clone()
        for _ in range(case["steps"]):
            bar = 2 * new - old
            g = bar ** 3 - (1 + S) * bar
            right = _along(Ti, 2 * new - 0.5 * old) - (dt * m / eps) * lam * _along(Ti, g)
            old, new = new, _along(T, right / (1.5 + dt * m * (eps * lam ** 2 + (S / eps) * lam)))
        return {"phi_nm1": old, "phi_n": new}
    ax = [_axis(n[a], k, 1.0, "dirichlet") for a in range(3)]
    c = case["amp"] / 4
    V, f = _pcg_inputs(case, [a["x"] for a in ax], seed)
    M3 = ax[2]["M"][:, None, None] * ax[1]["M"][None, :, None] * ax[0]["M"][None, None, :]
    u, r = torch.zeros_like(f), f.clone()
    p, rz, tiny = None, 0.0, None
    for _ in range(30):  # conjugate gradients to the rounding floor
        z = _fast(ax, r, c)
        new = float((M3 * r * z).sum())
        tiny = tiny or new * 1e-27
        if new <= tiny:
            break
        p = z if p is None else z + (new / rz) * p
        rz = new
        q = _apply(ax, p, 0.0) + V * p
        alpha = rz / float((M3 * p * q).sum())
        u += alpha * p
        r -= alpha * q
    return {"u": u, "iterations": None}
