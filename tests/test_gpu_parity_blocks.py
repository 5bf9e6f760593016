"""Mode products by parity blocks (even and odd modes of the symmetric mesh)
against the FP64 oracle, at the sizes where the halving, the tiles and the
block construction can go wrong: one and two nodes per axis, even and odd n,
n / 2 around the 16- and 32-wide tiles, and axes whose even and odd
eigenvalues nearly coincide (k = 24, n = 383 and k = 14, n = 433: there the
half problems are diagonalised by themselves).  The bound is the one every
refined solve of the library is held to, 1e-12 of the largest value
(max(1e-12, kappa eps) where the conditioning is larger)."""

import numpy as np
import pytest

from oracle import apply_h, refined_solve, sem_1d
from paper_2310_00226_gb300.inputs import random_rhs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRIDS = [
    ((1, 1, 1), 2, "dirichlet"), ((1, 3, 2), 1, "dirichlet"), ((2, 5, 8), 3, "dirichlet"),
    ((31, 32, 33), 1, "dirichlet"), ((63, 65, 61), 2, "dirichlet"), ((62, 32, 95), 3, "dirichlet"),
    ((129, 17, 64), 1, "dirichlet"), ((383, 23, 47), 24, "dirichlet"), ((27, 433, 13), 14, "dirichlet"),
    ((3, 4, 2), 1, "neumann"), ((33, 31, 64), 1, "neumann"), ((23, 342, 12), 11, "neumann"),
]


def kappa(axes, c):
    return (sum(s.lam[-1] for s in axes) + c) / (sum(s.lam[0] for s in axes) + c)


def check(n3, k, bc, prec, sweeps, run):
    L, c = (1.0, 1.3, 0.8), 1.5
    axes = [sem_1d(k, (n + 1) // k if bc == "dirichlet" else (n - 1) // k, 0.0, Lb, bc) for n, Lb in zip(n3, L)]
    F = random_rhs(*n3, seed=sum(n3))
    ref = refined_solve(F, *axes, c, 1)
    from paper_2310_00226_gb300 import sem3d
    with sem3d.Plan(*n3, k, L, c, bc) as p:
        p.set_precision(prec, sweeps)
        f = torch.from_numpy(F).cuda()
        u = torch.full_like(f, float("nan"))
        run(sem3d, p, f, u)
        p.sync_check()
        err = np.abs(u.cpu().numpy() - ref).max() / np.abs(ref).max()
    assert err <= max(1e-12, kappa(axes, c) * np.finfo(float).eps), err


@pytest.mark.parametrize("n3,k,bc", GRIDS)
def test_fp64_solve(n3, k, bc):
    check(n3, k, bc, "fp64", 1, lambda m, p, f, u: p.solve(f, u))


# FP32 tier with two sweeps (by parity blocks): every tile configuration, which
# is pinned per pass shape for the process, on grids of its own.
FP32_GRIDS = [((1, 1, 2), 1), ((5, 8, 11), 3), ((31, 33, 32), 1), ((65, 127, 63), 2), ((129, 19, 255), 2)]


@pytest.mark.parametrize("cfg", range(6))
@pytest.mark.parametrize("n3,k", FP32_GRIDS)
def test_fp32_refined_solve(n3, k, cfg):
    def run(m, p, f, u):
        for a in range(3):
            p.set_tuned_config(a, cfg)
        p.solve(f, u)
    check(n3, k, "dirichlet", "fp32", 2, run)


# Split-bf16 solves in parity order (all axes >= 255): even and odd n, pads in
# either half of the x pitch, output tiles of 128 to 256, both boundary
# conditions, k with and without the vector residuals, k > 8 and Neumann data
# (FP64 residuals), one node more and less than the rule's limit.
FOLD_GRIDS = [
    ((255, 255, 255), 4, "dirichlet"), ((256, 257, 271), 1, "dirichlet"), ((275, 257, 260), 3, "dirichlet"),
    ((254, 255, 289), 1, "dirichlet"), ((323, 255, 259), 2, "dirichlet"), ((266, 256, 261), 5, "neumann"),
    ((269, 259, 299), 10, "dirichlet"),
]


@pytest.mark.parametrize("residual", ["mixed", "fp64"])
@pytest.mark.parametrize("n3,k,bc", FOLD_GRIDS)
def test_refined_solve_in_parity_order(n3, k, bc, residual):
    def run(m, p, f, u):
        p.set_residual(residual)
        p.solve(f, u)
    check(n3, k, bc, "bf16x3", 3 if bc == "dirichlet" else 4, run)


def test_parity_order_with_double_fp32_residuals_and_fp64_fmas():
    # every residual in double-FP32: 2^-48 of the operator's terms, amplified by
    # the conditioning (the bound), and the exact residual in FP64 FMAs
    from paper_2310_00226_gb300 import sem3d
    n3, k, L, c = (255, 259, 267), 4, (1.0, 1.3, 0.8), 1.5
    axes = [sem_1d(k, (n + 1) // k, 0.0, Lb) for n, Lb in zip(n3, L)]
    F = random_rhs(*n3, seed=5)
    f = torch.from_numpy(F).cuda()
    ref = refined_solve(F, *axes, c, 1)
    with sem3d.Plan(*n3, k, L, c) as p:
        p.set_precision("bf16x3", 3)
        for residual, exact, bound in (("df", "fixed", kappa(axes, c) * 2.0**-48), ("mixed", "fp64", 1e-12)):
            p.set_residual(residual)
            p.set_exact_residual(exact)
            u = torch.full_like(f, float("nan"))
            p.solve(f, u)
            p.sync_check()
            assert np.abs(u.cpu().numpy() - ref).max() / np.abs(ref).max() <= bound


def test_batch_of_both_orders_is_bit_identical_to_single_solves():
    from paper_2310_00226_gb300 import sem3d
    probs = [((255, 256, 257), 1), ((63, 95, 127), 2), ((257, 260, 299), 3), ((255, 511, 127), 4), ((263, 255, 255), 4)]
    plans = [sem3d.Plan(*n3, k, (1.0, 1.0, 1.0), 0.5 * q) for q, (n3, k) in enumerate(probs)]
    fs = [torch.from_numpy(random_rhs(*n3, seed=q)).cuda() for q, (n3, _) in enumerate(probs)]
    for residual in ("mixed", "fp64"):
        for p in plans:
            p.set_precision("bf16x3", 3)
            p.set_residual(residual)
        us = [torch.full_like(f, float("nan")) for f in fs]
        sem3d.solve_batched(plans, fs, us)
        plans[0].sync_check()
        for p, f, u in zip(plans, fs, us):
            one = torch.full_like(f, float("nan"))
            p.solve(f, one)
            p.sync_check()
            assert torch.equal(one, u)
    for p in plans:
        p.close()


@pytest.mark.parametrize("ne3", [(1, 1, 1), (2, 3, 1), (45, 2, 3)])
@pytest.mark.parametrize("k", range(1, 10))  # 9: the per-node kernel
def test_neumann_apply_by_elements(k, ne3):
    # tolerance: 1e-13 of the largest possible sum of the terms' magnitudes (at
    # most 3 (2k + 1) roundings of 2^-53, and rows that differ in their last digits)
    from paper_2310_00226_gb300 import sem3d
    L, c = (1.0, 1.4, 0.8), 0.7
    axes = [sem_1d(k, ne, 0.0, Lb, "neumann") for ne, Lb in zip(ne3, L)]
    U = random_rhs(*[ax.n for ax in axes], seed=k)
    u = torch.from_numpy(U).cuda()
    Au = torch.full_like(u, float("nan"))
    with sem3d.Plan(*[ax.n for ax in axes], k, L, c, bc="neumann") as p:
        p.apply(u, Au)
        p.sync_check()
    scale = (sum(abs(ax.H_sparse()).sum(axis=1).max() for ax in axes) + c) * np.abs(U).max()
    assert np.abs(Au.cpu().numpy() - apply_h(U, *axes, c)).max() <= 1e-13 * scale


@pytest.mark.parametrize("k,ne3", [(1, (6, 4, 8)), (1, (150, 3, 2)), (2, (3, 5, 4)), (2, (70, 2, 9)), (4, (2, 3, 2)),
                                   (4, (40, 5, 3)), (4, (33, 2, 2))])
def test_double_fp32_residual_in_pairs(k, ne3):
    # every residual in double-FP32: 2^-48 of the operator's terms, amplified by the conditioning
    from paper_2310_00226_gb300 import sem3d
    L, c = (1.0, 1.3, 0.8), 1.5
    n3 = [k * ne - 1 for ne in ne3]
    axes = [sem_1d(k, ne, 0.0, Lb) for ne, Lb in zip(ne3, L)]
    F = random_rhs(*n3, seed=k)
    f = torch.from_numpy(F).cuda()
    u = torch.full_like(f, float("nan"))
    with sem3d.Plan(*n3, k, L, c) as p:
        p.set_precision("bf16x3", 4)
        p.set_residual("df")
        p.solve(f, u)
        p.sync_check()
    ref = refined_solve(F, *axes, c, 1)
    assert np.abs(u.cpu().numpy() - ref).max() / np.abs(ref).max() <= max(1e-12, kappa(axes, c) * 2.0**-48)


def test_parity_order_where_an_axis_has_more_than_one_tile():
    # the orders launch different numbers of kernels per solve
    from paper_2310_00226_gb300 import sem3d

    def launches(n3):
        f = torch.ones(n3[::-1], dtype=torch.float64, device="cuda")
        u = torch.empty_like(f)
        with sem3d.Plan(*n3, 1, (1.0, 1.0, 1.0), 1.0) as p:
            p.set_precision("bf16x3", 3)
            p.solve(f, u)
            before = p.launch_count()
            p.solve(f, u)
            p.sync_check()
            return p.launch_count() - before

    node, parity = launches((254, 300, 300)), launches((300, 257, 255))
    assert node != parity
    assert launches((255, 256, 256)) == launches((255, 255, 255)) == node
    assert launches((255, 255, 257)) == launches((257, 255, 255)) == launches((255, 257, 256)) == parity


# Two sweeps are the fewest that take parity order; with the mixed schedule the
# first update then goes from the double-FP32 pair straight to FP64, without the
# pair's low parts.  Bound: the error falls from the bare solve's e0 to one
# sweep's e1 (both in node order, measured here) by e1 / e0, and the next sweep
# may do up to four times worse: 4 e1^2 / e0, some 1e-11 (stale or missing low
# parts would be 1e-8).
@pytest.mark.parametrize("n3,k", [((271, 263, 299), 4), ((272, 258, 264), 1), ((257, 275, 260), 3)])
def test_two_sweeps_in_parity_order(n3, k):
    from paper_2310_00226_gb300 import sem3d
    L, c = (1.0, 1.3, 0.8), 1.5
    F = random_rhs(*n3, seed=k)
    ref = refined_solve(F, *[sem_1d(k, (n + 1) // k, 0.0, Lb) for n, Lb in zip(n3, L)], c, 1)
    f = torch.from_numpy(F).cuda()
    u, v = torch.empty_like(f), torch.empty_like(f)
    err = lambda: np.abs(u.cpu().numpy() - ref).max() / np.abs(ref).max()  # noqa: E731
    with sem3d.Plan(*n3, k, L, c) as p:
        e = []
        for sweeps in (0, 1, 2):
            u.fill_(float("nan"))
            p.set_precision("bf16x3", sweeps)
            p.solve(f, u)
            p.sync_check()
            e.append(err())
        assert e[2] <= 4 * e[1] ** 2 / e[0], e
        v.fill_(float("nan"))
        sem3d.solve_batched([p], [f], [v])
        p.sync_check()
        assert torch.equal(u, v)
