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

from oracle import refined_solve, sem_1d
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
