"""The fixed-point residual in each of its three output forms, for every degree
it serves: split bf16 (node order), FP64 (the TF32 tier), FP32 (parity order).
Bound: that of the other refined solves, max(1e-12, kappa eps)."""

import numpy as np
import pytest

from oracle import refined_solve, sem_1d
from paper_2310_00226_gb300.inputs import random_rhs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _error(n3, k, prec, sweeps):
    from paper_2310_00226_gb300 import sem3d
    L, c = (1.0, 1.3, 0.8), 1.5
    axes = [sem_1d(k, (n + 1) // k, 0.0, Lb) for n, Lb in zip(n3, L)]
    F = random_rhs(*n3, seed=k)
    ref = refined_solve(F, *axes, c, 1)
    f = torch.from_numpy(F).cuda()
    u = torch.full_like(f, float("nan"))
    with sem3d.Plan(*n3, k, L, c) as p:
        p.set_precision(prec, sweeps)
        p.set_residual("fp64")  # every residual
        p.solve(f, u)
        p.sync_check()
    kappa = (sum(s.lam[-1] for s in axes) + c) / (sum(s.lam[0] for s in axes) + c)
    return np.abs(u.cpu().numpy() - ref).max() / np.abs(ref).max(), max(1e-12, kappa * np.finfo(float).eps)


@pytest.mark.parametrize("prec,sweeps", [("bf16x3", 3), ("tf32", 8)])
@pytest.mark.parametrize("k", range(1, 9))
def test_split_and_fp64_outputs(k, prec, sweeps):
    err, bound = _error([k * ne - 1 for ne in (5, 3, 7)], k, prec, sweeps)
    assert err <= bound, err


@pytest.mark.parametrize("n3,k", [((257, 255, 256), 1), ((259, 274, 264), 5), ((275, 257, 263), 6), ((258, 265, 279), 7),
                                  ((255, 271, 263), 8)])
def test_fp32_output(n3, k):
    err, bound = _error(n3, k, "bf16x3", 3)
    assert err <= bound, err
