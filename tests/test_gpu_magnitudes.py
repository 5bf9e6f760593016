"""Right-hand sides near the ends of the range.  The solves by parity blocks
form sums of mirrored values; where a value is in the range of the tier's
arithmetic, the solve must come out as it does at ordinary magnitudes.  A large
shift c keeps the operator's products in range, so that the right-hand side is
what limits.  Bound: that of the other refined solves, 1e-12."""

import numpy as np
import pytest

from oracle import refined_solve, sem_1d
from paper_2310_00226_gb300.inputs import random_rhs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SMALL, FOLD = ((31, 33, 63), 2), ((271, 257, 263), 2)


def _solved(n3, k, prec, sweeps, residual, scales, rhs, batched=False):
    from paper_2310_00226_gb300 import sem3d
    c = 1e6
    axes = [sem_1d(k, (n + 1) // k, 0.0, 1.0) for n in n3]
    F = np.ones(n3[::-1]) if rhs == "ones" else random_rhs(*n3, seed=3)
    F /= np.abs(F).max()
    ref = refined_solve(F, *axes, c, 1)
    one = torch.from_numpy(F).cuda()
    errs = []
    with sem3d.Plan(*n3, k, (1.0, 1.0, 1.0), c) as p:
        p.set_precision(prec, sweeps)
        if residual:
            p.set_residual(residual)
        for scale in scales:
            f = one * scale
            u = torch.full_like(f, float("nan"))
            sem3d.solve_batched([p], [f], [u]) if batched else p.solve(f, u)
            p.sync_check()
            errs.append(np.abs(u.cpu().numpy() / scale - ref).max() / np.abs(ref).max())
    return errs


@pytest.mark.parametrize("rhs", ["ones", "noise"])
def test_fp64_solve_near_overflow(rhs):
    errs = _solved(*SMALL, "fp64", 1, None, (1.0, 8e307, 1.2e308, 1.7e308), rhs)
    assert np.max(errs) <= 1e-12, errs  # (NaN fails)


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("rhs", ["ones", "noise"])
def test_fp32_solve_near_overflow(rhs, batched):
    errs = _solved(*SMALL, "fp32", 2, None, (1.0, 1.6e38, 1.8e38, 3.3e38), rhs, batched)
    assert np.max(errs) <= 1e-12, errs  # (NaN fails)


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("residual,top", [("fp64", 3e38), ("mixed", 1e38)])
@pytest.mark.parametrize("rhs", ["ones", "noise"])
def test_parity_order_solve_near_overflow(rhs, residual, top, batched):
    # on both sides of the magnitude from which the folded array is scaled, 2^110
    scales = (1.0, 0.999 * 2.0**110, 1.001 * 2.0**110, 6e37, top)
    errs = _solved(*FOLD, "bf16x3", 3, residual, scales, rhs, batched)
    assert np.max(errs) <= 1e-12, errs  # (NaN fails)
