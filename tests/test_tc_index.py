"""Offsets of the tensor-core passes' output rows in arrays of more than 2^32
entries: the arithmetic on the CPU, and one refined solve whose arrays are
below that limit at the node-order pitch and above it in parity order."""

import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2310_00226_gb300", "csrc")


@pytest.fixture(scope="module")
def row_offset(tmp_path_factory):
    d = tmp_path_factory.mktemp("tc_index")
    src = d / "off.cpp"
    src.write_text('#include "tc_index.h"\nextern "C" unsigned long long off(int pass, int row, int batch, int Px, int ny)'
                   ' { return sem3d::tc_row_offset(pass, row, batch, Px, ny); }\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(d / "off.so")], check=True)
    f = ctypes.CDLL(str(d / "off.so")).off
    f.restype = ctypes.c_ulonglong
    return f


def node_pitch(n):
    return (n + 15) // 16 * 16


def parity_pitch(n):
    return node_pitch(n - n // 2) + node_pitch(n // 2)


@pytest.mark.parametrize("nx,ny,nz", [(1602, 1626, 1626),  # 2^32 between the two pitches
                                      (1999, 1999, 1999), (99, 3999, 19999), (255, 255, 255)])
def test_row_offsets(row_offset, nx, ny, nz):
    for Px in (node_pitch(nx), parity_pitch(nx)):
        for i in (0, 1, nx - 1):
            for l in (0, 1, nz // 2, nz - 1):
                assert row_offset(1, i, l, Px, ny) == i + Px * ny * l
            for j in (0, 1, ny - 1):
                assert row_offset(2, i + Px * j, 0, Px, ny) == i + Px * j
    if nx == 1602:
        assert node_pitch(nx) * ny * nz < 2**32 < parity_pitch(nx) * ny * nz


@pytest.mark.gpu
@pytest.mark.slow
def test_refined_solve_above_2_32_padded_entries():
    # k = 1 with lumped mass: products of sines are the discrete eigenvectors,
    # so the solution is the right-hand side over the sum of the eigenvalues
    # (2 - 2 cos(m pi / (n + 1))) / h^2.  Bound: max(1e-12, kappa eps), that of
    # the other refined solves.
    torch = pytest.importorskip("torch")
    from paper_2310_00226_gb300 import sem3d
    n3, modes, c = (1602, 1626, 1626), (2, 3, 5), 1.0
    if torch.cuda.mem_get_info()[0] < 190e9:
        pytest.skip("needs 190 GB of device memory")
    lam = lambda n, m: (2 - 2 * math.cos(m * math.pi / (n + 1))) * (n + 1) ** 2  # noqa: E731
    s = [torch.sin(torch.arange(1, n + 1, dtype=torch.float64, device="cuda") * (m * math.pi / (n + 1)))
         for n, m in zip(n3, modes)]
    total = sum(lam(n, m) for n, m in zip(n3, modes)) + c
    kappa = sum(lam(n, n) for n in n3) / sum(lam(n, 1) for n in n3)
    plane = s[1][:, None] * s[0][None, :]
    f = torch.empty((n3[2], n3[1], n3[0]), dtype=torch.float64, device="cuda")
    for l in range(n3[2]):
        torch.mul(plane, s[2][l], out=f[l])
    u = torch.full_like(f, float("nan"))
    with sem3d.Plan(*n3, 1, (1.0, 1.0, 1.0), c) as p:
        p.set_precision("bf16x3", 3)
        p.solve(f, u)
        p.sync_check()
    err = max(float((u[l] * total - f[l]).abs().max()) for l in range(n3[2]))
    del f, u
    torch.cuda.empty_cache()
    assert err <= max(1e-12, kappa * np.finfo(float).eps), err
