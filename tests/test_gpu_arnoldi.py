"""GMRES at the sizes where the one-cluster Arnoldi step begins, leaves CTAs
empty, fills a thread's rows unevenly and ends: the solution of a manufactured
system within 1e-6 (true residual 1e-10 on well-conditioned systems), a
breakdown on a NaN, and restarts at the largest basis the cluster form takes
and one beyond it."""
import numpy as np
import pytest

from paper_1606_00545_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    from paper_1606_00545_gb300 import hecgpu
    hecgpu.load_library()
    return hecgpu


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("restart", [1, 8, 32, 33])
@pytest.mark.parametrize("n", [1, 2, 255, 257, 4095, 4097, 8192, 8193])
def test_gmres_sizes(H, n, restart, mixed):
    import torch
    A = synth.tridiagonal(n, seed=3) if n > 1 else synth.CSR([0, 1], [0], [2.0])
    x_true = synth.rhs_uniform(n, 1)
    b = np.zeros(n)
    rows = np.repeat(np.arange(n), np.diff(A.row_ptr))
    np.add.at(b, rows, A.val * x_true[A.col])
    M = H.hec_build(A.row_ptr, A.col, A.val)
    x = torch.zeros(n, dtype=torch.float64, device="cuda:0")
    bd = torch.tensor(b, device="cuda:0")
    fl = H.X0_ZERO | (H.MIXED_FP32 if mixed else 0)
    info = H.krylov_solve(M, None, bd, x, tol=1e-10, maxit=4000, restart=restart, flags=fl)
    assert info["status"] == H.OK and info["rel_resid"] <= 1e-10
    err = np.linalg.norm(x.cpu().numpy() - x_true) / np.linalg.norm(x_true)
    assert err <= 1e-6
    bd[n // 2] = float("nan")
    info = H.krylov_solve(M, None, bd, x, tol=1e-10, maxit=50, restart=restart, flags=fl)
    assert info["status"] == H.BREAKDOWN
