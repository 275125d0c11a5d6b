"""The Gram-Schmidt projections inside GMRES: the launch is sized for a whole
cycle, the vectors are the step's, and the CTAs go to the groups of eight
vectors that the step has.  The steps' solution where that split changes (8, 9,
16, 17 vectors; more rows than CTAs and fewer), and the time of a cycle's first
steps, which must not depend on the length of the cycle."""
import numpy as np
import pytest

from paper_1606_00545_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    from paper_1606_00545_gb300 import hecgpu
    hecgpu.load_library()
    return hecgpu


def system(H, n):
    import torch
    A = synth.tridiagonal(n, seed=3)
    x_true = synth.rhs_uniform(n, 1)
    b = np.zeros(n)
    np.add.at(b, np.repeat(np.arange(n), np.diff(A.row_ptr)), A.val * x_true[A.col])
    return H.hec_build(A.row_ptr, A.col, A.val), torch.tensor(b, device="cuda:0"), x_true


@pytest.mark.parametrize("n", [8193, 20001, 200003])
@pytest.mark.parametrize("restart", [7, 8, 9, 17, 40, 128])
def test_gmres_across_vector_groups(H, n, restart):
    """A well-conditioned system, unpreconditioned, to 1e-10: the solution to 1e-6."""
    import torch
    M, b, x_true = system(H, n)
    x = torch.zeros_like(b)
    info = H.krylov_solve(M, None, b, x, tol=1e-10, maxit=4000, restart=restart, flags=H.X0_ZERO)
    assert info["status"] == H.OK and info["rel_resid"] <= 1e-10
    assert np.linalg.norm(x.cpu().numpy() - x_true) <= 1e-6 * np.linalg.norm(x_true)


def test_first_steps_cost_the_same_in_a_long_cycle(H):
    """Four steps of GMRES(128) and of GMRES(8) do the same work; within 1.5x
    (split by the cycle's groups, 17 of 304 CTAs would read the basis)."""
    import torch
    M, b, _ = system(H, 1500000)
    ms = {}
    for restart in (8, 128):
        x = torch.zeros_like(b)
        t = []
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            H.krylov_solve(M, None, b, x, tol=0.0, maxit=4, restart=restart, flags=H.X0_ZERO)
            e1.record()
            torch.cuda.synchronize()
            t.append(e0.elapsed_time(e1))
        ms[restart] = min(t[1:])
    assert ms[128] <= 1.5 * ms[8], ms
