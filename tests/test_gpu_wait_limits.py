"""A device wait that runs out ends the solve it belongs to: the status is
HEC_ERR_TIMEOUT after the step that met it, not after the budget of steps (each
of which would wait again), and the handles work afterwards.  The wait is made
to run out by a negative spin limit: the applies issue no copy."""
import ctypes as C

import numpy as np
import pytest

from paper_1606_00545_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    from paper_1606_00545_gb300 import hecgpu
    hecgpu.load_library()
    return hecgpu


def system(H, name, blocks):
    """(matrix, its handle, scheduled preconditioner): every triangular-solve kernel."""
    if name == "long":
        A, k, nb, ov, kernel, parts = synth.stencil27_irregular(9, 4, 5), 0, 4, 1, H.TRSV_AUTO, 0
    else:
        A, k, nb, ov = synth.poisson2d_5pt(40), 0, blocks, min(1, blocks - 1)
        kernel = H.TRSV_RESIDENT if name == "resident" else H.TRSV_STREAMED
        parts = {"resident": 0, "streamed": 1, "split": 2}[name]
    M = H.hec_build(A.row_ptr, A.col, A.val)
    P = H.ilu_k_setup(M, k, nb, ov)
    H.level_schedule(P, parts=parts, kernel=kernel)
    return A, M, P


@pytest.mark.parametrize("eager", [False, True])
@pytest.mark.parametrize("name,method,mixed", [
    ("streamed", "GMRES", False), ("streamed", "GMRES", True), ("streamed", "BICGSTAB", False),
    ("streamed", "CG", False), ("split", "BICGSTAB", False), ("resident", "GMRES", False),
    ("resident", "GMRES", True), ("resident", "CG", False), ("long", "GMRES", True)])
def test_timeout_ends_the_solve(H, name, method, mixed, eager):
    import torch
    A, M, P = system(H, name, 1 if method == "CG" else 2)  # CG: a symmetric preconditioner
    b = torch.tensor(synth.rhs_uniform(A.n, 1), device="cuda:0")
    x = torch.zeros_like(b)
    flags = H.X0_ZERO | (H.MIXED_FP32 if mixed else 0) | (H.SOLVE_EAGER if eager else 0)
    o = H.SolveOpts_t(getattr(H, method), flags, -1000)
    inf = H.SolveInfo_t()
    rc = H.load_library().krylov_solve(M.handle, P.handle, b.data_ptr(), x.data_ptr(), 1e-8, 20000,
                                       30, C.byref(o), None, C.byref(inf))
    assert rc == H.ERR_TIMEOUT and inf.status == H.ERR_TIMEOUT
    assert inf.iters <= 1 and inf.kernel_launches < 40
    assert H.hec_precond_status(P) == H.ERR_TIMEOUT
    info = H.krylov_solve(M, P, b, x, tol=1e-8, maxit=2000, restart=30, method=getattr(H, method),
                          flags=flags)
    assert info["status"] == H.OK and info["rel_resid"] <= 1e-8
    assert H.hec_precond_status(P) == H.OK


@pytest.mark.parametrize("name", ["streamed", "split", "resident", "long"])
def test_waits_that_end_while_copies_land(H, name):
    """Limits of a few polls: the waits end while the copies are landing, so
    warps and lanes may see different outcomes.  Every apply returns, with a
    timeout or with the full result, and the next one is right."""
    import torch
    A, M, P = system(H, name, 2)
    r = synth.rhs_uniform(A.n, 1)
    for dt, ap in ((torch.float32, H.hec_precond_apply_f32), (torch.float64, H.hec_precond_apply)):
        rd = torch.tensor(r, dtype=dt, device="cuda:0")
        z0 = torch.empty_like(rd)
        ap(P, rd, z0)
        assert H.hec_precond_status(P) == H.OK
        z = torch.empty_like(rd)
        for limit in [1] * 8 + [2, 3, 4, 6, 8, 12, 16, 24, 32, 64, 128, 256, 1024]:
            ap(P, rd, z, spin_limit=limit)
            st = H.hec_precond_status(P)
            assert st in (H.OK, H.ERR_TIMEOUT)
            if st == H.OK:
                assert torch.equal(z, z0), limit
        ap(P, rd, z)
        assert H.hec_precond_status(P) == H.OK and torch.equal(z, z0)
