"""The long-row triangular-solve kernel (FP32 applies of blocks whose factor
rows exceed 8 entries and whose vector fits in shared memory) against the
oracle, entry by entry within the rounding bound of a sequential FP32 sum: a
row's sum in groups of 4 entries per lane and then pairwise has fewer
roundings, so the same bound holds."""
import numpy as np
import pytest

from paper_1606_00545_gb300 import synth
from ras_bound import check_apply

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    from paper_1606_00545_gb300 import hecgpu
    hecgpu.load_library()
    return hecgpu


@pytest.fixture(scope="module")
def orc():
    import oracle
    return oracle


# rows of up to 40 entries (groups of 1 to 16 lanes), of up to 300 (several
# pseudo-levels of 128), dense triangles (one row per level, up to 199
# entries), one row past a group boundary, and blocks of one owned row
CASES = {
    "irregular27_ras4": lambda: (synth.stencil27_irregular(9, 4, 5), 0, 4, 1),
    "powerlaw_300": lambda: (synth.random_powerlaw_rows(900, 3.0, 0.8, 300, seed=4), 0, 3, 1),
    "dense_200": lambda: (synth.random_sparse(200, 1.0, seed=3), 0, 1, 0),
    "dense_13_blocks_13": lambda: (synth.random_sparse(13, 1.0, seed=5), 0, 13, 3),
    "random_ilu2": lambda: (synth.random_sparse(1500, 0.004, seed=2), 2, 2, 1),
}


def _apply(H, P, r):
    import torch
    z = torch.full((len(r),), float("nan"), dtype=torch.float32, device="cuda:0")
    H.hec_precond_apply_f32(P, torch.tensor(r, dtype=torch.float32, device="cuda:0"), z)
    assert H.hec_precond_status(P) == H.OK
    return z.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("case", sorted(CASES))
def test_long_rows_parity(H, orc, case):
    A, k, nb, ov = CASES[case]()
    M = H.hec_build(A.row_ptr, A.col, A.val)
    P = H.ilu_k_setup(M, k, nb, ov)
    H.level_schedule(P)
    lens = [np.diff(P.factor(b)[0]).max() for b in range(nb)]
    assert max(lens) > 9 and P.info()["trsv_resident"] == 0
    R = orc.RAS(A, k, nb, ov)
    for seed in (1, 2):
        r = synth.rhs_uniform(A.n, seed)
        check_apply(orc, R, r, _apply(H, P, r), fp32=True, what=case)
    # the layout query still gives the streamed layout, unchanged
    S = H.ilu_k_setup(M, k, nb, ov)
    H.level_schedule(S, kernel=H.TRSV_STREAMED, parts=1)
    la, lb = P.layout(fp32=True), S.layout(fp32=True)
    assert np.array_equal(la["pack"], lb["pack"]) and np.array_equal(la["chunks"], lb["chunks"])
    # new values of the same pattern: the refilled units equal freshly packed ones
    val2 = np.asarray(A.val) * (1.0 + 0.25 * np.sin(np.arange(A.nnz)))
    H.hec_refactor(M, P, val2)
    M2 = H.hec_build(A.row_ptr, A.col, val2)
    P2 = H.ilu_k_setup(M2, k, nb, ov)
    H.level_schedule(P2)
    r = synth.rhs_uniform(A.n, 3)
    assert np.array_equal(_apply(H, P, r), _apply(H, P2, r))


def test_long_rows_bounded_wait(H):
    """Nothing is issued (negative spin limit): the waits run out, the status
    says so, and the handle works again."""
    import torch
    A, k, nb, ov = CASES["irregular27_ras4"]()
    M = H.hec_build(A.row_ptr, A.col, A.val)
    P = H.ilu_k_setup(M, k, nb, ov)
    H.level_schedule(P)
    r = synth.rhs_uniform(A.n, 1)
    z0 = _apply(H, P, r)
    z = torch.zeros(A.n, dtype=torch.float32, device="cuda:0")
    H.hec_precond_apply_f32(P, torch.tensor(r, dtype=torch.float32, device="cuda:0"), z,
                            spin_limit=-1000)
    assert H.hec_precond_status(P) == H.ERR_TIMEOUT
    assert np.array_equal(_apply(H, P, r), z0)
