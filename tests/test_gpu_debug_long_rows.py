"""The long-row kernel in the library compiled with HEC_DEBUG: every dependency
slot and row slot of every unit is checked against the block's vector, every
gathered index against n.  Rows of up to 300 entries, units of one and many
rows, dense triangles: no violation, results within the rounding bound.

A process loads one copy of the library, so the debug build runs in a child
process."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import ctypes as C, os, sys
sys.path.insert(0, ROOT); sys.path.insert(0, os.path.join(ROOT, "tests"))
import numpy as np
import torch
from paper_1606_00545_gb300 import build, synth
build.build(debug=True)
from paper_1606_00545_gb300 import hecgpu as H
lib = H.load_library(H.DEBUG_LIB_PATH)
import oracle as orc
orc.build()
from ras_bound import check_apply
torch.cuda.set_device(0)
rec = (C.c_int32 * 8)()
assert lib.hec_debug_record(rec, 1) == H.OK  # a debug build
cases = {
    "irregular27_ras4": (synth.stencil27_irregular(9, 4, 5), 0, 4, 1),
    "powerlaw_300": (synth.random_powerlaw_rows(900, 3.0, 0.8, 300, seed=4), 0, 3, 1),
    "dense_200": (synth.random_sparse(200, 1.0, seed=3), 0, 1, 0),
    "wide_levels": (synth.random_sparse_rows(20000, 11, seed=6), 0, 1, 0),
    "regular27_ilu1": (synth.stencil27_lognormal(12, 1.0, 5), 1, 2, 1),
}
for name, (A, k, nb, ov) in cases.items():
    M = H.hec_build(A.row_ptr, A.col, A.val)
    P = H.ilu_k_setup(M, k, nb, ov)
    H.level_schedule(P)
    assert max(np.diff(P.factor(b)[0]).max() for b in range(nb)) > 9
    r = synth.rhs_uniform(A.n, 3)
    z = torch.full((A.n,), float("nan"), dtype=torch.float32, device="cuda:0")
    H.hec_precond_apply_f32(P, torch.tensor(r, dtype=torch.float32, device="cuda:0"), z)
    st = H._lib.hec_precond_status(P.handle, None)
    assert lib.hec_debug_record(rec, 1) == H.OK
    assert list(rec) == [0] * 8, (name, list(rec))
    assert st == H.OK, (name, st)
    check_apply(orc, orc.RAS(A, k, nb, ov), r, z.double().cpu().numpy(), fp32=True, what=name)
print("DEBUG_LONG_OK")
'''


def test_debug_build_runs_long_rows_without_violations():
    code = "ROOT = %r\n" % ROOT + CHILD
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and "DEBUG_LONG_OK" in r.stdout, (r.stdout[-3000:], r.stderr[-3000:])
