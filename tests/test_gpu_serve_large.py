"""The solve server with many lanes on systems of the single-system path, of
every triangular-solve kernel (resident, streamed, long-row), many right-hand
sides each, so that the applies of one solve run beside other solves' kernels:
every request returns, converged, and a request's steps and solution are those
of the same request alone, bit for bit (its arithmetic is fixed by itself)."""
import time

import numpy as np
import pytest

from paper_1606_00545_gb300 import synth

pytestmark = pytest.mark.gpu

# (stencil, side, ILU level); the small ones take the one-CTA batched path
SYSTEMS = [(27, 60, 0), (5, 280, 1), (7, 41, 0), (27, 34, 1), (7, 48, 1), (5, 98, 1), (7, 16, 0)]
PER_SYSTEM = 8


@pytest.fixture(scope="module")
def H():
    from paper_1606_00545_gb300 import hecgpu
    hecgpu.load_library()
    return hecgpu


def serve(H, mats, lanes, requests):
    """{(system, i): (status, steps, solution)} of keyed requests, in the order given."""
    out = {}
    S = H.Server(lanes=lanes, flags=H.MIXED_FP32)
    for s, A in enumerate(mats):  # resident under its key
        S.submit(A, synth.rhs_uniform(A.n, 40 + s), ilu_k=SYSTEMS[s][2], key=s + 1, tag=10 ** 6)
    ticket = {}
    for s, i in requests:
        t = S.submit(None if i else mats[s], synth.rhs_uniform(mats[s].n, 1000 * s + i),
                     ilu_k=SYSTEMS[s][2], key=s + 1, tag=1000 * s + i)
        ticket[t] = (s, i)
    t0 = time.monotonic()
    left = len(requests) + len(mats)
    while left:
        assert time.monotonic() - t0 < 120, "requests that do not return: %s" % S.stats()
        for r in S.poll(wait_ms=100):
            left -= 1
            if r["ticket"] in ticket:
                s = ticket[r["ticket"]][0]
                out[ticket[r["ticket"]]] = (r["status"], r["iters"],
                                            S.solution(r["ticket"], mats[s].n))
    S.close()
    return out


def test_large_systems_beside_each_other(H):
    mats = [synth.serving_matrix({"stencil": st, "side": side, "k": k, "seed": 60 + i}, 1.0)
            for i, (st, side, k) in enumerate(SYSTEMS)]
    # round-robin over the systems, so that lanes hold different ones
    requests = [(s, i) for i in range(1, PER_SYSTEM + 1) for s in range(len(mats))]
    together = serve(H, mats, 8, requests)
    assert sorted(together) == sorted(requests)
    assert all(v[0] == H.OK for v in together.values()), {k: v[:2] for k, v in together.items()}
    alone = serve(H, mats, 1, [(s, i) for s in range(4) for i in (1, 4, 8)])
    for key, (status, steps, x) in alone.items():
        assert status == H.OK and steps == together[key][1], key
        assert np.array_equal(x, together[key][2]), key
