"""The affine chains where their lane split, their ring of stages and their blocks of 32 dimensions change,
with domains whose dimension changes along the horizon, in one chunk and in several, and the convexity test
of the terminal cost in either, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2407_05433_gb300 import eclqr, synth

pytestmark = pytest.mark.gpu
TOL = 1e-9


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2407_05433_gb300 import build as b
    b.build()
    eclqr.load()


def _run(pbs, **kw):
    b = eclqr.Batch(pbs, **kw)
    try:
        b.run()
        return b.results()
    finally:
        b.close()


def _problem(seed, N, n, m):
    q = np.zeros(N + 1, np.int32)
    if n > 2 and m > 2:
        q[N // 2] = 1
    q[N] = min(2, n // 2)
    return synth.make_problem(seed, N, n, m, 0, q)


@pytest.mark.parametrize("n,m", [(1, 1), (4, 2), (5, 3), (8, 3), (9, 4), (16, 8), (17, 5), (32, 10)])
@pytest.mark.parametrize("kw", [{}, {"chunk": 6}, {"team_warps": 1}, {"team_warps": 8}])
def test_chains(n, m, kw):
    pbs = [_problem(3 + N, N, n, m) for N in (1, 2, 5, 6, 7, 31, 32, 33, 65)]
    for pb, r in zip(pbs, _run(pbs, **kw)):
        s = oracle.solve(pb)
        assert s.ok and r["status"] == 0
        for k in ("x", "u", "lam"):
            ref = getattr(s, k)
            e = np.max(np.abs(r[k] - ref)) / max(1.0, np.max(np.abs(ref)))
            assert e <= TOL, (pb.N, k, e)


@pytest.mark.parametrize("chunk", [40, 5])
def test_terminal_cost_has_to_be_convex(chunk):
    pb = _problem(2, 20, 6, 3)
    pb.Q[-1] = -np.eye(6)
    (r,) = _run([pb], chunk=chunk)
    s = oracle.solve(pb)
    assert not s.ok and eclqr.STATUS_NAMES[r["status"]] == oracle.STATUS_NAMES[s.status]
