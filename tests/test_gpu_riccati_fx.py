"""The integer Riccati sweep at the edges of its range: the smallest and largest dimensions, more controls
than states, domains without coordinates, states and controls in very different units, several chunks, and
teams of every size, against the oracle."""
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


def _check(pb, tol=TOL, scale=(1.0, 1.0), ref=None, **kw):
    b = eclqr.Batch([pb], **kw)
    try:
        b.run()
        (r,) = b.results()
    finally:
        b.close()
    s = oracle.solve(ref if ref is not None else pb)
    assert s.ok and r["status"] == 0
    for k, f in (("x", scale[0]), ("u", scale[1])):
        e = np.max(np.abs(r[k] / f - getattr(s, k))) / max(1.0, np.max(np.abs(getattr(s, k))))
        assert e <= tol, (k, e)


def _problem(seed, N, n, m, p, qN, **kw):
    q = np.zeros(N + 1, np.int32)
    q[N] = qN
    return synth.make_problem(seed, N, n, m, p, q, **kw)


@pytest.mark.parametrize("n,m,p,qN", [(1, 1, 0, 0), (1, 16, 3, 1), (2, 5, 5, 2), (5, 1, 0, 1), (7, 3, 3, 7), (17, 3, 1, 4),
                                      (31, 16, 9, 8), (32, 16, 12, 8)])
@pytest.mark.parametrize("chunk", [40, 7])
def test_dimensions_at_the_edges(n, m, p, qN, chunk):
    _check(_problem(3, 20, n, m, p, qN, cross=True), chunk=chunk)


@pytest.mark.parametrize("team", [1, 2, 4, 8])
def test_team_sizes(team):
    _check(_problem(5, 16, 13, 5, 2, 6, cross=True), team_warps=team)


@pytest.mark.parametrize("k", [4, 10])
def test_units_of_states_and_controls(k):
    """States in units of 2^(+-k) and controls of 2^(+-k) (exact scalings) give the same solution in the
    original units; the FP64 stages around the sweep may lose the units' spread, 2^k."""
    pb = _problem(8, 24, 6, 3, 1, 2, cross=True)
    sx = 2.0 ** (k * np.array([1, -1, 0, 1, -1, 0]))
    su = 2.0 ** (k * np.array([-1, 1, 0]))
    sc = pb.copy()
    sc.A = pb.A * sx[None, :, None] / sx[None, None, :]
    sc.B = pb.B * sx[None, :, None] / su[None, None, :]
    sc.c, sc.s0 = pb.c * sx, pb.s0 * sx
    sc.C, sc.D, sc.E = pb.C / sx, pb.D / su, pb.E / sx
    sc.Q = pb.Q / sx[None, :, None] / sx[None, None, :]
    sc.M = pb.M / sx[None, :, None] / su[None, None, :]
    sc.R = pb.R / su[None, :, None] / su[None, None, :]
    sc.qv, sc.rv = pb.qv / sx, pb.rv / su
    _check(sc, tol=TOL * 2.0 ** k, scale=(sx, su), ref=pb, kkt_refine=0)
