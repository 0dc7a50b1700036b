"""The integer Riccati sweep by itself, without the refinement that would hide its errors, and at the ends of its
range: values whose condition is far beyond FP64's 2^53, curvature below the sweep's resolution, offsets that
small pivots carry past the columns' scale.  Against the KKT solution of extended precision."""
import os

import numpy as np
import pytest

from oracle import exact
from paper_2407_05433_gb300 import eclqr, synth

pytestmark = pytest.mark.gpu
RAW = dict(refine=0, corr_refine=0, kkt_refine=0)
EPS = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2407_05433_gb300 import build as b
    b.build()
    eclqr.load()


def _errors(pb, **kw):
    """(status, finite, errors of x and u relative to their largest entry, the exact solution)"""
    b = eclqr.Batch([pb], **kw)
    try:
        b.run()
        (r,) = b.results()
    finally:
        b.close()
    e = exact.exact_kkt(pb)
    err = [float(np.max(np.abs(r[k] - e[k])) / np.max(np.abs(e[k]))) for k in ("x", "u")]
    return r["status"], all(np.isfinite(r[k]).all() for k in ("x", "u", "lam")), err, e


def _feasible(pb):
    """c such that the drawn trajectory satisfies the dynamics of changed A and B"""
    pb.c = pb.x_star[1:] - np.einsum("sij,sj->si", pb.A, pb.x_star[:-1]) - np.einsum("sij,sj->si", pb.B, pb.u_star)
    return pb


def _without_control(seed, n, growth, stages):
    """A grows by about growth a stage, and for so many stages nothing can be done about it: P's condition grows
    by at least growth^2 a stage."""
    pb = synth.make_problem(seed, 60, n, 2, 0, 0)
    pb.A = pb.A * growth
    pb.B[8:8 + stages] = 0.0
    return _feasible(pb)


@pytest.mark.parametrize("n,m", [(1, 1), (1, 16), (2, 5), (5, 1), (17, 3), (31, 16), (32, 16)])
@pytest.mark.parametrize("chunk", [40, 7])
def test_dimensions_at_the_edges_without_refinement(n, m, chunk):
    """Without constraint rows, whose elimination has a conditioning of its own."""
    status, _, err, _ = _errors(synth.make_problem(3, 20, n, m, 0, 0, cross=True), chunk=chunk, **RAW)
    assert status == 0 and max(err) <= 1e-9, err


@pytest.mark.parametrize("chunk", [50, 7])
@pytest.mark.parametrize("seed,n", [(6000, 7), (6001, 4)])
@pytest.mark.parametrize("growth,stages", [(2.0, 31), (2.0, 37), (4.0, 13), (4.0, 19)])
def test_values_of_a_condition_beyond_fp64(growth, stages, seed, n, chunk):
    """From 2^52 to 2^76 and more by the growth alone."""
    status, _, err, _ = _errors(_without_control(seed, n, growth, stages), chunk=chunk)
    assert status == 0 and max(err) <= 1e-9, err


@pytest.mark.parametrize("chunk", [50, 7])
@pytest.mark.parametrize("seed,n", [(6000, 7), (6001, 4), (6004, 7)])
@pytest.mark.parametrize("stages", [25, 28])
def test_curvature_below_the_resolution_is_forgotten_not_amplified(stages, seed, n, chunk):
    """A condition of 2^100 to 2^170: the sweep cannot resolve the controls' effect across such a stretch, and
    nor can a rollout in FP64, whose rounding the stretch amplifies by the product of its |A_i|.  The solution is
    off by no more than that (the factor: rounding in 60 stages of n terms)."""
    pb = _without_control(seed, n, 4.0, stages)
    status, finite, err, _ = _errors(pb, chunk=chunk, **RAW)
    grown = np.prod([np.linalg.norm(a, 2) for a in pb.A[8:8 + stages]])
    assert status == 0 and finite
    assert max(err) <= 60 * n * EPS * grown, (err, grown)


@pytest.mark.parametrize("seed", [401, 403, 405])
def test_offsets_that_a_small_pivot_lifts(seed):
    """Two columns of B parallel to 1e-7, cheap controls and linear costs of 1e6 on them: the second pivot is 1e-14 of
    the first and its offset the largest, so that their common exponent is raised.  x is as good as
    the cancellation between large controls allows."""
    n, m = 2 + seed % 9, 3
    pb = synth.make_problem(seed, 20, n, m, 0, 0, cross=False)
    pb.R, pb.rv = pb.R * 1e-10, pb.rv * 1e6
    pb.B[:, :, 1] = pb.B[:, :, 0] + 1e-7 * pb.B[:, :, 1]
    status, _, (ex, eu), e = _errors(_feasible(pb), **RAW)
    size = max(1.0, float(np.max(np.abs(e["u"])) / np.max(np.abs(e["x"]))))
    assert status == 0 and eu <= 1e-9 and ex <= 20 * (n + m) * EPS * size * 8, (ex, eu, size)


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("m", [3, 8, 16])
def test_a_row_that_collects_the_offsets_of_many_small_pivots(m, sign):
    """R's first m - 1 rows are parallel to 2^-26, their linear costs just below a power of two, and the last row is
    coupled to every pivot as strongly as a positive definite R allows: its offset grows with each.  u is -R^{-1} r."""
    k, d = m - 2, 2.0 ** -26 * 1.001
    R = np.ones((m, m))
    R[1:-1, 1:-1] += d * np.eye(k)
    R[-1, -1] = 7.99
    R[-1, 1:-1] = R[1:-1, -1] = 1.0 + 0.97 * np.sqrt(6.99 * d / k)
    pb = synth.make_problem(1, 3, 2, m, 0, 0)
    pb.R[:], pb.B[:], pb.M[:], pb.rv[:] = R, 0.0, 0.0, 0.0
    pb.rv[:, 1:-1] = 0.9999 * sign
    status, _, (ex, eu), _ = _errors(_feasible(pb), **RAW)
    assert status == 0 and ex <= 1e-12 and eu <= m * EPS * np.linalg.cond(R), (ex, eu)


@pytest.mark.parametrize("chunk", [50, 7])
def test_the_sweep_reads_the_triangle_that_was_tested(chunk):
    """A draw in units up to 2^48 apart (golden/near_singular_units.npz) whose reduced terminal Hessian is singular to
    rounding: positive definite by the lower triangle, which the convexity test factors, indefinite by the upper
    one.  Status OK, and the residual at the floor that FP64 sets (8 ulp of every row's |K||w| + |b|)."""
    g = np.load(os.path.join(os.path.dirname(__file__), "golden", "near_singular_units.npz"))
    N, n, m = (int(v) for v in g["dims"])
    pb = synth.ECLQRProblem(N=N, n=n, m=m, **{k: g[k] for k in (
        "p", "q", "A", "B", "c", "C", "D", "d", "E", "e", "Q", "M", "R", "qv", "rv", "s0")})
    b = eclqr.Batch([pb], chunk=chunk)
    try:
        b.run()
        (r,) = b.results()
    finally:
        b.close()
    floor = EPS * float(np.max(exact.residual_scale(pb, exact.exact_kkt(pb))))
    assert r["status"] == 0 and np.isfinite(r["x"]).all() and r["resid"] <= 8 * floor, (r["resid"], floor)
