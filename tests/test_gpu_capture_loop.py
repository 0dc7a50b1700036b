"""The refinement recorded as a conditional loop: a replay gives the bits of the eager call, for problems that
need no pass, one or several, one group and several, at the pass limit, and in mixed precision."""
import numpy as np
import pytest

from paper_2407_05433_gb300 import eclqr, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2407_05433_gb300 import build as b
    b.build()
    eclqr.load()


def _results(b):
    return [{k: np.array(v) for k, v in r.items()} for r in b.results()]


@pytest.mark.parametrize("kw", [dict(), dict(kkt_refine=1), dict(refine=0), dict(refine_tol=1e-14), dict(riccati_fp32=1)])
@pytest.mark.parametrize("draws", [(3,), (612, 344, 0, 1, 5, 252)])
def test_replay_gives_the_bits_of_the_eager_call(draws, kw):
    b = eclqr.Batch([synth.config("batched_uneven", index=j) for j in draws], **kw)
    try:
        b.run()
        want = _results(b)
        b.capture()
        for _ in range(2):
            for t in (b.x, b.u, b.lam, b.mu, b.eta, b.alpha, b.resid):
                t.zero_()
            b.replay()
            for r, w in zip(_results(b), want):
                for k in w:
                    assert np.array_equal(r[k], w[k], equal_nan=True), k
    finally:
        b.close()
