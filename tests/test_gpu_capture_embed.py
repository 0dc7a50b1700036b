"""A captured pass as a part of a larger graph: what eclqr_refine records on a caller's capturing stream can be
cloned and used as a child graph; Batch.capture, whose graph stays its own, records the refinement as a loop."""
import ctypes as ct

import pytest

from paper_2407_05433_gb300 import eclqr, synth

pytestmark = pytest.mark.gpu
RELAXED = 2


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2407_05433_gb300 import build as b
    b.build()
    eclqr.load()


@pytest.fixture(scope="module")
def cudart():
    return ct.CDLL("libcudart.so.13")


def _batch(draws=(3, 0), **kw):
    return eclqr.Batch([synth.config("batched_uneven", index=j) for j in draws], **kw)


@pytest.mark.parametrize("kw", [dict(), dict(kkt_refine=2), dict(riccati_fp32=1)])
def test_a_callers_capture_can_be_a_child_graph_and_be_cloned(cudart, kw):
    import torch
    b = _batch(**kw)
    graph, outer, clone, node, ex = (ct.c_void_p() for _ in range(5))
    try:
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            b.run()
            torch.cuda.synchronize()
            want = [t.clone() for t in (b.x, b.u, b.lam, b.mu, b.resid)]
            raw = ct.c_void_p(s.cuda_stream)
            assert cudart.cudaStreamBeginCapture(raw, RELAXED) == 0
            b.run()
            assert cudart.cudaStreamEndCapture(raw, ct.byref(graph)) == 0
            assert cudart.cudaGraphClone(ct.byref(clone), graph) == 0
            assert cudart.cudaGraphCreate(ct.byref(outer), 0) == 0
            assert cudart.cudaGraphAddChildGraphNode(ct.byref(node), outer, None, ct.c_size_t(0), graph) == 0
            assert cudart.cudaGraphInstantiate(ct.byref(ex), outer, ct.c_ulonglong(0)) == 0
            for t in (b.x, b.u, b.lam, b.mu, b.resid):
                t.zero_()
            assert cudart.cudaGraphLaunch(ex, raw) == 0
            torch.cuda.synchronize()
        for t, w in zip((b.x, b.u, b.lam, b.mu, b.resid), want):
            assert torch.equal(t, w)
    finally:
        if ex.value:
            cudart.cudaGraphExecDestroy(ex)
        for g in (outer, clone, graph):
            if g.value:
                cudart.cudaGraphDestroy(g)
        b.close()


def test_a_batchs_own_graph_holds_the_loop_and_a_callers_does_not():
    """The launches that Batch.capture records do not depend on how many passes are allowed."""
    import torch
    own, callers = [], []
    for most in (1, 8):
        b = _batch(kkt_refine=most)
        try:
            own.append(b.capture())
            before = b.launches()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, capture_error_mode="relaxed"):
                b.run()
            callers.append(b.launches() - before)
            del g
        finally:
            b.close()
    assert own[0] == own[1] and callers[1] > callers[0]


def test_the_switch_is_checked():
    b = _batch()
    try:
        assert eclqr.eclqr_capture_loop(b.h, 2) == eclqr.EINVAL and eclqr.eclqr_capture_loop(None, 1) == eclqr.EINVAL
    finally:
        b.close()
