"""Priorities of the two streams of a pruned tree's evaluation.

The far field runs beside the near field, one step more urgent than it, and both stay
within a step of the caller's stream: a server that runs its short requests on urgent
streams must not find their far field behind the long kernels of the others.  The
evaluation is captured into a graph on streams of every priority, and the priorities of
its kernel nodes (which are those of the streams they were captured from) are read back.
"""
import ctypes

import numpy as np
import pytest

from paper_1105_3505_gb300 import build, workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CAPTURE_THREAD_LOCAL = 1
NODE_KERNEL = 0
ATTRIBUTE_PRIORITY = 8


@pytest.fixture(scope="module")
def lfmm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    from paper_1105_3505_gb300 import lfmm as m
    m.load()
    torch.cuda.init()
    return m


def _cu():
    cu = ctypes.CDLL("libcuda.so.1")

    def call(name, *args):
        r = getattr(cu, name)(*args)
        assert r == 0, (name, r)

    return call


def _kernel_priorities(cu, graph):
    n = ctypes.c_size_t(0)
    cu("cuGraphGetNodes", graph, None, ctypes.byref(n))
    nodes = (ctypes.c_void_p * n.value)()
    cu("cuGraphGetNodes", graph, nodes, ctypes.byref(n))
    found = []
    for node in nodes:
        kind = ctypes.c_int(-1)
        cu("cuGraphNodeGetType", ctypes.c_void_p(node), ctypes.byref(kind))
        if kind.value != NODE_KERNEL:
            continue
        value = (ctypes.c_int * 16)()  # the attribute union, 64 bytes
        cu("cuGraphKernelNodeGetAttribute", ctypes.c_void_p(node), ATTRIBUTE_PRIORITY, value)
        found.append(value[0])
    return found


@pytest.mark.parametrize("precision,p", [("mixed", 8), ("df", 16), ("df", 9)])
def test_far_field_one_step_above_near_field(lfmm, precision, p):
    cu = _cu()
    prec = {"mixed": lfmm.LFMM_MIXED, "df": lfmm.LFMM_DF}[precision]
    prob = workloads.uniform_box(4000, 3000, 700, seed=21)
    dev = torch.device("cuda:0")
    s, t, f = (torch.from_numpy(a).to(dev) for a in (prob.src, prob.tgt, prob.f))
    u = torch.empty(t.shape[0], dtype=torch.float64, device=dev)
    torch.cuda.synchronize()
    least, greatest = ctypes.c_int(0), ctypes.c_int(0)
    cu("cuCtxGetStreamPriorityRange", ctypes.byref(least), ctypes.byref(greatest))
    least, greatest = least.value, greatest.value
    assert greatest < least  # smaller is more urgent
    with lfmm.Plan(s, t, opts=lfmm.make_opts(prec, p, 16, tree=lfmm.LFMM_TREE_PRUNED)) as pl:
        want = pl.eval(f).cpu().numpy()
        # up and down the range, so that a plan also changes the priority it used last
        # (the streams outlive the plan, which ends on the one it used last)
        for c in [least, greatest, *range(greatest, least + 1)]:
            stream, graph = ctypes.c_void_p(), ctypes.c_void_p()
            cu("cuStreamCreateWithPriority", ctypes.byref(stream), 1, c)
            cu("cuStreamBeginCapture_v2", stream, CAPTURE_THREAD_LOCAL)
            lfmm.lfmm_eval(pl.handle, f, u, stream.value)
            cu("cuStreamEndCapture", stream, ctypes.byref(graph))
            found = _kernel_priorities(cu, graph)
            cu("cuGraphDestroy", graph)
            assert set(found) == ({c, c - 1} if c > greatest else {c, c + 1}), (c, found)
            # the far field's launches outnumber the near field's one
            assert found.count(min(found)) >= 3, (c, found)
            lfmm.lfmm_eval(pl.handle, f, u, stream.value)
            cu("cuStreamSynchronize", stream)
            assert np.array_equal(u.cpu().numpy(), want)
