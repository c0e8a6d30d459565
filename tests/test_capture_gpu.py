"""A captured apply is kernel nodes only, so its graph may be cloned, placed in
another graph, instantiated twice at once and used as the body of a
conditional; captures own their scratch and give it back.

The driver's own graph calls are used through ctypes: torch instantiates a
graph once and keeps it."""
import ctypes as C

import numpy as np
import pytest

import workloads as W
from cases import box_layers, cyl_small

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

KERNEL_NODE = 0


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2111_06893_gb300 import build
    build.build()


def cu(name, *args):
    assert getattr(C.CDLL("libcuda.so.1"), name)(*args) == 0, name


def ptr(v=None):
    return C.c_void_p(v)


def capture(stream, calls):
    g = ptr()
    cu("cuStreamBeginCapture_v2", ptr(stream.cuda_stream), 0)
    try:
        for c in calls:
            c()
    finally:
        cu("cuStreamEndCapture", ptr(stream.cuda_stream), C.byref(g))
    return g


def instantiate(g):
    e = ptr()
    cu("cuGraphInstantiateWithFlags", C.byref(e), g, C.c_ulonglong(0))
    return e


def launch(e, stream):
    cu("cuGraphLaunch", e, ptr(stream.cuda_stream))


def node_types(g):
    n = C.c_size_t(0)
    cu("cuGraphGetNodes", g, None, C.byref(n))
    if n.value == 0:
        return []
    nodes = (C.c_void_p * n.value)()
    cu("cuGraphGetNodes", g, nodes, C.byref(n))
    out = []
    for i in range(n.value):
        t = C.c_int(-1)
        cu("cuGraphNodeGetType", ptr(nodes[i]), C.byref(t))
        out.append(t.value)
    return out


def field(n, dtype, seed):
    return torch.tensor(np.random.default_rng(seed).uniform(-1, 1, size=n), dtype=dtype, device="cuda")


def context(kind, stream):
    from paper_2111_06893_gb300 import thermonoise
    if kind == "mesh":
        return thermonoise.setup(cyl_small(4, 2), stream=stream)
    return thermonoise.Context(stream=stream).build_batch([cyl_small(3, 1), box_layers(4), cyl_small(3, 2)])


@pytest.mark.parametrize("kind", ["mesh", "batch"])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_captured_apply_is_an_ordinary_graph(kind, dtype):
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        ctx = context(kind, st)
        u = field(ctx.ndof, dtype, 1)
        ref = ctx.apply_operator(u)
        ref2 = ctx.apply_operator(ref)
        y, y2 = torch.zeros_like(u), torch.zeros_like(u)
        st.synchronize()
        g = capture(st, [lambda: ctx.apply_operator(u, y), lambda: ctx.apply_operator(y, y2)])
        assert set(node_types(g)) == {KERNEL_NODE}
        clone, outer, node = ptr(), ptr(), ptr()
        cu("cuGraphClone", C.byref(clone), g)
        cu("cuGraphCreate", C.byref(outer), 0)
        cu("cuGraphAddChildGraphNode", C.byref(node), outer, None, C.c_size_t(0), g)
        execs = [instantiate(x) for x in (g, g, clone, outer)]
        for x in (g, clone, outer):
            cu("cuGraphDestroy", x)
        for e in execs:
            y.zero_()
            y2.zero_()
            launch(e, st)
            st.synchronize()
            assert torch.equal(y, ref) and torch.equal(y2, ref2)
        for e in execs:
            cu("cuGraphExecDestroy", e)


def test_captured_apply_in_a_conditional_body():
    """An if node whose condition is true by default."""
    st = torch.cuda.Stream()

    class Params(C.Structure):  # CUgraphNodeParams with a conditional node's
        _fields_ = [("type", C.c_int), ("reserved0", C.c_int * 3), ("handle", C.c_ulonglong), ("kind", C.c_int),
                    ("size", C.c_uint), ("graphs", C.POINTER(C.c_void_p)), ("ctx", C.c_void_p),
                    ("rest", C.c_longlong * 26)]

    with torch.cuda.stream(st):
        ctx = context("mesh", st)
        u = field(ctx.ndof, torch.float32, 2)
        ref, y = ctx.apply_operator(u), torch.zeros_like(u)
        st.synchronize()
        outer, handle, cur, node = ptr(), C.c_ulonglong(0), ptr(), ptr()
        cu("cuGraphCreate", C.byref(outer), 0)
        cu("cuCtxGetCurrent", C.byref(cur))
        cu("cuGraphConditionalHandleCreate", C.byref(handle), outer, cur, C.c_uint(1), C.c_uint(1))
        prm = Params(type=13, handle=handle.value, kind=0, size=1, ctx=cur.value)
        assert C.sizeof(prm) == 256
        cu("cuGraphAddNode_v2", C.byref(node), outer, None, None, C.c_size_t(0), C.byref(prm))
        body = ptr(prm.graphs[0])
        cu("cuStreamBeginCaptureToGraph", ptr(st.cuda_stream), body, None, None, C.c_size_t(0), 0)
        ctx.apply_operator(u, y)
        end = ptr()
        cu("cuStreamEndCapture", ptr(st.cuda_stream), C.byref(end))
        assert set(node_types(body)) == {KERNEL_NODE}
        e = instantiate(outer)
        launch(e, st)
        st.synchronize()
        assert torch.equal(y, ref)
        cu("cuGraphExecDestroy", e)
        cu("cuGraphDestroy", outer)


def test_captures_give_their_scratch_back():
    """Many captures one after another, each destroyed before the next: the
    free memory stays where the first one left it (a block is 18 N^2 numbers
    per element, 2 MiB at the least as the device hands it out)."""
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        br = [0.25 * i for i in range(21)]
        from paper_2111_06893_gb300 import thermonoise
        ctx = thermonoise.setup(W.box(br, br, [-0.3 * i for i in range(11)], 4, W.FUSED_SILICA), stream=st)
        u = field(ctx.ndof, torch.float64, 3)
        ref, y = ctx.apply_operator(u), torch.zeros_like(u)
        block = 18 * 25 * 4000 * 8  # 14.4 MB
        st.synchronize()
        left = []
        for _ in range(40):
            g = capture(st, [lambda: ctx.apply_operator(u, y)])
            e = instantiate(g)
            cu("cuGraphDestroy", g)
            y.zero_()
            launch(e, st)
            st.synchronize()
            assert torch.equal(y, ref)
            cu("cuGraphExecDestroy", e)
            st.synchronize()
            left.append(torch.cuda.mem_get_info()[0])
        assert left[0] - left[-1] < 10 * block


def test_first_fp64_apply_beside_a_capture_of_another_stream():
    """The scratch is allocated without disturbing a capture in progress (the
    kernels have run before, on another context: loading them would)."""
    st, other = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(st):
        warm, ctx = context("mesh", st), context("mesh", st)
        u = field(ctx.ndof, torch.float64, 4)
        ref, y = warm.apply_operator(u), torch.zeros_like(u)
        st.synchronize()
        g = capture(other, [lambda: ctx.apply_operator(u, y)])
        assert node_types(g) == []
        cu("cuGraphDestroy", g)
        assert torch.equal(y, ref)
