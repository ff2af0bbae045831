"""Renders under stream capture.  Calls that need no scratch (one or two
cameras, native calls of three, every other size) capture without memory nodes,
so that their graph can be instantiated more than once and used as a child
graph; every captured call replays to the bits of the direct one."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import lf_synth  # noqa: E402

pytestmark = pytest.mark.gpu

MEM_ALLOC, MEM_FREE = 10, 11   # CUgraphNodeType
RELAXED = 2                    # CUstreamCaptureMode


def _ok(rc):
    assert rc == 0, f"CUDA driver error {rc}"


def _capture(cu, stream, call):
    """(graph, the types of its nodes) of what `call` does on `stream`."""
    g, n = ctypes.c_void_p(), ctypes.c_size_t()
    _ok(cu.cuStreamBeginCapture_v2(stream, RELAXED))
    call()
    _ok(cu.cuStreamEndCapture(stream, ctypes.byref(g)))
    _ok(cu.cuGraphGetNodes(g, None, ctypes.byref(n)))
    nodes = (ctypes.c_void_p * n.value)()
    _ok(cu.cuGraphGetNodes(g, nodes, ctypes.byref(n)))
    types = []
    for node in nodes:
        t = ctypes.c_int()
        _ok(cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(t)))
        types.append(t.value)
    return g, types


@pytest.mark.parametrize("n,size,scratch", [(1, (256, 192), False), (3, (256, 192), False), (24, (256, 192), True),
                                            (12, (300, 200), False), (40, (500, 331), False), (1, (9, 7), False),
                                            (30, (9, 7), False)])
def test_captured_renders(n, size, scratch):
    from paper_1805_06019_gb300 import rlfc

    U, V, W, H = 4, 4, 256, 192
    lf = torch.from_numpy(lf_synth.make_lightfield(U, V, W, H, [0.0, 0.7], 1.0, preset_id=520)).cuda()
    st = rlfc.Stream(rlfc.encode(lf, U, V, 3, [0, 2, 2], tau_p=2, tau_b=32))
    rng = np.random.default_rng(n)
    uv = torch.from_numpy(np.stack([rng.uniform(0, U - 1, n), rng.uniform(0, V - 1, n)], 1).astype(np.float32)).cuda()
    disp = torch.from_numpy(rng.choice([0.0, 0.7, -1.3], n).astype(np.float32)).cuda()
    want = st.render(uv, disp, *size)
    out = torch.zeros_like(want)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    handle = ctypes.c_void_p(stream.cuda_stream)
    graph, types = _capture(cu, handle, lambda: st.render(uv, disp, *size, out, stream=stream))
    execs = []
    try:
        if not scratch:
            assert MEM_ALLOC not in types and MEM_FREE not in types
        for _ in range(1 if scratch else 2):
            e = ctypes.c_void_p()
            _ok(cu.cuGraphInstantiateWithFlags(ctypes.byref(e), graph, ctypes.c_ulonglong(0)))
            execs.append(e)
        for e in execs:
            for _ in range(2):
                out.zero_()
                torch.cuda.synchronize()
                _ok(cu.cuGraphLaunch(e, handle))
                torch.cuda.synchronize()
                assert torch.equal(out, want)
    finally:
        for e in execs:
            cu.cuGraphExecDestroy(e)
        cu.cuGraphDestroy(graph)
