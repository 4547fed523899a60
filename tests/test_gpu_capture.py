"""Direct calls recorded into a CUDA graph: every kernel is a plain node (no programmatic edge, on neither of
the call's streams), and the graph computes what the call computes.

The graph is recorded and read through the driver's interface: its edges come with their type there.
"""
import ctypes

import numpy as np
import pytest

from tests import _cases as C

pytestmark = pytest.mark.gpu

THREAD_LOCAL, EDGE_PROGRAMMATIC = 1, 1


class _Edge(ctypes.Structure):
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte),
                ("reserved", ctypes.c_ubyte * 5)]


@pytest.mark.parametrize("kw", [dict(N=32, L=1, B=5, Ly=420, Lx=400),      # probe kernels on the side stream
                                dict(N=32, L=3, B=5), dict(N=128, L=2, B=3), dict(N=256, L=2, B=2)])
def test_captured_call(kw):
    import torch
    from paper_2012_12686_gb300.adorym import Engine
    cuda = ctypes.CDLL("libcuda.so.1")

    def check(rc):
        assert rc == 0, rc

    case = C.small_case(M=1, loss="lsq", seed=61, **kw)
    p = case["problem"]
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    d, b, probe, pos = t(case["delta"]), t(case["beta"]), t(case["probe"].astype(np.complex64)), t(case["pos"])
    meas = 0.5 + torch.rand((p["B"], p["N"], p["N"]), generator=torch.Generator("cuda").manual_seed(1), device="cuda")
    stream = torch.cuda.Stream()
    eng = Engine(0, stream.cuda_stream)
    oid = eng.register_object(d, b)
    out = [torch.zeros((), dtype=torch.float64, device="cuda"), torch.zeros_like(d), torch.zeros_like(b),
           torch.zeros_like(probe), torch.zeros_like(pos), torch.zeros_like(meas)]
    torch.cuda.synchronize()
    eng.loss_grad(p, oid, probe, pos, meas, *out)
    torch.cuda.synchronize()
    ref = [x.cpu().numpy() for x in out]
    for x in out:
        x.zero_()
    torch.cuda.synchronize()

    s, graph, exe, n = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_size_t()
    check(cuda.cuStreamBeginCapture_v2(s, THREAD_LOCAL))
    eng.loss_grad(p, oid, probe, pos, meas, *out)
    check(cuda.cuStreamEndCapture(s, ctypes.byref(graph)))
    check(cuda.cuGraphGetEdges_v2(graph, None, None, None, ctypes.byref(n)))
    ends = [(ctypes.c_void_p * n.value)() for _ in range(2)]
    edges = (_Edge * n.value)()
    check(cuda.cuGraphGetEdges_v2(graph, *ends, edges, ctypes.byref(n)))
    assert n.value >= 5
    assert not [e for e in edges if e.type == EDGE_PROGRAMMATIC]

    check(cuda.cuGraphInstantiateWithFlags(ctypes.byref(exe), graph, ctypes.c_ulonglong(0)))
    check(cuda.cuGraphLaunch(exe, s))
    torch.cuda.synchronize()
    assert eng.check() == 0
    for x, y in zip(out, ref):   # the object gradient is summed in FP64 in any order
        assert C.rel(x.cpu().numpy(), y) <= 1e-6
    check(cuda.cuGraphExecDestroy(exe))
    check(cuda.cuGraphDestroy(graph))
    eng.close()
