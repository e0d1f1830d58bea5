"""hs_keygen captured into the caller's graph: at the f sets it is one kernel
and no allocation, so the graph can be instantiated more than once; the keys
are those of a plain call."""
import ctypes as C

import numpy as np
import pytest

from paper_2512_23969_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ps,count", [("128f", 1), ("128f", 40), ("256f", 7), ("shake-192f", 3), ("robust-128f", 5), ("toy", 9)])
def test_captured_keygen(hs, ps, count):
    import torch
    rt = C.CDLL("libcudart.so.13")
    ok = lambda rc: rc == 0 or pytest.fail("CUDA error %d" % rc)                                  # noqa: E731
    wl = inputs.make(ps, 1, num_keys=count, seed=610 + count)
    seeds = torch.from_numpy(np.ascontiguousarray(wl.seeds)).cuda()
    pk, sk = hs.hs_keygen(ps, seeds)
    got = torch.zeros_like(pk), torch.zeros_like(sk)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph, execs, n = C.c_void_p(), [C.c_void_p(), C.c_void_p()], C.c_size_t()
    stream = C.c_void_p(st.cuda_stream)
    ok(rt.cudaStreamBeginCapture(stream, 1))
    hs.hs_keygen(ps, seeds, pk=got[0], sk=got[1], stream=st)
    ok(rt.cudaStreamEndCapture(stream, C.byref(graph)))
    ok(rt.cudaGraphGetNodes(graph, None, C.byref(n)))
    assert n.value == 1
    for e in execs:
        ok(rt.cudaGraphInstantiate(C.byref(e), graph, C.c_ulonglong(0)))
        for t in got:
            t.zero_()
        torch.cuda.synchronize()
        ok(rt.cudaGraphLaunch(e, stream))
        torch.cuda.synchronize()
        assert torch.equal(got[0], pk) and torch.equal(got[1], sk)
    for e in execs:
        ok(rt.cudaGraphExecDestroy(e))
    ok(rt.cudaGraphDestroy(graph))
