"""opts.variant caps the resident CTAs or blocks of every kernel of a call,
seen in the launches that a stream capture records (nothing runs).
"""
import ctypes as C

import numpy as np
import pytest

from synth.configs import CONFIGS, load_mechanism, reactor_states

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _captured_grids(call, stream):
    """Blocks of every kernel that call() launches on the stream."""
    cu = C.CDLL("libcuda.so.1")
    ok = lambda rc: rc == 0 or pytest.fail(f"CUDA driver call: {rc}")  # noqa: E731
    s = C.c_void_p(stream.cuda_stream)
    ok(cu.cuStreamBeginCapture_v2(s, 2))  # relaxed
    graph = C.c_void_p()
    try:
        call()
    finally:
        rc = cu.cuStreamEndCapture(s, C.byref(graph))
    ok(rc)
    count = C.c_size_t()
    ok(cu.cuGraphGetNodes(graph, None, C.byref(count)))
    nodes = (C.c_void_p * count.value)()
    ok(cu.cuGraphGetNodes(graph, nodes, C.byref(count)))
    grids = []
    for node in nodes:
        kind = C.c_int()
        ok(cu.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)))
        if kind.value == 0:  # a kernel
            params = (C.c_uint32 * 64)()  # the function, then the grid's three sizes
            ok(cu.cuGraphKernelNodeGetParams_v2(C.c_void_p(node), params))
            grids.append(params[2] * params[3] * params[4])
    ok(cu.cuGraphDestroy(graph))
    return grids


@pytest.mark.parametrize("method,opts", [("integrate_rkf45", dict(form=1)), ("integrate_rkf45", dict(form=2)),
                                         ("integrate_ros4", {})])
def test_variant_caps_every_kernel(method, opts):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1608_05794_gb300.ck as ck
    gm = ck.load_mechanism(load_mechanism(CONFIGS["small"]["mech"]))
    n = 60000
    y, p = reactor_states("small", n=n)
    y, p = (torch.as_tensor(np.array(a), device="cuda") for a in (y, p))
    dt, st = torch.full_like(p, 1e-6), torch.empty(n, dtype=torch.int32, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for cap in (1, 2):
        o = ck.SolverOpts.make(variant=cap, **opts)
        grids = _captured_grids(lambda: getattr(ck, method)(gm, p, y, dt, st, opts=o, stream=stream), stream)
        assert grids and max(grids) <= cap * sms, grids
        assert len(grids) == (2 if opts.get("form") == 1 else 1)
