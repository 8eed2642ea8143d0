"""opts.variant caps the resident CTAs or blocks of every kernel of a call, and
the teams it leaves are as wide as those of a small batch, seen in the launches
that a stream capture records (nothing runs).
"""
import ctypes as C

import numpy as np
import pytest

from synth.configs import CONFIGS, load_mechanism, reactor_states

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _captured(call, stream):
    """(blocks, threads a block) of every kernel that call() launches on the stream."""
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
            params = (C.c_uint32 * 64)()  # the function, then the sizes of the grid and of a block
            ok(cu.cuGraphKernelNodeGetParams_v2(C.c_void_p(node), params))
            grids.append((params[2] * params[3] * params[4], params[5] * params[6] * params[7]))
    ok(cu.cuGraphDestroy(graph))
    return grids


def _setup(name, n, method):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1608_05794_gb300.ck as ck
    gm = ck.load_mechanism(load_mechanism(CONFIGS[name]["mech"]))
    y, p = reactor_states(name, n=n)
    y, p = (torch.as_tensor(np.array(a), device="cuda") for a in (y, p))
    dt, st = torch.full_like(p, 1e-6), torch.empty(n, dtype=torch.int32, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()

    def call(opts):
        return _captured(lambda: getattr(ck, method)(gm, p, y, dt, st, opts=opts, stream=stream), stream)
    return ck, torch.cuda.get_device_properties(0).multi_processor_count, call


@pytest.mark.parametrize("method,opts", [("integrate_rkf45", dict(form=1)), ("integrate_rkf45", dict(form=2)),
                                         ("integrate_ros4", {})])
def test_variant_caps_every_kernel(method, opts):
    ck, sms, call = _setup("small", 60000, method)
    for cap in (1, 2):
        grids = call(ck.SolverOpts.make(variant=cap, **opts))
        assert grids and max(g for g, _ in grids) <= cap * sms, grids
        assert len(grids) == (2 if opts.get("form") == 1 else 1)


def test_capped_teams_are_wide():
    # two warps a reactor are for SMs that are full of teams
    ck, sms, call = _setup("medium", 4000, "integrate_rkf45")
    assert [t for _, t in call(ck.SolverOpts.make(form=2))] == [64]
    assert [t for _, t in call(ck.SolverOpts.make(form=2, variant=3))] == [128]
    ck, sms, call = _setup("medium", 1000, "integrate_rkf45")
    assert [t for _, t in call(ck.SolverOpts.make(form=2))] == [128]
