"""Calls that take device buffers on a context's own stream, made while the
program captures a blocking stream: the capture stays valid and the calls work.
"""
import ctypes as C

import numpy as np
import pytest

import kg_inputs as KI

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2109_11001_gb300 as kg
    kg.load()
    return kg


def test_capture_of_a_blocking_stream(kg):
    import torch
    m = KI.random_walk_melt(30, 41, 0.85, 1.0, 5)
    p = kg.make_params([(m.n_chains, m.chain_len, m.box, m.kappa)], precision=kg.KG_FP64, seed=1)
    ctx = kg.kg_create(p, 0, None, None)
    x, v = torch.from_numpy(m.x).cuda(), torch.from_numpy(m.v).cuda()
    out, F = torch.zeros_like(x), torch.zeros_like(x)
    kg.kg_load_config(ctx, 0, x, v)
    kg.kg_forces(ctx, 0, F)
    torch.cuda.synchronize()
    cu = C.CDLL("libcuda.so.1")
    stream, graph = C.c_void_p(), C.c_void_p()
    try:
        assert cu.cuStreamCreate(C.byref(stream), 0) == 0                # blocking: ordered with the default stream
        assert cu.cuStreamBeginCapture_v2(stream, 2) == 0                # relaxed: this thread may go on working
        try:
            kg.kg_load_config(ctx, 0, x, v)
            kg.kg_get_config(ctx, 0, out)
            kg.kg_forces(ctx, 0, F)
        finally:
            ended = cu.cuStreamEndCapture(stream, C.byref(graph))
        assert ended == 0
        assert np.array_equal(out.cpu().numpy(), m.x) and float(F.abs().max()) > 0
    finally:
        if graph.value:
            cu.cuGraphDestroy(graph)
        cu.cuStreamDestroy_v2(stream)
        kg.kg_destroy(ctx)
