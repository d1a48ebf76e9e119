"""A context on its own stream takes inputs that work queued on the default
stream is still producing, and memory that such work still uses.
"""
import numpy as np
import pytest

import kg_inputs as KI

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])        # binary64, mixed
def test_inputs_still_being_computed(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2109_11001_gb300 as kg
    kg.load()
    m = KI.random_walk_melt(30, 41, 0.85, 1.0, 5)
    p = kg.make_params([(m.n_chains, m.chain_len, m.box, m.kappa)], precision=precision, seed=1)
    x, v = torch.from_numpy(m.x).cuda(), torch.from_numpy(m.v).cuda()
    xd, vd = torch.zeros_like(x), torch.zeros_like(v)
    ctx = kg.kg_create(p, 0, None, kg.torch_allocator())
    try:
        torch.cuda.synchronize()
        torch.cuda._sleep(200_000_000)               # ~0.1 s of the default stream
        xd.copy_(x), vd.copy_(v)
        kg.kg_load_config(ctx, 0, xd, vd)
        out, vel = np.zeros_like(m.x), np.zeros_like(m.v)
        kg.kg_get_config(ctx, 0, out, vel)
    finally:
        kg.kg_destroy(ctx)
    assert np.array_equal(out, m.x)
    assert np.array_equal(vel, m.v.astype(np.float32).astype(np.float64) if precision else m.v)
