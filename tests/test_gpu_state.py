"""kg_get_config into every kind of memory gives the same bytes: host arrays,
device memory of the context's GPU (written in place), a device address that
binary64 stores cannot take, outputs that share memory (in the order x, v,
pid), and each output alone.
"""
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


@pytest.mark.parametrize("precision", [0, 1])
def test_state_into_any_memory(kg, precision):
    import torch
    melts = [KI.random_walk_melt(11, 37, 0.85, 1.0, 61), KI.random_walk_melt(25, 41, 0.85, 2.0, 62)]
    p = kg.make_params([(m.n_chains, m.chain_len, m.box, m.kappa) for m in melts], precision=precision, seed=4,
                       fene_qmin=0.01)
    ctx = kg.kg_create(p, 0, None, None)
    try:
        kg.kg_set_potential_schedule(ctx, [kg.stage(2.0, 10 ** 9, 0.004)])
        for i, m in enumerate(melts):
            kg.kg_load_config(ctx, i, m.x, m.v)
        kg.kg_step(ctx, 25)
        get = kg.load().kg_get_config
        for i, m in enumerate(melts):
            x, v, pid = np.zeros((3, m.M)), np.zeros((3, m.M)), np.zeros(m.M, dtype=np.int32)
            kg.kg_get_config(ctx, i, x, v, pid)
            assert np.abs(x - m.x).max() > 0 and np.array_equal(np.sort(pid), np.arange(m.M))
            dx, dv = (torch.zeros(3, m.M, dtype=torch.float64, device="cuda") for _ in range(2))
            dp = torch.zeros(m.M, dtype=torch.int32, device="cuda")
            kg.kg_get_config(ctx, i, dx, dv, dp)
            assert all(np.array_equal(a.cpu().numpy(), b) for a, b in ((dx, x), (dv, v), (dp, pid)))
            one = torch.zeros_like(dv)
            kg.kg_get_config(ctx, i, None, one)
            assert np.array_equal(one.cpu().numpy(), v)
            raw = torch.zeros(24 * m.M + 8, dtype=torch.uint8, device="cuda")
            assert get(ctx, i, raw.data_ptr() + 4, dv.data_ptr(), None) == kg.KG_OK
            assert raw[4:4 + 24 * m.M].cpu().numpy().tobytes() == x.tobytes()
            assert get(ctx, i, dx.data_ptr(), dx.data_ptr(), None) == kg.KG_OK
            assert np.array_equal(dx.cpu().numpy(), v)
    finally:
        kg.kg_destroy(ctx)
