"""The captured step loop where mixed contexts of one thread per monomer take it,
just above the largest resident size: the same bits as one launch per step, for
passes that end anywhere, odd starts and re-sorts inside a call.
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


@pytest.fixture(scope="module")
def melt(kg):
    import torch
    n = torch.cuda.get_device_properties(0).multi_processor_count
    return KI.random_walk_melt(10 * n + 1, 128, 0.85, 2.0, 33)      # 1280 monomers per SM and one chain


def _run(kg, m, calls, interval, one_by_one):
    p = kg.make_params([(m.n_chains, m.chain_len, m.box, m.kappa)], seed=3, fene_qmin=0.01, sort_interval=interval)
    ctx = kg.kg_create(p, 0, None, None)
    try:
        kg.kg_set_potential_schedule(ctx, [kg.stage(2.0, 71, 0.004), kg.stage(5.0, 10 ** 9, 0.004)])
        kg.kg_load_config(ctx, 0, m.x, m.v)
        kg.kg_profile(ctx, one_by_one)               # timing the step kernel launches every step on its own
        out = []
        for n in calls:
            kg.kg_step(ctx, n)
            x, v = np.zeros_like(m.x), np.zeros_like(m.v)
            kg.kg_get_config(ctx, 0, x, v)
            out += [x, v]
        return out, kg.kg_profile_read(ctx)[1]
    finally:
        kg.kg_destroy(ctx)


# the second: re-sorts at the same steps in both, 30 apart and inside calls (the tests sit at each ten steps)
@pytest.mark.parametrize("calls,interval", [((1, 33, 64, 7, 40), 10 ** 9), ((1, 50, 40, 33), 30)])
def test_loop_matches_one_launch_per_step(kg, melt, calls, interval):
    (a, timed_a), (b, timed_b) = (_run(kg, melt, calls, interval, o) for o in (0, 1))
    assert timed_a == 0 and timed_b == sum(calls)    # launches of their own in the second run only
    assert all(np.array_equal(p, q) for p, q in zip(a, b))
