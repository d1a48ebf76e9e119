"""The captured step loop (rebuild chain and a few steps per pass of a while
node) against one launch per step: the same bits in both precisions, for
numbers of steps that end inside a pass, odd starts (the other gather buffer),
list builds at every few steps and passes without any.
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


def _run(kg, m, calls, one_by_one, **options):
    p = kg.make_params([(m.n_chains, m.chain_len, m.box, m.kappa)], seed=3, fene_qmin=0.01, **options)
    ctx = kg.kg_create(p, 0, None, None)
    try:
        kg.kg_set_potential_schedule(ctx, [kg.stage(2.0, 57, 0.004), kg.stage(5.0, 10 ** 9, 0.004)])
        kg.kg_load_config(ctx, 0, m.x, m.v)
        kg.kg_profile(ctx, one_by_one)           # timing the step kernel launches every step on its own
        out = []
        for n in calls:
            kg.kg_step(ctx, n)
            x, v = np.zeros_like(m.x), np.zeros_like(m.v)
            kg.kg_get_config(ctx, 0, x, v)
            out += [x, v]
        return out
    finally:
        kg.kg_destroy(ctx)


# two threads per monomer and binary64 systems take the loop at every size
@pytest.mark.parametrize("options", [dict(threads_per_monomer=2), dict(precision=0)])
@pytest.mark.parametrize("skin", [0.1, 0.3, 0.8])
def test_loop_matches_one_launch_per_step(kg, options, skin):
    m = KI.random_walk_melt(30, 41, 0.85, 1.0, 17)
    calls = (1, 10, 13, 40, 1, 33, 64, 11)
    a, b = (_run(kg, m, calls, o, skin=skin, **options) for o in (0, 1))
    assert all(np.array_equal(p, q) for p, q in zip(a, b))
