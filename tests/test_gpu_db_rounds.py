"""Commit rounds of a double-bridging sweep where their layout changes, against
the oracle's sequential loop: many swaps in one sweep, chains longer than a
block keeps in registers, uneven melts finished in different rounds, a melt
with no attempts, fewer attempts than a block has threads.
"""
import numpy as np
import pytest

import kg_inputs as KI
import oracle as O

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


@pytest.mark.parametrize("sizes,attempts", [
    ([(400, 10)], [4000]), ([(6, 2500)], [40000]), ([(100, 20), (7, 200), (30, 40)], [3000, 0, 500]),
    ([(60, 30)], [100]), ([(60, 30)], [257])])
def test_sweep_matches_the_sequential_loop(kg, sizes, attempts):
    melts = [KI.random_walk_melt(c, n, 0.85, 0.5, 900 + i) for i, (c, n) in enumerate(sizes)]
    p = kg.make_params([(m.n_chains, m.chain_len, m.box, m.kappa) for m in melts], seed=21, fene_qmin=0.01)
    ctx = kg.kg_create(p, 0, None, None)
    try:
        kg.kg_set_potential_schedule(ctx, [kg.stage(2.0, 10 ** 9, 0.005)])
        for i, m in enumerate(melts):
            kg.kg_load_config(ctx, i, m.x, m.v)
        for sweep in range(2):                   # the second one starts from the first one's topology
            st = kg.kg_db_sweep_k(ctx, attempts)
            want = dict(attempted=0, empty=0, accepted=0)
            for i, m in enumerate(melts):
                x, pid = np.zeros_like(m.x), np.zeros(m.M, dtype=np.int32)
                kg.kg_get_config(ctx, i, x, None, pid)
                q = O.params(m.n_chains, m.chain_len, m.box, m.kappa, n_exp=2.0, seed=21, dt=0.005, stream=i,
                             fene_qmin=0.01)
                if sweep == 0:
                    m.pid = np.arange(m.M, dtype=np.int32)
                s = O.db_sweep(q, m.x, m.v, m.pid, sweep, attempts[i])
                assert np.array_equal(pid, m.pid)
                assert np.array_equal(x, m.x)
                for k, n in zip(want, s):
                    want[k] += n
            assert {k: getattr(st, k) for k in want} == want
        assert want["accepted"] > 0 or sum(attempts) < 1000
    finally:
        kg.kg_destroy(ctx)
