"""A double-bridging sweep whose candidate capacity is exceeded only once the
drawn swaps are decided (the drawn bond has two partners, the partner bond more
than the library holds), beside a melt of ordinary attempts on many blocks:
the sweep ends at once with KG_ERR_CAPACITY, no swap of any melt is committed,
and after a load the context sweeps as a new one does.
"""
import time

import numpy as np
import pytest

import kg_inputs as KI
import oracle as O

pytestmark = pytest.mark.gpu
CROWD = 52


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


def crowded(box=10.0):
    """Parallel chains of three: chain 0 beside chain 1, and CROWD - 2 more within reach of chain 1 only."""
    x = np.zeros((3, CROWD, 3))
    x[0, 0], x[0, 1] = 1.6, 0.8
    x[0, 2:] = np.linspace(0.0, 0.01, CROWD - 2)[:, None]
    x[2] = 0.96 * np.arange(3)
    x += 4.0
    return np.ascontiguousarray(x.reshape(3, -1)), box


def seed_that_draws_chain_0():
    """Seed whose attempt 0 of sweep 0 in melt 0 draws a bond of chain 0 (two bonds a chain)."""
    for seed in range(1, 1 << 16):
        w = O.philox4x32_10(np.array([0, 0, 0, 1], dtype=np.uint32), np.array([seed, 0], dtype=np.uint32))
        if (((int(w[1]) << 32) | int(w[0])) * 2 * CROWD) >> 64 < 2:
            return seed
    raise AssertionError("no seed")


def _sweep(kg, ctx, attempts, learned):
    return kg.kg_db_sweep_learned_k(ctx, attempts, 0.5) if learned else kg.kg_db_sweep_k(ctx, attempts)


def _pids(kg, ctx, sizes):
    out = []
    for i, m in enumerate(sizes):
        pid = np.zeros(m, dtype=np.int32)
        kg.kg_get_config(ctx, i, None, None, pid)
        out.append(pid)
    return out


@pytest.mark.parametrize("learned", [False, True])
def test_capacity_in_a_partner_set(kg, learned):
    x, box = crowded()
    q = O.params(CROWD, 3, box, 1.0, n_exp=2.0, seed=1, dt=0.005)
    pid = np.arange(3 * CROWD, dtype=np.int32)
    for b in (0, 1):                                 # the drawn bond's set fits, its partner's does not
        assert 0 < O.db_partners(q, x, pid, 0, b) <= kg.KG_DB_CAND_MAX < O.db_partners(q, x, pid, 1, b)
    m = KI.random_walk_melt(400, 20, 0.85, 1.0, 900)
    seed = seed_that_draws_chain_0()
    p = kg.make_params([(CROWD, 3, box, 1.0), (m.n_chains, m.chain_len, m.box, m.kappa)], seed=seed, fene_qmin=0.01)
    sizes, stage = (3 * CROWD, m.M), [kg.stage(2.0, 10 ** 9, 0.005)]

    def load(ctx):
        kg.kg_load_config(ctx, 0, x)
        kg.kg_load_config(ctx, 1, m.x, m.v)
        kg.kg_set_counters(ctx, 0, 0)

    ctx = kg.kg_create(p, 0, None, None)
    try:
        kg.kg_set_potential_schedule(ctx, stage)
        load(ctx)
        want = _sweep(kg, ctx, [0, 4000], learned).accepted
        assert want > 0
        after = _pids(kg, ctx, sizes)
        load(ctx)
        t = time.monotonic()
        with pytest.raises(kg.KGError) as e:
            _sweep(kg, ctx, [1, 4000], learned)
        assert e.value.status == kg.KG_ERR_CAPACITY
        assert time.monotonic() - t < 1.0            # far below any bounded wait
        assert all(np.array_equal(a, np.arange(k)) for a, k in zip(_pids(kg, ctx, sizes), sizes))
        with pytest.raises(kg.KGError):
            _sweep(kg, ctx, [0, 4000], learned)      # refused until the next load
        load(ctx)
        assert _sweep(kg, ctx, [0, 4000], learned).accepted == want
        assert all(np.array_equal(a, b) for a, b in zip(_pids(kg, ctx, sizes), after))
    finally:
        kg.kg_destroy(ctx)
