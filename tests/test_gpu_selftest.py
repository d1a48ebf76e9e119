"""kg_persistent_selftest works in every mixed context, those whose steps take
other launches by default included: a two-step launch that ends, and one in
which a block never arrives.
"""
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


@pytest.mark.parametrize("chains,rho,tpm", [(40, 0.85, 1), (40, 0.85, 2), (400, 0.85, 2), (20, 0.0005, 1)])
def test_selftest(kg, chains, rho, tpm):
    m = KI.random_walk_melt(chains, 50, rho, 1.0, 301)
    p = kg.make_params([(m.n_chains, m.chain_len, m.box, m.kappa)], seed=5, fene_qmin=0.01, threads_per_monomer=tpm)
    ctx = kg.kg_create(p, 0, None, None)
    try:
        kg.kg_set_potential_schedule(ctx, [kg.stage(2.0, 10 ** 9, 0.001)])
        kg.kg_load_config(ctx, 0, m.x, m.v)
        kg.kg_step(ctx, 10)
        assert kg.kg_persistent_selftest(ctx, -1, 1 << 20) == kg.KG_OK
        kg.kg_step(ctx, 10)
        assert kg.kg_persistent_selftest(ctx, 0, 20000) == kg.KG_ERR_TIMEOUT     # block 0 never arrives
        kg.kg_load_config(ctx, 0, m.x, m.v)
        kg.kg_step(ctx, 10)
    finally:
        kg.kg_destroy(ctx)
