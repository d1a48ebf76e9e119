"""A primitive-path call whose first list build meets a cell with more monomers
than the build accepts ends with KG_ERR_CAPACITY, moves nothing, and leaves the
context to work as before; its work space comes from memory that other work
has filled with values that are no indices.
"""
import numpy as np
import pytest

import kg_inputs as KI
from conftest import relaxed_melt

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
def melt():
    return relaxed_melt(110, 11, 1.0, 17)


@pytest.mark.parametrize("precision", [0, 1])        # binary64, mixed
@pytest.mark.parametrize("steps", [0, 2, 20, 21])    # direct passes, captured loop
def test_a_cell_over_capacity(kg, melt, precision, steps):
    import torch
    crowd = 0.1 + 0.5 * np.random.default_rng(3).random(melt.x.shape)      # 1,210 monomers in one cell
    p = kg.make_params([(melt.n_chains, melt.chain_len, melt.box, melt.kappa)], precision=0, seed=3)
    ctx = kg.kg_create(p, 0, torch.cuda.current_stream().cuda_stream, kg.torch_allocator())
    try:
        kg.kg_load_config(ctx, 0, melt.x, melt.v)
        x, y = np.zeros_like(melt.x), np.zeros_like(melt.x)
        lpp, _ = kg.kg_primitive_path(ctx, 0, melt.n_chains, steps, x_out=x, precision=precision)
        kg.kg_load_config(ctx, 0, crowd, melt.v)
        junk = [torch.full((n << 20,), 0x7f, dtype=torch.uint8, device="cuda") for n in (1, 2, 4, 8, 16)]
        torch.cuda.synchronize()
        del junk                                     # blocks that the next allocations are cut from
        with pytest.raises(kg.KGError) as e:
            kg.kg_primitive_path(ctx, 0, melt.n_chains, steps, x_out=y, precision=precision)
        assert e.value.status == kg.KG_ERR_CAPACITY
        assert np.array_equal(y, crowd)
        kg.kg_load_config(ctx, 0, melt.x, melt.v)
        again, _ = kg.kg_primitive_path(ctx, 0, melt.n_chains, steps, x_out=y, precision=precision)
        assert np.array_equal(again, lpp) and np.array_equal(y, x)
    finally:
        kg.kg_destroy(ctx)
