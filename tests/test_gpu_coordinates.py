"""Cells and offsets of coordinates where the integer forms of floor and of the
binary64-binary32 conversions can go wrong: on and one ulp beside cell
boundaries and box images, zeros of both signs, subnormal and tiny values,
negative and far images.  Verlet lists bit-exact against all pairs of the
oracle.
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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("images", [0, 1, 3000])
def test_lists_at_special_coordinates(kg, precision, images):
    m = KI.random_walk_melt(50, 20, 0.85, 0.0, 23)
    rl = 2.0 ** (1 / 6) + 0.3
    rng = np.random.default_rng(images)
    x = rng.uniform(0.0, m.box, m.x.shape)
    h = m.box / int(m.box // rl)
    edges = np.arange(int(m.box // rl) + 1) * h
    edges[-1] = m.box
    special = np.concatenate([edges, np.nextafter(edges, 1e9), np.nextafter(edges, -1e9),
                              [0.0, -0.0, 5e-324, -5e-324, 1e-310, 1e-45, -1e-40, 1e-38, -1e-20, 2.0 ** -30]])
    pick = rng.integers(0, 3, x.shape[1])                      # one coordinate of every other monomer
    on = np.arange(0, x.shape[1], 2)
    x[pick[on], on] = rng.choice(special, on.size)
    if images:
        x += m.box * rng.integers(-images, images + 1, x.shape)
    p = kg.make_params([(m.n_chains, m.chain_len, m.box, m.kappa)], precision=precision, seed=1)
    ctx = kg.kg_create(p, 0, None, None)
    try:
        kg.kg_load_config(ctx, 0, x, m.v)
        offs, nbr = kg.kg_get_nlist(ctx, 0, m.M)
    finally:
        kg.kg_destroy(ctx)
    op = O.params(m.n_chains, m.chain_len, m.box, m.kappa, n_exp=12, seed=1, stream=0, dt=0.01)
    oo, on_ = O.nlist(op, x, rl, use_cells=False)
    assert np.array_equal(offs, oo) and np.array_equal(nbr, on_)
