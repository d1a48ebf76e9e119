"""Pairs a little inside the cutoff in the binary64 step, whose binary32 near
test must not lose them whatever the cell side and the skin: one step against
the oracle, with monomer pairs at 1e-6.5 to 1e-4.3 below r_c (relative), in
usual cells and in the largest.
"""
import numpy as np
import pytest

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


def pairs(n, box, seed):
    """n pairs of parallel straight chains of three, each pair a perpendicular vector of almost r_c apart; the
    pairs on distinct sites of a lattice, out of each other's reach."""
    g = np.random.default_rng(seed)
    k = int(box / 6.0)
    assert n <= k ** 3
    site = np.stack(np.unravel_index(g.choice(k ** 3, n, replace=False), (k, k, k)))
    a, b = (v / np.linalg.norm(v, axis=0) for v in g.standard_normal((2, 3, n)))
    b -= a * (a * b).sum(0)
    b /= np.linalg.norm(b, axis=0)
    gap = O.rc() * (1.0 - 10.0 ** g.uniform(-6.5, -4.3, n))
    x = np.empty((3, n, 2, 3))
    first = (site + g.uniform(0.0, 0.05, (3, n))) * (box / k)
    for i in range(3):
        x[:, :, 0, i] = first + 0.97 * i * a
        x[:, :, 1, i] = x[:, :, 0, i] + gap * b
    return np.ascontiguousarray(x.reshape(3, -1))


# box, pairs of chains, skin, cell_scale; the last two: 3 cells of side 66.7 and 400
@pytest.mark.parametrize("box,n,skin,scale", [(60.0, 900, 0.3, 1.0), (60.0, 500, 3.0, 3.0), (200.0, 300, 20.0, 3.0),
                                              (1200.0, 600, 130.0, 3.0)])
def test_no_near_pair_is_lost(kg, box, n, skin, scale):
    x = pairs(n, box, 5)
    v = np.zeros_like(x)
    p = kg.make_params([(2 * n, 3, box, 1.0)], precision=kg.KG_FP64, seed=7, skin=skin, cell_scale=scale)
    ctx = kg.kg_create(p, 0, None, None)
    try:
        kg.kg_set_potential_schedule(ctx, [kg.stage(12.0, 10 ** 9, 0.01)])
        kg.kg_load_config(ctx, 0, x, v)
        kg.kg_step(ctx, 1)
        got = np.zeros_like(v)
        kg.kg_get_config(ctx, 0, None, got)
    finally:
        kg.kg_destroy(ctx)
    q = O.params(2 * n, 3, box, 1.0, n_exp=12.0, seed=7, dt=0.01)
    O.run(q, x, v, 0, 1)
    # forces of a few hundred at most: binary64 rounding of the positions (2^-53 box) times the stiffness, times dt
    assert np.abs(got - v).max() < 0.01 * 1e4 * 2.0 ** -52 * box
