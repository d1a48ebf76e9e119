"""cos(theta) counts at bonds so short that their squares have few digits in
binary32 (1e-24 to 1e-12): the same bins as in binary64.
"""
import numpy as np
import pytest

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


@pytest.mark.parametrize("power", [-12.0, -16.0, -20.0, -22.0, -24.0])
def test_cosines_of_tiny_bonds(kg, power):
    chains, bins, box = 40, 100, 9.0
    g = np.random.default_rng(7)
    b = g.standard_normal((3, chains, 2))
    b *= 10.0 ** g.uniform(power - 0.5, power + 0.5, (1, chains, 2)) / np.sqrt((b * b).sum(0))
    x = np.concatenate([-b[:, :, :1], np.zeros((3, chains, 1)), b[:, :, 1:]], axis=2)   # exact differences
    cs = (b[:, :, 0] * b[:, :, 1]).sum(0) / np.sqrt((b[:, :, 0] ** 2).sum(0) * (b[:, :, 1] ** 2).sum(0))
    at = (cs + 1.0) * 0.5 * bins
    assert np.abs(at - np.rint(at)).min() > 1e-6     # no cosine on an edge
    want = np.bincount(np.floor(at).astype(int), minlength=bins)
    p = kg.make_params([(chains, 3, box, 0.0)], precision=kg.KG_FP64, seed=3)
    ctx = kg.kg_create(p, 0, None, None)
    try:
        kg.kg_load_config(ctx, 0, np.ascontiguousarray(x.reshape(3, -1)), np.zeros((3, 3 * chains)))
        bond, cos = np.zeros(bins), np.zeros(bins)
        # without energies: no state to evaluate
        assert kg.load().kg_observables(ctx, 0, None, None, kg.binding.ptr(bond), kg.binding.ptr(cos), bins) == kg.KG_OK
    finally:
        kg.kg_destroy(ctx)
    assert np.array_equal(cos, want) and bond[0] == 2 * chains
