"""Dilute contexts (many Verlet cells per monomer): device memory in proportion
to the cells at the rate of the plain arrays, and the same bits as one launch
per step, on both sides of the numbers of cells where the route changes.
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


def counting_allocator(kg):
    import torch
    keep, total = {}, [0]

    def alloc(n, user):
        t = torch.empty(int(n), dtype=torch.uint8, device="cuda")
        keep[t.data_ptr()] = t
        total[0] += int(n)
        return t.data_ptr()

    def free(p, user):
        keep.pop(int(p or 0), None)

    B = kg.binding
    a = B.kg_allocator(B.ALLOC_FN(alloc), B.FREE_FN(free), None)
    a._keep = (keep, alloc, free)
    return a, total


def _run(kg, m, one_by_one, flags):
    p = kg.make_params([(m.n_chains, m.chain_len, m.box, m.kappa)], seed=9, fene_qmin=0.01, flags=flags)
    alloc, total = counting_allocator(kg)
    ctx = kg.kg_create(p, 0, None, alloc)
    try:
        used = total[0]
        kg.kg_set_potential_schedule(ctx, [kg.stage(2.0, 10 ** 9, 0.004)])
        kg.kg_load_config(ctx, 0, m.x, m.v)
        kg.kg_profile(ctx, one_by_one)
        kg.kg_step(ctx, 1)
        kg.kg_step(ctx, 120)
        x, v = np.zeros_like(m.x), np.zeros_like(m.v)
        kg.kg_get_config(ctx, 0, x, v)
        return x, v, used
    finally:
        kg.kg_destroy(ctx)


# cells per monomer of 1,000 monomers: 4.1, 8.0, 22 (below and above the buckets' limit), 85, 1250
@pytest.mark.parametrize("rho", [0.1, 0.05, 0.02, 0.004, 0.0003])
@pytest.mark.parametrize("flags", [0, 2])
def test_memory_and_bits(kg, rho, flags):
    m = KI.random_walk_melt(20, 50, rho, 1.0, 3)
    cells = 64 * ((int(m.box / (2.0 ** (1 / 6) + 0.3)) + 3) // 4) ** 3
    x, v, used = _run(kg, m, 0, flags)
    # 40 B a cell for the plain arrays of both grids, the buckets up to 8 cells a monomer, 4 kB a monomer, fixed parts
    assert used < 40 * cells + 650 * min(cells, 8 * m.M + 512) + 4096 * m.M + (4 << 20)
    y, w, _ = _run(kg, m, 1, flags)
    assert np.array_equal(x, y) and np.array_equal(v, w)
