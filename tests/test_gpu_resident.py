"""The resident MD loop (one cooperative launch of many steps, one thread per
monomer) against one launch per step: the same bits, list rebuilds, re-sorts
and double-bridging sweeps included, at the edges of a block, of a scan
segment and of the number of monomers the GPU holds at once, and with two
contexts stepped from two threads on their own streams.
"""
import threading

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


def _run(kg, melts, one_by_one, skin=0.3, cell_scale=0.0, stream=None, flags=0):
    p = kg.make_params([(m.n_chains, m.chain_len, m.box, m.kappa) for m in melts], seed=9, fene_qmin=0.01, skin=skin,
                       sort_interval=40 if not flags else 10 ** 9, cell_scale=cell_scale, flags=flags)
    ctx = kg.kg_create(p, 0, stream, None)
    try:
        # n = 2, then 5 (another instantiation), a stage change inside a call
        kg.kg_set_potential_schedule(ctx, [kg.stage(2.0, 71, 0.004), kg.stage(5.0, 10 ** 9, 0.004)])
        for i, m in enumerate(melts):
            kg.kg_load_config(ctx, i, m.x, m.v)
        kg.kg_profile(ctx, one_by_one)           # timing the step kernel launches every step on its own
        kg.kg_step(ctx, 1)
        for _ in range(2):
            kg.kg_step(ctx, 60)
            kg.kg_db_sweep_k(ctx, [m.M // 10 for m in melts])
        out = []
        for i, m in enumerate(melts):
            x, v, pid = np.zeros_like(m.x), np.zeros_like(m.v), np.zeros(m.M, dtype=np.int32)
            kg.kg_get_config(ctx, i, x, v, pid)
            out += [x, v, pid]
        return out, kg.kg_profile_read(ctx)[2]
    finally:
        kg.kg_destroy(ctx)


def _capacities():
    """Monomers that the kernel with four threads per monomer holds, and the one with one."""
    import torch
    n = torch.cuda.get_device_properties(0).multi_processor_count
    return 128 * n, 640 * n


# chains x N: the smallest box, one monomer under / over whole blocks, a batch
# of uneven melts, coarse cells (long candidate runs), a large skin
@pytest.mark.parametrize("sizes,skin,scale", [
    ([(8, 37)], 0.3, 0.0), ([(5, 77), (3, 149)], 0.3, 0.0), ([(32, 32)], 0.6, 0.0), ([(25, 41)], 0.4, 0.0),
    ([(40, 50), (25, 120), (90, 20), (11, 97)], 0.3, 0.0), ([(60, 100)], 0.5, 2.5)])
def test_resident_launches_match_one_launch_per_step(kg, sizes, skin, scale):
    melts = [KI.random_walk_melt(c, n, 0.85, 1.0 + 0.5 * i, 700 + i) for i, (c, n) in enumerate(sizes)]
    a, la = _run(kg, melts, 0, skin, scale)
    b, lb = _run(kg, melts, 1, skin, scale)
    assert all(np.array_equal(p, q) for p, q in zip(a, b))
    assert la < lb / 5                           # many steps per launch


# 24 monomers (whole chains) in one cell: more list entries than a set of the small kernel
# keeps; 45: more members than a bucket holds, the counting sort instead
@pytest.mark.parametrize("crowd", [24, 45])
def test_a_crowded_cell(kg, crowd):
    m = KI.random_walk_melt(110, 3, 0.85, 0.0, 51)
    k = np.arange(crowd)
    m.x[:, :crowd] = 0.1 + 0.3 * np.stack([k % 4, k // 4 % 4, k // 16])
    out = []
    for one_by_one in (0, 1):
        p = kg.make_params([(m.n_chains, m.chain_len, m.box, m.kappa)], seed=9, fene_qmin=0.01)
        ctx = kg.kg_create(p, 0, None, None)
        try:
            kg.kg_set_potential_schedule(ctx, [kg.stage(2.0, 10 ** 9, 1e-8)])
            kg.kg_load_config(ctx, 0, m.x, m.v)
            kg.kg_profile(ctx, one_by_one)
            kg.kg_step(ctx, 1)
            kg.kg_step(ctx, 30)                  # starts with the rebuild that the re-sort after a load asks for
            x, v = np.zeros_like(m.x), np.zeros_like(m.v)
            kg.kg_get_config(ctx, 0, x, v)
            F = np.zeros_like(m.x)
            kg.kg_forces(ctx, 0, F)
            out.append((x, v, F))
        finally:
            kg.kg_destroy(ctx)
    assert all(np.array_equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("kind", [0, 1])
def test_both_sides_of_a_capacity(kg, kind):
    cap = _capacities()[kind]
    for extra in (0, 1):                         # every block resident; one block more takes the next kernel
        m = KI.random_walk_melt(cap // 128 + extra, 128, 0.85, 2.0, 31)
        a, la = _run(kg, [m], 0)
        b, lb = _run(kg, [m], 1)
        assert all(np.array_equal(p, q) for p, q in zip(a, b))
        assert la < lb / 5


# one tile of 256 monomers for every block; a few blocks with a second, which
# only the flag asks for
@pytest.mark.parametrize("extra,flags", [(0, 0), (3, 2)])
def test_tiles(kg, extra, flags):
    import torch
    n = torch.cuda.get_device_properties(0).multi_processor_count
    m = KI.random_walk_melt(10 * n + extra, 128, 0.85, 2.0, 33)
    a, la = _run(kg, [m], 0, flags=flags)
    b, lb = _run(kg, [m], 1, flags=flags)
    assert all(np.array_equal(p, q) for p, q in zip(a, b))
    assert la < lb / 5


def test_two_contexts_on_two_threads(kg):
    import torch
    melts = [[KI.random_walk_melt(150, 100, 0.85, 1.5, 41 + k)] for k in range(2)]
    alone = [_run(kg, m, 0)[0] for m in melts]
    got = [None, None]
    streams = [torch.cuda.Stream() for _ in range(2)]

    def work(k):
        for _ in range(5):
            got[k] = _run(kg, melts[k], 0, stream=streams[k].cuda_stream)[0]

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k in range(2):
        assert all(np.array_equal(p, q) for p, q in zip(alone[k], got[k]))
