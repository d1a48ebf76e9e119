"""Observables at the sizes where their kernels change path, against plain
binary64 sums on the same positions: pair counts (exact) in boxes whose cell
stencil wraps or holds every cell, with narrow bins and with r_max on a cell
boundary; S(q) with large wave vectors on far unwrapped positions; <R^2(n)> at
the edges of its lag windows, chunks and shared-memory layout; histograms.
"""
import contextlib

import numpy as np
import pytest

import kg_inputs as KI
import oracle.structure as SF

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


@contextlib.contextmanager
def _ctx(kg, melts):
    p = kg.make_params([(m.n_chains, m.chain_len, m.box, m.kappa) for m in melts], precision=kg.KG_FP64, seed=3)
    ctx = kg.kg_create(p, 0, None, None)
    try:
        for i, m in enumerate(melts):
            kg.kg_load_config(ctx, i, m.x, m.v)
        yield ctx
    finally:
        kg.kg_destroy(ctx)


# r_max as a share of L / 2 (None: two cells of the 1.3 sigma grid); 2048 bins: many pairs near a bin edge
@pytest.mark.parametrize("share,bins", [(1.0, 37), (0.45, 100), (None, 64), (0.3, 2048), (0.02, 2048)])
def test_pair_counts_are_exact(kg, share, bins):
    melts = [KI.random_walk_melt(8, 37, 0.85, 0.0, 5), KI.random_walk_melt(30, 50, 0.85, 2.0, 6),
             KI.random_walk_melt(101, 29, 0.85, 1.0, 7)]
    with _ctx(kg, melts) as ctx:
        for i, m in enumerate(melts):
            r_max = 2 * m.box / int(m.box / 1.3) if share is None else share * 0.5 * m.box
            g = kg.kg_pair_distribution(ctx, i, r_max, bins)
            assert np.allclose(g, SF.pair_distribution(m.x, m.box, r_max, bins), rtol=1e-12, atol=0)


def test_structure_factor_of_far_positions_and_large_vectors(kg):
    m = KI.random_walk_melt(30, 50, 0.85, 2.0, 8)
    far = m.x + m.box * np.array([[3.0], [-7.0], [1000.0]])
    rng = np.random.default_rng(2)
    hkl = rng.integers(-200, 201, (131, 3))              # not a multiple of the vectors per thread
    with _ctx(kg, [m]) as ctx:
        S = [kg.kg_structure_factor(ctx, 0, hkl)]
        kg.kg_load_config(ctx, 0, far, m.v)
        S.append(kg.kg_structure_factor(ctx, 0, hkl))
        one = kg.kg_structure_factor(ctx, 0, hkl[:1])
        nan = m.x.copy()
        nan[1, 17] = np.nan
        kg.kg_load_config(ctx, 0, nan, m.v)
        assert np.isnan(kg.kg_structure_factor(ctx, 0, hkl)).all()
    # phases in binary32: 2 pi 2^-25 a term at most, M of them
    for got, x in zip(S, (m.x, far)):
        assert np.allclose(got, SF.structure_factor(x - m.box * np.round(x / m.box), m.box, hkl), rtol=1e-5, atol=1e-4)
    assert one[0] == S[1][0]


def _r2n(x, chains, N):
    p = np.asarray(x, dtype=np.longdouble).reshape(3, chains, N)
    out = np.zeros(N)
    for n in range(1, N):
        out[n] = float(((p[:, :, n:] - p[:, :, :-n]) ** 2).sum() / (chains * (N - n)))
    return out


# chain lengths around a lag window (4), the conflict-free padding (32) and a
# chunk of 256 terms; few long chains (one chain over several blocks)
@pytest.mark.parametrize("chains,N", [(100, 3), (80, 4), (64, 5), (40, 33), (9, 257), (7, 1030), (2, 4099)])
def test_r2n(kg, chains, N):
    m = KI.random_walk_melt(chains, N, 0.85, 2.0, 11)
    with _ctx(kg, [m]) as ctx:
        for x in (m.x, m.x * 1e-3, m.x + 4096.0):
            kg.kg_load_config(ctx, 0, x, m.v)
            r2n = np.zeros(N)
            # without energies: x * 1e-3 is no state to evaluate
            assert kg.load().kg_observables(ctx, 0, None, kg.binding.ptr(r2n), None, None, 0) == kg.KG_OK
            want = _r2n(x, chains, N)
            # binary64 positions: each term off by a few 2^-53 |x| |d|
            tol = 16 * 2.0 ** -53 * max(1.0, np.abs(x).max() / np.sqrt(want[1]))
            assert np.abs(r2n[1:] / want[1:] - 1).max() < tol and r2n[0] == 0


@pytest.mark.parametrize("bins", [1, 7, 100, 3000])
def test_histograms_are_exact(kg, bins):
    melts = [KI.random_walk_melt(33, 31, 0.85, 2.0, 13), KI.random_walk_melt(20, 50, 0.85, 0.5, 14)]
    rng = np.random.default_rng(4)
    for m in melts:                                      # generated bonds all have one length, 0.97
        m.x += 0.02 * rng.standard_normal(m.x.shape)
    with _ctx(kg, melts) as ctx:
        for i, m in enumerate(melts):
            b, c = np.zeros(bins), np.zeros(bins)
            kg.kg_observables(ctx, i, None, b, c, bins)
            p = m.x.reshape(3, m.n_chains, m.chain_len)
            d = np.diff(p, axis=2)
            d -= m.box * np.rint(d / m.box)
            r = np.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
            hb = np.floor(r / 1.5 * bins).astype(int).ravel()
            e, f = d[:, :, :-1], d[:, :, 1:]
            cs = (e * f).sum(0) / (r[:, :-1] * r[:, 1:])
            hc = np.clip(np.floor((cs + 1.0) * 0.5 * bins).astype(int).ravel(), 0, bins - 1)
            wb = np.bincount(hb[(hb >= 0) & (hb < bins)], minlength=bins)
            wc = np.bincount(hc, minlength=bins)
            # numpy's order of the same binary64 operations may move a value that sits on an edge
            assert np.abs(b - wb).sum() <= 2 and np.abs(c - wc).sum() <= 2
            assert b.sum() == wb.sum() and c.sum() == wc.sum()
