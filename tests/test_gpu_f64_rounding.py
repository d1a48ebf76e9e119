"""Rounding of the binary64 step's forces: one step from rest without friction
and noise (u = dt F), against the forces in extended precision, no further off
than the plain formulas evaluated in binary64 one operation after the other from
correctly rounded squared lengths.  Positions are binary32 numbers, so that every
difference is exact and the rounding seen is that of the force terms: a squared
length from fused multiply-adds adds about 0.4 ulp to the 0.3 each of its
rounding and its inverse's (a factor 1.2 here), an inverse from the square of a
reciprocal square root about 0.8 (2.3).
"""
import numpy as np
import pytest

from conftest import relaxed_melt

pytestmark = pytest.mark.gpu
DT = 2.0 ** -10                                      # u / dt is exact


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


def forces(x, box, N, kappa, n, k, T):
    """Eqs. 4, 6 and 10 in the type T, r^-n as a product of 1 / r^2 (n even)."""
    M = x.shape[1]
    X, L = x.astype(np.longdouble), np.longdouble(box)

    def dot(a, b):
        return (a * b).sum(0).astype(T)

    rc2 = T(2) ** (T(1) / T(3))
    c1, c2 = T(6) * T(2) ** (T(n) / T(6)) / T(n - 6), T(2) * T(n) / T(n - 6)

    def mlj(r2):
        i2 = T(1) / r2
        i6 = i2 * i2 * i2
        rn = i6
        for _ in range(n // 2 - 3):
            rn = rn * i2
        return np.where(r2 < rc2, (T(6) * c2 * i6 - T(n) * c1 * rn) * i2, T(0))

    F = np.zeros((3, M), T)
    for i in range(M):
        d = x - x[:, i:i + 1]
        d -= box * np.rint(d / box)
        j = np.nonzero((d * d).sum(0) < 1.3)[0]
        j = j[(j != i) & ~((np.abs(j - i) == 1) & (j // N == i // N))]
        D = X[:, j] - X[:, i:i + 1]
        D = D - L * np.rint(D / L)
        F[:, i] = (mlj(dot(D, D)) * D.astype(T)).sum(1)
    p = X.reshape(3, -1, N)
    G = np.zeros(p.shape, T)
    b = p[:, :, 1:] - p[:, :, :-1]
    r2, b1, b2 = dot(b, b), b[:, :, :-1], b[:, :, 1:]
    b12, b = dot(b1, b2), b.astype(T)
    f = T(k) / (T(1) - r2 / T(2.25)) + mlj(r2)
    G[:, :, :-1] += f * b
    G[:, :, 1:] -= f * b
    b1, b2, l1, l2 = b[:, :, :-1], b[:, :, 1:], r2[:, :-1], r2[:, 1:]
    inv = T(1) / np.sqrt(l1 * l2)
    cs = b12 * inv
    g1, g2 = T(kappa) * (b2 * inv - cs / l1 * b1), T(kappa) * (b1 * inv - cs / l2 * b2)
    G[:, :, :-2] -= g1
    G[:, :, 1:-1] += g1 - g2
    G[:, :, 2:] += g2
    return F + G.reshape(3, -1)


@pytest.mark.parametrize("chains,N,kappa,n", [(20, 50, 1.5, 12), (10, 100, 3.5, 12), (20, 50, 0.0, 12), (20, 50, 2.5, 8)])
def test_forces_of_a_step(kg, chains, N, kappa, n):
    rms = np.zeros(2)
    for seed in (1, 2, 3):
        m = relaxed_melt(chains, N, kappa, seed)
        m.x, m.box = m.x.astype(np.float32).astype(np.float64), float(np.float32(m.box))
        p = kg.make_params([(chains, N, m.box, kappa)], precision=kg.KG_FP64, seed=1, gamma=0.0)
        ctx = kg.kg_create(p, 0, None, None)
        try:
            kg.kg_set_potential_schedule(ctx, [kg.stage(float(n), 10 ** 9, DT)])
            kg.kg_load_config(ctx, 0, m.x, np.zeros_like(m.x))
            kg.kg_step(ctx, 1)
            u = np.zeros_like(m.x)
            kg.kg_get_config(ctx, 0, None, u)
        finally:
            kg.kg_destroy(ctx)
        k = kg.kg_kn(float(n))
        want = forces(m.x, m.box, N, kappa, n, k, np.longdouble)
        scale = np.sqrt((want ** 2).sum(0).mean())
        for i, got in enumerate((u / DT, forces(m.x, m.box, N, kappa, n, k, np.float64))):
            rms[i] += ((got - want) ** 2).sum(0).mean() / scale ** 2
    assert np.sqrt(rms[0] / rms[1]) < 1.6, np.sqrt(rms / 3)
