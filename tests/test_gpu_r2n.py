"""<R^2(n)> (kg_r2n_noalloc) on both sides of every line of its dispatch: short
chains in binary64, one or four lags a thread, several blocks a chain, a last
block of short chains that is not full.
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


def r2n(kg, x):
    """(3, chains, N) positions -> <R^2(n)>, rows padded by five doubles."""
    import torch
    _, chains, N = x.shape
    rows = torch.full((3, chains * N + 5), float("nan"), dtype=torch.float64, device="cuda")
    rows[:, :chains * N] = torch.from_numpy(x.reshape(3, -1)).cuda()
    out = torch.full((N,), -1.0, dtype=torch.float64, device="cuda")
    kg.kg_r2n_noalloc(rows, rows.shape[1], chains, N, out, torch.cuda.current_stream().cuda_stream)
    return out.cpu().numpy()


def plain(x):
    _, chains, N = x.shape
    out = np.zeros(N)
    for n in range(1, N):
        out[n] = ((x[:, :, n:] - x[:, :, :-n]) ** 2).sum() / (chains * (N - n))
    return out


def walk(chains, N, seed):
    g = np.random.default_rng(seed)
    b = g.standard_normal((3, chains, N))
    b *= 0.97 / np.sqrt((b * b).sum(0))
    b[:, :, 0] = g.uniform(0.0, 40.0, (3, chains))
    return np.cumsum(b, axis=2)


@pytest.mark.parametrize("chains,N", [(1, 2), (1, 3), (43, 3), (64, 2), (6, 20), (7, 20), (1, 20), (1000, 19), (1, 21),
                                      (5, 32), (3, 129), (2, 1537), (299, 777), (300, 777), (300, 700), (151, 1537)])
def test_every_path(kg, chains, N):
    x = walk(chains, N, 7)
    got, want = r2n(kg, x), plain(x)
    # a sum of N terms one after the other, positions of binary64 rounding 2^-53 max |x| against bonds of 0.97
    tol = (N + 16 * np.abs(x).max()) * 2.0 ** -53
    assert got[0] == 0 and np.abs(got[1:] / want[1:] - 1).max() < tol


# one monomer far away, two monomers almost at one place, straight rods: lags that do not see the far one keep
# the rounding of binary64 (a chain of N sums N terms, 2^-53 each, in any order)
@pytest.mark.parametrize("chains,N", [(3, 100), (5, 800), (1, 2500)])
@pytest.mark.parametrize("kind", ["far", "near", "rod"])
def test_data_that_are_no_melt(kg, chains, N, kind):
    x, first = walk(chains, N, 9), 1
    if kind == "far":
        x[1, :, N // 2] += 1e9
        first = N // 2 + 1                           # no pair with the far monomer from here
    elif kind == "near":
        x[:, :, 1] = x[:, :, 0] + 1e-9
    else:
        x = x[:, :, :1] + 0.97 * np.arange(N)[None, None, :] * np.array([0.8, 0.6, 0.0])[:, None, None]
    got = r2n(kg, np.ascontiguousarray(x))
    y = x.astype(np.longdouble)
    for n in range(first, N, 1 + N // 200):
        want = ((y[:, :, n:] - y[:, :, :-n]) ** 2).sum() / (chains * (N - n))
        assert abs(got[n] / want - 1) < 4 * N * 2.0 ** -53
