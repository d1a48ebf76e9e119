"""Outputs into device memory that work queued on the default stream still
writes: a context on its own stream writes them after that work, in every call
that takes such a buffer.
"""
import numpy as np
import pytest

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
    return relaxed_melt(30, 20, 1.0, 17)


@pytest.mark.parametrize("precision", [0, 1])        # binary64, mixed
@pytest.mark.parametrize("call", ["get_config", "forces", "r2n", "paths"])
def test_output_still_being_filled(kg, melt, precision, call):
    import torch
    p = kg.make_params([(melt.n_chains, melt.chain_len, melt.box, melt.kappa)], precision=precision, seed=1)
    ctx = kg.kg_create(p, 0, None, kg.torch_allocator())
    read = {"get_config": lambda a: kg.kg_get_config(ctx, 0, a), "forces": lambda a: kg.kg_forces(ctx, 0, a),
            "r2n": lambda a: kg.kg_observables(ctx, 0, a),
            "paths": lambda a: kg.kg_primitive_path(ctx, 0, melt.n_chains, 3, x_out=a, precision=precision)}[call]
    try:
        kg.kg_load_config(ctx, 0, melt.x, melt.v)
        want = np.zeros(melt.chain_len) if call == "r2n" else np.zeros_like(melt.x)
        read(want)
        out = torch.empty(want.shape, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        torch.cuda._sleep(200_000_000)               # ~0.1 s of the default stream
        out.fill_(-7.0)
        read(out)
        got = out.cpu().numpy()                      # behind the fill on the default stream
    finally:
        kg.kg_destroy(ctx)
    assert np.array_equal(got, want)
