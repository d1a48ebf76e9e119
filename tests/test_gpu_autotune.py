"""The autotuner times no setting twice: block sizes and threads per monomer are
candidates only where the steps' kernels take them.
"""
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


# five skins and two cell sides; one thread a monomer in the resident loop (no block size), two in the captured
# loop (three); binary64 and the one launch of the flag: neither.  1300 monomers per SM: the captured loop, six a skin
@pytest.mark.parametrize("per_sm,precision,flags,trials", [(0, 1, 0, 5 * 4 + 2), (0, 0, 0, 5 + 2), (0, 1, 2, 5 + 2),
                                                           (1300, 1, 0, 5 * 6 + 2)])
def test_number_of_trials(kg, per_sm, precision, flags, trials):
    import torch
    chains = max(40, per_sm * torch.cuda.get_device_properties(0).multi_processor_count // 50)
    m = KI.random_walk_melt(chains, 50, 0.85, 1.0, 3)
    p = kg.make_params([(m.n_chains, m.chain_len, m.box, m.kappa)], precision=precision, seed=1, fene_qmin=0.01, flags=flags)
    best = kg.kg_autotune(p, [m.x], [m.v], kg.stage(2.0, -1, 0.002), 20)
    assert best.trials == trials
    assert best.block_size in (64, 128, 256) and best.threads_per_monomer in (1, 2) and 0.25 <= best.skin <= 0.6
    assert best.threads_per_monomer == 1 or trials > 7
