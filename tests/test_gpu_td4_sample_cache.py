"""The FP64 four-body cache of an MC normalisation sample holds its amplitudes and nothing else (the sum B,
one plane more, is kept for events), and a sample that is evaluated as events itself gets it then."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

N = 2_000_000


@pytest.fixture(scope="module")
def goo():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1710_08826_gb300 import goo as g
    return g


def test_memory_and_results(goo):
    import torch
    spec = synth.c4_spec(n_mc=N)
    K = len(spec["pdf"][2])
    cols = synth.four_body_phase_space(20_000, 6, **synth.TD4_MASSES)
    cols["t"] = np.random.default_rng(6).exponential(0.4, 20_000)
    theta = np.array(synth.param_values(spec))
    ctx = goo.Context(0)
    sample = {k: np.tile(v, N // 20_000) for k, v in cols.items()}
    mcds, ds = goo.Dataset.from_spec(ctx, spec, sample), goo.Dataset.from_spec(ctx, spec, cols)
    model = goo.Model(ctx, spec, mc=mcds)
    small = goo.Model(ctx, spec, mc=ds)
    nll, g = small.nll_grad(ds, theta, "f64")  # work space and tables
    other = goo.Dataset.from_spec(ctx, spec, cols)
    other_nll, other_g = small.nll_grad(other, theta, "f64")
    assert nll == other_nll and np.array_equal(g, other_g)  # the sample as events, and the same events alone
    free = torch.cuda.mem_get_info()[0]
    model.normalise(theta, "f64")
    held = free - torch.cuda.mem_get_info()[0]
    assert K * 16 * N <= held + (1 << 21) and held < (K + 0.5) * 16 * N, held / (16 * N)
    before = small.nll(ds, theta, "f64")
    big = model.nll(mcds, theta, "f64")
    assert big == model.nll(mcds, theta, "f64")
    # the sample is 100 copies of the events: N is the same mean, the NLL 100 times theirs
    assert big == pytest.approx(100.0 * before, rel=1e-12)
