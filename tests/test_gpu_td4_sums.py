"""The FP64 four-body evaluation takes B = sum b_k a_k from the amplitude cache where the cache has a
plane for it and forms it per event where it has not (a dataset whose cache was allocated for a model
of one amplitude less).  Both form B in one order: the results are the same bit for bit."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def goo():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1710_08826_gb300 import goo as g
    return g


@pytest.fixture(scope="module")
def ctx(goo):
    return goo.Context(0)


def _spec(K, shift=0.0):
    spec = synth.c4_spec(n_mc=2000)
    _, kin, amps, time = spec["pdf"]
    par = {p[0]: p for p in spec["params"]}
    params, out = [], []
    for k in range(K):
        ang, r12, r34, re, im, (br, bi) = amps[k % len(amps)]
        params += [(f"re{k}",) + par[re][1:], (f"im{k}",) + par[im][1:]]
        out.append((ang, r12, r34, f"re{k}", f"im{k}", (br + 0.1 * k + shift, bi)))
    params += [par[t] for t in time]
    return dict(spec, params=params, pdf=("td4", kin, out, time))


@pytest.mark.parametrize("K", [2, 10, 11, 15])
@pytest.mark.parametrize("n", [1, 257, 30_001])
def test_b_from_the_cache_or_per_event(goo, ctx, K, n):
    spec = _spec(K)
    cols = synth.four_body_phase_space(n + 2000, 5, **synth.TD4_MASSES)
    cols["t"] = np.random.default_rng(5).exponential(0.4, n + 2000)
    data, mc = {k: v[:n] for k, v in cols.items()}, {k: v[n:] for k, v in cols.items()}
    mcds = goo.Dataset.from_spec(ctx, spec, mc)
    theta = np.array(synth.param_values(spec))

    def evaluate(ds, spec):
        model = goo.Model(ctx, spec, mc=mcds)
        nll, g = model.nll_grad(ds, theta, "f64")
        return nll, g, model.nll(ds, theta, "f64"), np.asarray(model.eval_logf(ds, theta, "f64").cpu())
    fresh = evaluate(goo.Dataset.from_spec(ctx, spec, data), spec)
    ds = goo.Dataset.from_spec(ctx, spec, data)
    small = _spec(K - 1)
    goo.Model(ctx, small, mc=mcds).nll(ds, np.array(synth.param_values(small)), "f64")
    without = evaluate(ds, spec)
    assert fresh[0] == without[0] and fresh[2] == without[2]
    assert np.array_equal(fresh[1], without[1]) and np.array_equal(fresh[3], without[3])
    # another model of the same amplitudes and other constants b on the same dataset
    other = _spec(K, 0.3)
    a, b = evaluate(ds, other), evaluate(goo.Dataset.from_spec(ctx, other, data), other)
    assert a[0] == b[0] and a[0] != fresh[0] and np.array_equal(a[1], b[1])
