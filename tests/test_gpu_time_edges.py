"""Decay-time terms at their edges: observed times from 6 resolutions below zero to the end of
the range, and mixing for which the events of one launch lie on both sides of the moment
series' limit (and the series' two orders), against the oracle's Faddeeva form."""
import numpy as np
import pytest

import synth
from oracle import td4 as ot

pytestmark = pytest.mark.gpu

# as in the four-body parity tests: the oracle's convolved exponentials differ by rounding in
# FP64; FP32 sums carry 1e-7 per term
TOL_NLL = {"f64": 1e-9, "f32": 1e-6}
TOL_GRAD = {"f64": 1e-6, "f32": 1e-4}


@pytest.fixture(scope="module")
def goo():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1710_08826_gb300 import goo as g
    return g


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("x,y", [(0.004, 0.006), (0.0, 0.02), (0.03, 0.05), (-0.06, 0.02), (0.4, -0.3)])
def test_time_range_and_series_limit(goo, precision, x, y):
    spec = synth.c4_spec()
    theta = np.array(synth.param_values(spec))
    n = 3000
    data = synth.four_body_phase_space(n, 17, **synth.TD4_MASSES)
    rng = np.random.default_rng(3)
    data["t"] = np.concatenate([np.linspace(-0.3, 0.3, 1000), np.linspace(0.3, 10.0, 1000), rng.exponential(0.41, 1000)])
    mc = synth.four_body_phase_space(4000, 18, **synth.TD4_MASSES)
    mc["t"] = np.zeros(4000)
    if precision == "f32":
        data, mc = synth.round_to_f32(data, spec), synth.round_to_f32(mc, spec)
    m = ot.TD4Model(spec)
    theta[m.tp[0]], theta[m.tp[1]] = x, y
    ctx = goo.Context(0)
    ds, mcds = goo.Dataset.from_spec(ctx, spec, data), goo.Dataset.from_spec(ctx, spec, mc)
    model = goo.Model(ctx, spec, mc=mcds)
    nll, g = model.nll_grad(ds, theta, precision)
    rnll, rg = m.nll_grad(data, m.amplitudes(mc), theta)
    assert abs(nll - rnll) <= TOL_NLL[precision] * abs(rnll), (nll, rnll)
    assert np.max(np.abs(g - rg)) <= TOL_GRAD[precision] * np.max(np.abs(rg)), (g, rg)
    assert model.nll(ds, theta, precision) == pytest.approx(nll, rel=1e-12)
