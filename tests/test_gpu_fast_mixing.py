"""Decay-time terms past the moment series' limit, max(|x|, |y|) / tau * 6 sigma_t >= 0.35 (FP64) and
0.5 (FP32): no event, of whatever sign its time is, may take the series.  Observed times from 6
resolutions (or the limit of the range) below zero, the four-body and the three-body model, against
the oracle's Faddeeva form, and the per-event log f against the NLL."""
import numpy as np
import pytest

import synth
from oracle import td3 as o3
from oracle import td4 as o4

pytestmark = pytest.mark.gpu

# as in the parity tests of these models; FP32: the phase x t / tau reaches 180, where its rounding is 1e-5 of
# each term and random, 2e-7 of a sum of 2400 events
TOL_NLL = {"f64": 1e-9, "f32": 1e-6}
TOL_GRAD = {"f64": 1e-6, "f32": 1e-4}
# x, y, tau, sigma_t
POINTS = [(1.0, 0.05, 0.41, 0.05), (0.77, 0.0, 1.5, 1.0), (5.0, 0.1, 0.41, 0.05), (15.0, -0.2, 0.41, 0.05),
          (26.7, 0.06, 1.51, 0.1), (0.02, 0.9, 0.41, 0.1)]


@pytest.fixture(scope="module")
def goo():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1710_08826_gb300 import goo as g
    return g


@pytest.fixture(scope="module")
def ctx(goo):
    return goo.Context(0)


def _times(sigma, seed):
    lo = max(-0.49, -6.0 * sigma)
    return np.concatenate([np.linspace(lo, 0.0, 800), -np.geomspace(1e-9, 1e-3, 200), np.linspace(0.0, 10.0, 400),
                           np.random.default_rng(seed).exponential(0.5, 1000)])


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("point", POINTS)
@pytest.mark.parametrize("bodies", [3, 4])
def test_negative_times_past_the_series_limit(goo, ctx, bodies, point, precision):
    spec = synth.c4_spec() if bodies == 4 else synth.td3_spec()
    theta = np.array(synth.param_values(spec))
    t = _times(point[3], 7)
    if bodies == 4:
        data, mc = (synth.four_body_phase_space(n, s, **synth.TD4_MASSES) for n, s in ((t.size, 21), (4000, 22)))
        ref = o4.TD4Model(spec)
    else:
        kin = synth.TD3_MASSES
        data, mc = (synth.dalitz_candidates(n, s, kin["M"], kin["m1"], kin["m2"], kin["m3"])
                    for n, s in ((t.size, 21), (4000, 22)))
        ref = o3.TD3Model(spec)
    data["t"], mc["t"] = t, np.zeros(4000)
    if precision == "f32":
        data, mc = synth.round_to_f32(data, spec), synth.round_to_f32(mc, spec)
    theta[ref.tp] = point
    mcds = goo.Dataset.from_spec(ctx, spec, mc)
    ds, model = goo.Dataset.from_spec(ctx, spec, data), goo.Model(ctx, spec, mc=mcds)
    nll, g = model.nll_grad(ds, theta, precision)
    rnll, rg = ref.nll_grad(data, ref.amplitudes(mc) if bodies == 4 else mc, theta)
    assert abs(nll - rnll) <= TOL_NLL[precision] * max(abs(rnll), t.size), (nll, rnll)
    assert np.max(np.abs(g - rg)) <= TOL_GRAD[precision] * np.max(np.abs(rg)), (g, rg)
    assert model.nll(ds, theta, precision) == pytest.approx(nll, rel=1e-12)
    if bodies == 4:
        logf = model.eval_logf(ds, theta, precision).cpu().numpy()
        assert abs(-logf.sum() - rnll) <= TOL_NLL[precision] * max(abs(rnll), t.size)
