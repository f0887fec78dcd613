"""Events of weight 0 take no part in a weighted evaluation, wherever they lie: at a polynomial's zero
(whose derivative lanes x / r are infinite there), beyond an Argus endpoint that leaves no density, as one
or both events of a pair, and at ragged ends.  The result is that of the other events alone."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

# FP32: the same events in other pairs and other orders, 1e-7 per term
TOL = {"f64": 1e-12, "f32": 2e-6}


@pytest.fixture(scope="module")
def goo():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1710_08826_gb300 import goo as g
    return g


@pytest.fixture(scope="module")
def ctx(goo):
    return goo.Context(0)


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("form", ["zero_poly", "no_density"])
@pytest.mark.parametrize("n", [5, 1001, 20_001])
def test_masked_events_do_not_matter(goo, ctx, n, form, precision):
    spec = synth.c2_spec(bins=32)
    _, _, (sig, bkg) = spec["pdf"]
    theta = np.array(synth.param_values(spec))
    names = [p[0] for p in spec["params"]]
    cols = synth.round_to_f32({k: v[:n].copy() for k, v in synth.gen_c2(n=20_001, seed=34).items()}, spec)
    masked = np.random.default_rng(8).uniform(size=n) < 0.4
    masked[[0, n - 1]], masked[1] = True, False
    if form == "zero_poly":  # (1 - 8 dE)^2
        poly = next(l for l in bkg[1] if l[0] == "poly2")
        theta[names.index(poly[2])], theta[names.index(poly[3])] = -16.0, 64.0
        cols["dE"][masked] = 0.125
    else:
        spec = dict(spec, pdf=bkg)
        theta[names.index("m0")] = 5.2925
        cols["m"] = np.minimum(cols["m"], np.float32(5.2915)).astype(np.float64)
        cols["m"][masked] = np.float32(5.2975)
    w = np.where(masked, 0.0, np.random.default_rng(9).uniform(0.5, 1.5, n).astype(np.float32))
    model = goo.Model(ctx, spec)
    ds, rest = goo.Dataset.from_spec(ctx, spec, cols), goo.Dataset.from_spec(ctx, spec, {k: v[~masked] for k, v in cols.items()})
    ds.set_weights(w)
    rest.set_weights(w[~masked])
    nll, g = model.nll_grad(ds, theta, precision)
    rnll, rg = model.nll_grad(rest, theta, precision)
    assert abs(nll - rnll) <= TOL[precision] * max(abs(rnll), n), (nll, rnll)
    assert np.all(np.isfinite(g))
    assert np.max(np.abs(g - rg)) <= TOL[precision] * max(np.max(np.abs(rg)), n), (g, rg)
    assert model.nll(ds, theta, precision) == pytest.approx(nll, rel=1e-12)
