"""Floating-lineshape NLL + gradient (masses and widths included) against the oracle over the
kernel's shapes: 1 to 15 resonances (both slot counts, empty slots), with and without the
constant amplitude, event counts and ranges with odd ends (the FP32 kernel takes points in pairs
at even indices), and an MC sample smaller than a block."""
import numpy as np
import pytest

import synth
from oracle import dalitz as od
from test_gpu_coherent_shapes import _spec

pytestmark = pytest.mark.gpu

# FP64: the two sides' amplitudes differ by rounding; FP32: 1e-5 of each term, and a mass's gradient is a
# difference of an event sum and an MC sum of similar size
TOL = {"f64": 1e-8, "f32": 3e-4}


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
@pytest.mark.parametrize("n_res,nr,n_mc", [(1, True, 301), (2, False, 4000), (8, True, 4001), (9, True, 100), (15, True, 4000)])
def test_shapes_match_oracle(goo, ctx, precision, n_res, nr, n_mc):
    spec = _spec(n_res, nr)
    kin = synth.TD3_MASSES
    cands = synth.round_to_f32(synth.dalitz_candidates(40_000, 9, kin["M"], kin["m1"], kin["m2"], kin["m3"]), spec)
    mc = {k: v[-n_mc:] for k, v in cands.items()}
    ref = od.DalitzModel(spec)
    theta = np.array(synth.param_values(spec))
    mcds = goo.Dataset.from_spec(ctx, spec, mc)
    model = goo.Model(ctx, spec, mc=mcds)
    model.set_lineshapes("floating")
    for n in (1, 2, 257, 30_001):
        data = {k: v[:n] for k, v in cands.items()}
        ds = goo.Dataset.from_spec(ctx, spec, data)
        nll, g = model.nll_grad(ds, theta, precision)
        rnll, rg = ref.nll_grad(data, mc, theta)
        # a narrow resonance's mass derivative of one event is up to 2 m0 / (m0 Gamma0), about 30
        scale = max(np.max(np.abs(rg)), 30.0 * n)
        assert abs(nll - rnll) <= TOL[precision] * max(abs(rnll), n), (n, nll, rnll)
        assert np.max(np.abs(g - rg)) <= TOL[precision] * scale, (n, g, rg)
    edges = [0, 1, 8, 257, 257, 10_001, n]
    parts = [model.nll_partial(ds, a, b, theta, precision) for a, b in zip(edges[:-1], edges[1:])]
    tot = goo.combine_partials(parts, model.n_params)
    assert abs(tot[0] + tot[1] - nll) <= (1e-12 if precision == "f64" else 1e-6) * max(abs(nll), n)
    np.testing.assert_allclose(tot[3:], g, rtol=0, atol=(1e-10 if precision == "f64" else 1e-5) * scale)
