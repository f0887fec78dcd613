"""FP32 decay-time terms in the tails: 13.2 to 13.6 resolutions below zero the Gaussian is subnormal, 88 to
90 lifetimes above so is the exponential, and the rate, some 1e3 to 1e5 times larger, is not: such events
have a density in FP32 too (four- and three-body model; both the pair and the scalar kernels)."""
import numpy as np
import pytest

import synth
from oracle import td3 as o3
from oracle import td4 as o4

pytestmark = pytest.mark.gpu

# a subnormal of 2^-137 has 12 bits (2.4e-4), and a rate adds four terms of it: 1e-3 of log R per event; the
# normalisation adds 1e-6
TOL = 1e-3


@pytest.fixture(scope="module")
def goo():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1710_08826_gb300 import goo as g
    return g


@pytest.mark.parametrize("bodies,tail", [(4, "below"), (4, "above"), (3, "above")])
def test_subnormal_terms(goo, bodies, tail):
    spec = synth.c4_spec() if bodies == 4 else synth.td3_spec()
    theta = np.array(synth.param_values(spec))
    n = 40_000
    if bodies == 4:
        data, mc = (synth.four_body_phase_space(k, s, **synth.TD4_MASSES) for k, s in ((n, 23), (4000, 24)))
        ref = o4.TD4Model(spec)
    else:
        kin = synth.TD3_MASSES
        data, mc = (synth.dalitz_candidates(k, s, kin["M"], kin["m1"], kin["m2"], kin["m3"]) for k, s in ((n, 23), (4000, 24)))
        ref = o3.TD3Model(spec)
    u = np.random.default_rng(11).uniform(size=n)
    if tail == "below":
        theta[ref.tp] = (0.004, 0.006, 0.41, 0.03)
        data["t"] = -0.03 * (13.2 + 0.4 * u)
    else:
        theta[ref.tp] = (0.002, 0.003, 0.11, 0.03)  # the moment series up to z = 0.27
        data["t"] = 0.11 * (88.0 + 2.0 * u)
    mc["t"] = np.zeros(4000)
    data, mc = synth.round_to_f32(data, spec), synth.round_to_f32(mc, spec)
    amps = ref.amplitudes(data) if bodies == 4 else ref.amplitudes(data, theta)
    R = ref.rate(amps, data["t"], theta)
    P = np.abs(amps @ ref.coefficients(theta) if bodies == 4 else amps[0] @ ref.coefficients(theta)) ** 2
    # the rate normal, the term P = R / |A|^2 (about) subnormal but with 12 bits
    keep = (R > 2.0 ** -125) & (R < P * 2.0 ** -126) & (R > P * 2.0 ** -136)
    assert keep.sum() > 100
    data = {k: v[keep] for k, v in data.items()}
    ctx = goo.Context(0)
    mcds, ds = goo.Dataset.from_spec(ctx, spec, mc), goo.Dataset.from_spec(ctx, spec, data)
    model = goo.Model(ctx, spec, mc=mcds)
    if bodies == 4:
        rnll, _ = ref.nll_grad(data, ref.amplitudes(mc), theta)
    else:
        rnll, _ = ref.nll_grad(data, mc, theta)
    m = int(keep.sum())
    assert abs(model.nll(ds, theta, "f32") - rnll) <= TOL * m
    nll, g = model.nll_grad(ds, theta, "f32")
    assert abs(nll - rnll) <= TOL * m and np.all(np.isfinite(g))
