"""A resolution so small that t^2 / 2 sigma_t^2 leaves the FP32 range (sigma_t far below 1e-18, the resolution
switched off) gives the unsmeared decay-time terms: the FP32 NLL is the FP64 one, four- and three-body model."""
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


@pytest.mark.parametrize("sigma", [1e-15, 1e-17, 1e-19, 1e-22])
@pytest.mark.parametrize("mixing", [(0.004, 0.006), (5.0, 0.1)])
@pytest.mark.parametrize("bodies", [3, 4])
def test_unsmeared(goo, bodies, mixing, sigma):
    spec = synth.c4_spec() if bodies == 4 else synth.td3_spec()
    names = [p[0] for p in spec["params"]]
    theta = np.array(synth.param_values(spec))
    for k, v in (("x", mixing[0]), ("y", mixing[1]), ("sigma_t", sigma)):
        theta[names.index(k)] = v
    n = 3000
    kin = synth.TD3_MASSES
    if bodies == 4:
        data, mc = (synth.four_body_phase_space(k, s, **synth.TD4_MASSES) for k, s in ((n, 25), (2000, 26)))
    else:
        data, mc = (synth.dalitz_candidates(k, s, kin["M"], kin["m1"], kin["m2"], kin["m3"]) for k, s in ((n, 25), (2000, 26)))
    data["t"], mc["t"] = np.random.default_rng(5).exponential(0.41, n) % 9.0 + 1e-3, np.zeros(2000)
    data, mc = synth.round_to_f32(data, spec), synth.round_to_f32(mc, spec)
    ctx = goo.Context(0)
    model = goo.Model(ctx, spec, mc=goo.Dataset.from_spec(ctx, spec, mc))
    ds = goo.Dataset.from_spec(ctx, spec, data)
    want = model.nll(ds, theta, "f64")
    # FP32 against FP64 of the same sample, as in the parity tests of these models
    assert model.nll(ds, theta, "f32") == pytest.approx(want, rel=1e-6, abs=1e-6 * n)
