"""Floating lineshapes in FP32 with every coefficient scaled by 2e-20: |S|^2 is subnormal and so is its mean
over the normalisation sample, and the NLL is that of the unscaled coefficients (FP64 reference)."""
import numpy as np
import pytest

import synth
from test_gpu_coherent_shapes import _spec

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def goo():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1710_08826_gb300 import goo as g
    return g


@pytest.mark.parametrize("n_res,nr", [(8, True), (15, False)])
def test_scaled_coefficients(goo, n_res, nr):
    spec = _spec(n_res, nr)
    kin = synth.TD3_MASSES
    cands = synth.round_to_f32(synth.dalitz_candidates(12_000, 14, kin["M"], kin["m1"], kin["m2"], kin["m3"]), spec)
    data, mc = {k: v[:5001] for k, v in cands.items()}, {k: v[-4000:] for k, v in cands.items()}
    theta = np.array(synth.param_values(spec))
    ctx = goo.Context(0)
    model = goo.Model(ctx, spec, mc=goo.Dataset.from_spec(ctx, spec, mc))
    model.set_lineshapes("floating")
    ds = goo.Dataset.from_spec(ctx, spec, data)
    want = model.nll(ds, theta, "f64")
    theta[[p[0].startswith(("re_", "im_")) for p in spec["params"]]] *= 2e-20
    # |S|^2 of 4e-40 (1 + ...) in steps of 2^-149: 3.5e-6 each, of either sign; the largest are normal
    assert abs(model.nll(ds, theta, "f32") - want) <= 1e-4 * 5001
    nll = model.nll_grad(ds, theta, "f32")[0]
    assert abs(nll - want) <= 1e-4 * 5001
