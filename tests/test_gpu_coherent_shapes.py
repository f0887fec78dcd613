"""Coherent-sum NLL + gradient against the oracle over the kernels' shapes: 1 to 15 resonances
(both slot counts, empty slots), with and without the constant amplitude, at event counts around
a warp, a block and a grid-stride step."""
import numpy as np
import pytest

import synth
from oracle import dalitz as od

pytestmark = pytest.mark.gpu

# FP64: amplitudes of the two sides differ by rounding (1e-12 relative), sums are carried to 2^-48.
# FP32: each term is good to about 1e-5 of its size; with few events nothing averages out.
TOL = {"f64": 1e-9, "f32": 1e-4}


@pytest.fixture(scope="module")
def goo():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1710_08826_gb300 import goo as g
    return g


@pytest.fixture(scope="module")
def ctx(goo):
    return goo.Context(0)


def _spec(n_res, nr):
    kin = dict(synth.TD3_MASSES, r_res=1.5, r_par=5.0)
    M, m1, m2, m3 = (kin[k] for k in ("M", "m1", "m2", "m3"))
    params, amps = [], []
    for k, ((_, pair, spin, m0, w), (re, im)) in enumerate(zip(synth.TD3_RESONANCES[:n_res], synth.TD3_TRUTH)):
        params += [(f"m0_{k}", m0, True, 0.0), (f"w_{k}", w, True, 0.0), (f"re_{k}", re, False, 0.02),
                   (f"im_{k}", im, False, 0.02)]
        amps.append(("bw", pair, spin, f"m0_{k}", f"w_{k}", f"re_{k}", f"im_{k}"))
    if nr:
        params += [("re_nr", 0.5, False, 0.02), ("im_nr", 0.2, False, 0.02)]
        amps.append(("nr", "re_nr", "im_nr"))
    return dict(name="shapes", observables=[("s12", (m1 + m2) ** 2, (M - m3) ** 2), ("s13", (m1 + m3) ** 2, (M - m2) ** 2)],
                params=params, pdf=("coherent", kin, amps), norm=("mc", 4000, 3))


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("n_res,nr", [(1, False), (1, True), (5, True), (8, True), (9, False), (14, True), (15, True)])
def test_shapes_match_oracle(goo, ctx, precision, n_res, nr):
    spec = _spec(n_res, nr)
    kin = synth.TD3_MASSES
    cands = synth.round_to_f32(synth.dalitz_candidates(80_000, 8, kin["M"], kin["m1"], kin["m2"], kin["m3"]), spec)
    mc = {k: v[-4000:] for k, v in cands.items()}
    ref = od.DalitzModel(spec)
    theta = np.array(synth.param_values(spec))
    theta[[p[0].startswith(("re_", "im_")) for p in spec["params"]]] *= 1.05
    mcds = goo.Dataset.from_spec(ctx, spec, mc)
    model = goo.Model(ctx, spec, mc=mcds)
    coef = np.array([p[0].startswith(("re_", "im_")) for p in spec["params"]])
    for n in (1, 31, 257, 5000, 77_825):
        data = {k: v[:n] for k, v in cands.items()}
        nll, g = model.nll_grad(goo.Dataset.from_spec(ctx, spec, data), theta, precision)
        rnll, rg = ref.nll_grad(data, mc, theta)
        assert abs(nll - rnll) <= TOL[precision] * max(abs(rnll), n), (n, nll, rnll)
        assert np.max(np.abs(g - rg)[coef]) <= TOL[precision] * max(np.max(np.abs(rg[coef])), n), (n, g, rg)
