"""Every gradient lane of the floating-lineshape kernel on its own scale: the error of component p against
the sum of the magnitudes of its terms, sum_i |d log |S_i|^2 / d p| of the events and n sum_j |d |S_j|^2 / d p| /
sum_j |S_j|^2 of the normalisation sample, so that no coefficient, mass or width can be wrong by a
large fraction of itself behind a larger one."""
import numpy as np
import pytest
import torch

import synth
from oracle import dalitz as od
from test_gpu_coherent_shapes import _spec

pytestmark = pytest.mark.gpu

# FP64: sums carried to 2^-48, the two sides' amplitudes differ by rounding.  FP32: m0^2 - s at a resonance
# of width Gamma0 is good to 2^-25 m0 / Gamma0 (4e-7 for the narrowest here), and a mass's or width's terms are
# made of up to three sums several times their size
TOL = {"f64": 1e-11, "f32": 2e-5}


@pytest.fixture(scope="module")
def goo():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1710_08826_gb300 import goo as g
    return g


@pytest.fixture(scope="module")
def ctx(goo):
    return goo.Context(0)


def _scales(ref, data, mc, theta):
    def s2(cols, th):
        th = torch.as_tensor(th)
        with torch.no_grad():
            return ref.intensity(ref.amplitude_matrix(cols, th), th).numpy()
    n, s_mc, out = len(data["s12"]), s2(mc, theta), np.zeros(len(theta))
    for p in range(len(theta)):
        h = 1e-6 * max(abs(theta[p]), 0.1)
        up, dn = theta.copy(), theta.copy()
        up[p] += h
        dn[p] -= h
        out[p] = np.sum(np.abs(np.log(s2(data, up) / s2(data, dn)))) / (2 * h)
        out[p] += n * np.sum(np.abs(s2(mc, up) - s2(mc, dn))) / (2 * h) / np.sum(s_mc)
    return out


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("n_res,nr,n_mc", [(3, True, 4001), (8, True, 4001), (9, False, 100), (15, True, 4000)])
def test_each_lane_on_its_own_scale(goo, ctx, precision, n_res, nr, n_mc):
    spec = _spec(n_res, nr)
    kin = synth.TD3_MASSES
    cands = synth.round_to_f32(synth.dalitz_candidates(40_000, 12, kin["M"], kin["m1"], kin["m2"], kin["m3"]), spec)
    mc = {k: v[-n_mc:] for k, v in cands.items()}
    theta = np.array(synth.param_values(spec))
    theta[[p[0].startswith(("re_", "im_")) for p in spec["params"]]] *= 1.05
    ref = od.DalitzModel(spec)
    model = goo.Model(ctx, spec, mc=goo.Dataset.from_spec(ctx, spec, mc))
    model.set_lineshapes("floating")
    for n in (257, 30_001):
        data = {k: v[:n] for k, v in cands.items()}
        g = model.nll_grad(goo.Dataset.from_spec(ctx, spec, data), theta, precision)[1]
        rg, scale = ref.nll_grad(data, mc, theta)[1], _scales(ref, data, mc, theta)
        err = np.abs(g - rg) / scale
        print(f"n = {n}: {err.max():.2e} ({spec['params'][int(err.argmax())][0]})")
        assert np.all(err <= TOL[precision]), (n, err)
        if precision == "f32" and n == 30_001:  # a coefficient to a hundredth of the events' own fluctuation
            coef = [p[0].startswith(("re_", "im_")) for p in spec["params"]]
            assert np.max(np.abs(g - rg)[coef]) <= 0.01 * np.sqrt(n)
