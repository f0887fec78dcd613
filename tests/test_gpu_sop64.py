"""The FP64 event kernel of the sum-of-products models against the oracle: one to four products,
events beyond an Argus endpoint (an absent product), weights with zeros, and event counts around
a warp, a block and a grid-stride step."""
import numpy as np
import pytest

import synth
from oracle import model as om

pytestmark = pytest.mark.gpu

TOL_NLL, TOL_GRAD = 1e-11, 1e-9  # both sides in FP64; sums are carried to 2^-48


@pytest.fixture(scope="module")
def goo():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1710_08826_gb300 import goo as g
    return g


@pytest.fixture(scope="module")
def ctx(goo):
    return goo.Context(0)


def _spec(n_prod):
    """The first n_prod of: Argus x Poly2 x Expo, Gauss x Gauss x Expo, Poly2 x Expo, Gauss on m, dE, t."""
    spec = synth.c2_spec(bins=32)
    _, _, (sig, bkg) = spec["pdf"]
    extra = [("b1", 0.7, False, 0.01), ("b2", -0.02, False, 0.01), ("lam_3", -0.4, False, 0.01),
             ("mu_t", 3.0, False, 0.01), ("sig_t", 1.5, False, 0.01), ("f1", 0.3, False, 0.01), ("f2", 0.2, False, 0.01),
             ("f3", 0.25, False, 0.01)]
    prods = [bkg, sig, ("prod", [("poly2", "dE", "b1", "b2"), ("expo", "t", "lam_3"), ("gauss", "m", "mu_m", "sig_m")]),
             ("gauss", "t", "mu_t", "sig_t")][:n_prod]
    pdf = prods[0] if n_prod == 1 else ("add", ["f1", "f2", "f3"][:n_prod - 1], prods)
    return dict(spec, params=[p for p in spec["params"] if p[0] != "frac"] + extra, pdf=pdf)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("n_prod", [1, 2, 3, 4])
def test_products_weights_and_sizes(goo, ctx, n_prod, weighted):
    spec = _spec(n_prod)
    cols = synth.gen_c2(n=77_825, seed=31)
    if n_prod > 1:   # beyond the endpoint m0 = 5.29 the Argus product is absent
        cols["m"][::7] = np.random.default_rng(4).uniform(5.285, 5.2999, cols["m"][::7].size)
    w = np.random.default_rng(5).uniform(0.2, 2.0, 77_825) * (np.random.default_rng(6).uniform(size=77_825) > 0.2)
    w[0] = 0.5
    ref, model = om.TreeModel(spec), goo.Model(ctx, spec)
    theta = np.array(synth.param_values(spec)) * 1.002
    if n_prod == 1:  # every event has to lie below the endpoint
        theta[[p[0] for p in spec["params"]].index("m0")] = 5.31
    for n in (1, 255, 257, 77_825):
        data = {k: v[:n] for k, v in cols.items()}
        ds = goo.Dataset.from_spec(ctx, spec, data)
        if weighted:
            ds.set_weights(w[:n])
        nll, g = model.nll_grad(ds, theta, "f64")
        rnll, rg = ref.nll_grad(data, theta, weights=w[:n]) if weighted else ref.nll_grad(data, theta)
        assert abs(nll - rnll) <= TOL_NLL * max(abs(rnll), n), (n, nll, rnll)
        assert np.max(np.abs(g - rg)) <= TOL_GRAD * max(np.max(np.abs(rg)), n), (n, g, rg)
        assert model.nll(ds, theta, "f64") == pytest.approx(nll, rel=1e-12)


def test_no_density_is_reported(goo, ctx):
    # an Argus density alone vanishes beyond its endpoint: the evaluation counts those events
    spec = _spec(1)
    cols = {k: v[:1000] for k, v in synth.gen_c2(n=1000, seed=32).items()}
    cols["m"][[3, 900]] = 5.2999
    theta = np.array(synth.param_values(spec))
    with pytest.raises(goo.GooError) as e:
        goo.Model(ctx, spec).nll_grad(goo.Dataset.from_spec(ctx, spec, cols), theta, "f64")
    assert e.value.code == goo.GOO_ERR_NONPOSITIVE_PDF


@pytest.mark.parametrize("n_poly", [1, 2])
@pytest.mark.parametrize("zero", [False, True])
def test_polynomials_of_a_product(goo, ctx, n_poly, zero):
    # one polynomial in a product takes 1 / r from the other factors, two take reciprocals; where
    # the polynomial is zero the product vanishes and the others remain
    spec = synth.c2_spec(bins=32)
    _, _, (sig, bkg) = spec["pdf"]
    extra = [("q1", 0.05, False, 0.01), ("q2", 0.01, False, 0.01)]
    leaves = list(bkg[1])
    if n_poly == 2:
        leaves = [("poly2", "t", "q1", "q2") if l[0] == "expo" else l for l in leaves]
    spec = dict(spec, params=spec["params"] + (extra if n_poly == 2 else []),
                pdf=("add", spec["pdf"][1], [sig, ("prod", leaves)]))
    cols = {k: v[:20_001] for k, v in synth.gen_c2(n=20_001, seed=33).items()}
    theta = np.array(synth.param_values(spec))
    poly = next(l for l in leaves if l[0] == "poly2" and l[1] == "dE")
    names = [p[0] for p in spec["params"]]
    lanes = np.ones(len(names), bool)
    if zero:   # (1 - 8 dE)^2, zero for every ninth event; the lanes x / r leave out a vanished product
        theta[names.index(poly[2])], theta[names.index(poly[3])] = -16.0, 64.0
        cols["dE"][::9] = 0.125
        lanes[[names.index(poly[2]), names.index(poly[3])]] = False
    ref, model = om.TreeModel(spec), goo.Model(ctx, spec)
    nll, g = model.nll_grad(goo.Dataset.from_spec(ctx, spec, cols), theta, "f64")
    rnll, rg = ref.nll_grad(cols, theta)
    assert abs(nll - rnll) <= TOL_NLL * max(abs(rnll), 20_001), (nll, rnll)
    assert np.max(np.abs(g - rg)[lanes]) <= TOL_GRAD * max(np.max(np.abs(rg[lanes])), 20_001), (g, rg)
    assert np.all(np.isfinite(g))
