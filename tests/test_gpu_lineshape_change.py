"""Evaluations after a lineshape change: the caches, the Gram matrices and the likelihood are queued
so that their kernels overlap; the result is bit for bit that of a model and datasets built afresh
at the new lineshapes (every sum has a fixed order)."""
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


@pytest.fixture(scope="module")
def ctx(goo):
    return goo.Context(0)


def _spec(kind):
    if kind == "td3":
        return synth.td3_spec(), synth.TD3_MASSES
    return synth.c3_spec(n_mc=1000), synth.DALITZ_MASSES


def _cols(kind, kin, n, seed):
    cols = synth.dalitz_candidates(n, seed, kin["M"], kin["m1"], kin["m2"], kin["m3"])
    if kind == "td3":
        cols["t"] = np.random.default_rng(seed).exponential(0.4, n)
    return cols


@pytest.mark.parametrize("kind", ["dalitz", "td3"])
@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("n,n_mc", [(1, 50_000), (300_001, 1), (200_000, 70_001), (5_001, None)])
def test_same_as_built_afresh(goo, ctx, kind, precision, n, n_mc):
    spec, kin = _spec(kind)
    data = synth.round_to_f32(_cols(kind, kin, n, 3), spec)
    mc = data if n_mc is None else synth.round_to_f32(_cols(kind, kin, n_mc, 4), spec)   # None: one dataset for both

    def build():
        ds = goo.Dataset.from_spec(ctx, spec, data)
        mcds = ds if n_mc is None else goo.Dataset.from_spec(ctx, spec, mc)
        return ds, goo.Model(ctx, spec, mc=mcds), mcds
    ds, model, keep = build()
    theta = np.array(synth.param_values(spec))
    mass = next(i for i, name in enumerate(synth.param_names(spec)) if name.startswith("m0_"))
    walk, fresh = [], []
    for step in range(4):
        theta[mass] += 2e-3
        walk.append(model.nll_grad(ds, theta, precision))
        ds2, model2, keep2 = build()
        fresh.append(model2.nll_grad(ds2, theta, precision))
    for (a, ga), (b, gb) in zip(walk, fresh):
        assert a == b
        assert np.array_equal(ga, gb)
    assert n == 1 or len({a for a, _ in walk}) == 4
