"""Weighted FP32 sum of products with a fraction at its limit: the larger product has weight 0 and the other
lies 88 to 94 e-folds below it, where its share is a subnormal float.  The density is the other product's, and
events of a weight beside it count as ever."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def goo():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1710_08826_gb300 import goo as g
    return g


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("n", [5, 700])
def test_subnormal_shares(goo, n, order):
    params = [("mu", 5.0, False, 0.1), ("sig", 0.1, False, 0.1), ("lam", -0.3, False, 0.1), ("f", 1.0, False, 0.1),
              ("g", 0.0, False, 0.1)]
    gauss, expo = ("gauss", "x", "mu", "sig"), ("expo", "x", "lam")
    spec = dict(name="far", observables=[("x", 0.0, 10.0)], params=params, norm=("analytic",),
                pdf=("add", ["f" if order == 0 else "g"], [gauss, expo] if order == 0 else [expo, gauss]))
    theta = np.array([p[1] for p in params])
    # log of the exponential's density less the Gaussian's
    grid = np.linspace(6.0, 6.7, 20_001).astype(np.float32).astype(np.float64)
    gap = (-0.3 * grid - np.log(-np.expm1(-3.0) / 0.3)) + 0.5 * ((grid - 5.0) / 0.1) ** 2 + np.log(0.1 * np.sqrt(2.0 * np.pi))
    far = grid[(gap > 88.0) & (gap < 94.0)]
    x = np.resize(np.concatenate([far, np.linspace(4.5, 5.5, far.size).astype(np.float32).astype(np.float64)]), n)
    w = np.random.default_rng(2).uniform(0.5, 1.5, n).astype(np.float32).astype(np.float64)
    ctx = goo.Context(0)
    model = goo.Model(ctx, spec)
    ds = goo.Dataset.from_spec(ctx, spec, {"x": x})
    ds.set_weights(w)
    want = model.nll(ds, theta, "f64")
    # steps of 2^-149 / exp(-94) = 1e-3 for each event
    assert abs(model.nll(ds, theta, "f32") - want) <= 1e-3 * w.sum()
    assert abs(model.nll_grad(ds, theta, "f32")[0] - want) <= 1e-3 * w.sum()
