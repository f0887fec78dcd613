"""FP64 sum of products where the product with the larger exponent has weight 0 (a fraction at its limit)
and the other lies 672 to 724 e-folds below it: the density is the other's, down to where the
exponential of the difference is 0, in two and in three products."""
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
@pytest.mark.parametrize("n_prod", [2, 3])
def test_a_product_of_weight_zero(goo, n_prod, order):
    params = [("mu", 5.0, False, 0.1), ("sig", 0.1, False, 0.1), ("lam", -0.3, False, 0.1), ("f", 1.0, False, 0.1),
              ("g", 0.0, False, 0.1)]
    gauss, expo = ("gauss", "x", "mu", "sig"), ("expo", "x", "lam")
    prods = [gauss, expo] if order == 0 else [expo, gauss]
    fracs = ["f"] if order == 0 else ["g"]
    if n_prod == 3:
        prods, fracs = prods + [expo], fracs + ["g" if order == 0 else "f"]
    spec = dict(name="far", observables=[("x", 0.0, 10.0)], params=params, pdf=("add", fracs, prods), norm=("analytic",))
    theta = np.array([p[1] for p in params])
    x = 5.0 + 0.1 * np.array([36.8, 37.2, 37.5, 37.8, 38.0, 38.2])
    ctx = goo.Context(0)
    model = goo.Model(ctx, spec)
    ds = goo.Dataset.from_spec(ctx, spec, {"x": x})
    logn = np.log(0.1 * np.sqrt(2.0 * np.pi))  # the range holds the whole Gaussian
    want = float(np.sum(0.5 * ((x - 5.0) / 0.1) ** 2 + logn))
    # subnormal exponentials, rounded to 2^-1075: 1e-9 of the smallest, exp(-724.4)
    assert model.nll(ds, theta, "f64") == pytest.approx(want, abs=1e-7)
    nll, _ = model.nll_grad(ds, theta, "f64")  # the derivative by the fraction overflows
    assert nll == pytest.approx(want, abs=1e-7)
    assert float(-model.eval_logf(ds, theta, "f64").sum()) == pytest.approx(nll, abs=1e-9 * want)
