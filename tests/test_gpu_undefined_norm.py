"""A product whose normalisation is not a positive number (a polynomial of negative integral: log N is
NaN; a Gaussian that vanishes over the range: -log N is +inf) leaves no density wherever it is present,
whatever the other products are: both precisions report every such event, in every position of two to
four products, closed-form and grid normalisation, weighted or not."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N = 3001


@pytest.fixture(scope="module")
def goo():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1710_08826_gb300 import goo as g
    return g


@pytest.fixture(scope="module")
def ctx(goo):
    return goo.Context(0)


def _spec(undefined, position, n_prod, grid):
    params = [("a1", -1.0, False, 0.1), ("a2", 0.0, False, 0.1), ("mu", 1e3, False, 0.1), ("sig", 0.3, False, 0.1),
              ("mu2", 5.0, False, 0.1), ("sig2", 1e-7, False, 0.1), ("lam", -0.3, False, 0.1), ("m", 4.0, False, 0.1),
              ("s", 2.0, False, 0.1), ("f1", 0.3, False, 0.1), ("f2", 0.2, False, 0.1), ("f3", 0.2, False, 0.1)]
    # 1 - x over [0, 10] integrates to -40 (and is positive below 1); a Gaussian 330 widths off, or so narrow
    # that it vanishes at every bin centre
    bad = {"poly": ("poly2", "x", "a1", "a2"),
           "gauss": ("gauss", "x", "mu2", "sig2") if grid else ("gauss", "x", "mu", "sig")}[undefined]
    good = [("expo", "x", "lam"), ("gauss", "x", "m", "s"), ("expo", "x", "lam")][:n_prod - 1]
    return dict(name="undefined", observables=[("x", 0.0, 10.0)], params=params,
                pdf=("add", ["f1", "f2", "f3"][:n_prod - 1], good[:position] + [bad] + good[position:]),
                norm=("grid", [64]) if grid else ("analytic",))


@pytest.mark.parametrize("grid", [False, True])
@pytest.mark.parametrize("n_prod,position", [(2, 0), (2, 1), (3, 0), (3, 1), (4, 2), (4, 3)])
@pytest.mark.parametrize("undefined", ["poly", "gauss"])
def test_no_event_has_a_density(goo, ctx, undefined, n_prod, position, grid):
    spec = _spec(undefined, position, n_prod, grid)
    x = np.random.default_rng(1).uniform(0.0, 10.0, N)
    model = goo.Model(ctx, spec)
    theta = np.array([p[1] for p in spec["params"]])
    for weighted in (False, True):
        ds = goo.Dataset.from_spec(ctx, spec, {"x": x})
        if weighted:
            ds.set_weights(np.full(N, 0.5))
        for precision in ("f64", "f32"):
            for call in (model.nll, model.nll_grad):
                with pytest.raises(goo.GooError) as e:
                    call(ds, theta, precision)
                assert e.value.code == goo.GOO_ERR_NONPOSITIVE_PDF
                assert f"for {N} events" in str(e.value)
