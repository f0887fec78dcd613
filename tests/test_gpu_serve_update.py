"""A toy server takes its normalisation from the Gram matrix as it is when the server is made: after new
events in the MC sample (goo_dataset_update, the lineshapes unchanged) its fits are those of a model made
on those events."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

KIN = synth.DALITZ_MASSES


@pytest.fixture(scope="module")
def goo():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1710_08826_gb300 import goo as g
    return g


def test_server_after_an_update_of_the_sample(goo):
    ctx = goo.Context(0)
    spec = synth.c3_spec(n_mc=400_000)
    theta = np.array(synth.param_values(spec))
    obs = [o[0] for o in spec["observables"]]
    first, second = (synth.round_to_f32(synth.dalitz_candidates(400_000, s, KIN["M"], KIN["m1"], KIN["m2"], KIN["m3"]), spec)
                     for s in (3, 4))
    start = theta.copy()
    start[[not p[2] for p in spec["params"]]] *= 1.05

    def fits(model):
        server = goo.Server(model, theta)
        tickets = [server.submit(n, 1710600 + n, start) for n in (2000, 9000)]
        for _ in range(2000):
            queued, active, _ = server.step()
            if queued == 0 and active == 0:
                break
        return [server.result(t) for t in tickets]

    mcds = goo.Dataset.from_spec(ctx, spec, first)
    model = goo.Model(ctx, spec, mc=mcds)
    old = fits(model)
    mcds.update([second[o] for o in obs])
    new = fits(model)
    want = fits(goo.Model(ctx, spec, mc=goo.Dataset.from_spec(ctx, spec, second)))
    for o, a, b in zip(old, new, want):
        assert np.array_equal(a[0], b[0]) and not np.array_equal(a[0], o[0])
