"""The Gram matrices' sums apart from the amplitudes: every element against the FP64 sum, on the host, of the
library's own cached amplitudes, at sample sizes around one event per thread, a run of events summed
plainly, a block, and a million."""
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


@pytest.fixture(scope="module")
def ctx(goo):
    return goo.Context(0)


@pytest.fixture(scope="module")
def sample():
    kin = synth.TD3_MASSES
    return synth.round_to_f32(synth.dalitz_candidates(1_000_003, 13, kin["M"], kin["m1"], kin["m2"], kin["m3"]), _spec(1, True))


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("n_res,nr", [(2, False), (8, True), (15, True)])
@pytest.mark.parametrize("n", [1, 15, 17, 385, 6145, 1_000_003])
def test_sums(goo, ctx, sample, n, n_res, nr, precision):
    spec = _spec(n_res, nr)
    theta = np.array(synth.param_values(spec))
    mcds = goo.Dataset.from_spec(ctx, spec, {k: v[:n] for k, v in sample.items()})
    model = goo.Model(ctx, spec, mc=mcds)
    G = model.gram(theta, precision)
    a = model.amplitudes(mcds, theta, precision).astype(np.complex128)
    if nr:
        a = np.concatenate([a, np.ones((n, 1))], axis=1)
    ref, size = a.T @ a.conj() / n, np.abs(a).T @ np.abs(a) / n
    # FP32: 32 FMAs of a run of 16 events round a partial sum of 8 events on average, 2^-25 * 52 / 16 of an
    # event's product per event and run, independent from run to run: 8 standard deviations are 3.1e-6 / sqrt(n).
    # FP64: chains of FMAs, then 2^-48 per addition
    tol = 1e-13 if precision == "f64" else 3.1e-6 / np.sqrt(n) + 1e-12
    err = np.abs(G - ref) / size
    print(f"n = {n}: {err.max():.2e}")
    assert np.all(err <= tol), err.max()
