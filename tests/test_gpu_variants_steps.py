"""The variant kernel's transports at their edges against the oracle with the
same variants (FP64 contract, 1e-9): a constant general field and no field,
sub-steps and 0 to 5 plane corrections (full, tiny and standing steps of the
map propagation), smoothed state 0 alone and every state."""
import numpy as np
import pytest

import oracle
from paper_2105_01796_gb300 import synth
from tests.test_gpu_parity import FP64, compare, gpu_fit, handle  # noqa: F401
from tests.test_gpu_variants import BACKWARD, ELOSS, kopts, states_err

pytestmark = pytest.mark.gpu

ALL = dict(BACKWARD, **ELOSS)


@pytest.mark.parametrize("h_max,n_iter", [(50.0, 3), (50.0, 1), (50.0, 2), (7.0, 5), (50.0, 0)])
@pytest.mark.parametrize("method", [None, ELOSS, ALL], ids=["rts", "eloss", "all"])
def test_map_steps(handle, method, h_max, n_iter):  # noqa: F811
    ev = synth.make_event(synth.scaled(synth.WORKLOADS["fringe30_100k"], 97))
    opt = dict(h_max=h_max, n_iter=n_iter)
    r = oracle.fit_batch(ev, with_states=True, method=method, **opt)
    g = gpu_fit(handle, ev, FP64, with_states=True, **kopts(method), **opt)
    compare(g, r, FP64)
    assert states_err(g, r, ev) < 1e-9
    one = gpu_fit(handle, ev, FP64, **kopts(method), **opt)  # no states wanted
    for k in ("params", "cov", "chi2", "status"):
        assert np.array_equal(one[k], g[k], equal_nan=True), k


@pytest.mark.parametrize("field", [(0.4, -0.8, 1.7), (0.0, 0.0, 0.0)])
@pytest.mark.parametrize("method", [BACKWARD, ELOSS, ALL], ids=["backward", "eloss", "all"])
def test_constant_fields(handle, method, field):  # noqa: F811
    ev = dict(synth.make_event(synth.scaled(synth.WORKLOADS["uneven30_1m"], 333)))
    ev["bfield"] = np.array(field)
    r = oracle.fit_batch(ev, with_states=True, method=method)
    g = gpu_fit(handle, ev, FP64, with_states=True, **kopts(method))
    compare(g, r, FP64)
    assert states_err(g, r, ev) < 1e-9
