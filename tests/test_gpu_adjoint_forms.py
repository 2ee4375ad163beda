"""The adjoint's two kernels -- one thread per track, and a team of warps per 32
tracks whose reverse pass is a pipeline over them -- against each other and
against the fit: every value is computed by the same operations in the same
order, so chi2, the smoothed state 0 and the seed gradients are equal bit for
bit, and so are the values and those of the FP64 fit at zero alignment; the
alignment gradient sums over the tracks in any order (1e-12 of its scale).
Uneven tracks with holes in a part-filled last team, sub-steps (more steps than
the pipeline hands on), long corrections, fields along z, along no axis and
none."""
import numpy as np
import pytest

import paper_2105_01796_gb300 as kf
from paper_2105_01796_gb300 import synth
from tests.test_gpu_adjoint import _smoother_weights, _whole, handle  # noqa: F401
from tests.test_gpu_parity import FP64, gpu_fit

pytestmark = pytest.mark.gpu

VALUES = ("chi2", "params", "cov")


@pytest.mark.parametrize("objective", ["chi2", "whole"])
@pytest.mark.parametrize("nonzero", [False, True], ids=["zero", "aligned"])
@pytest.mark.parametrize("field,h_max,n_iter", [((0.0, 0.0, 2.0), 50.0, 3), ((0.4, -0.8, 1.7), 50.0, 3),
                                                ((0.4, -0.8, 1.7), 7.0, 2), ((0.0, 0.0, 2.0), 7.0, 3),
                                                ((0.0, 0.0, 0.0), 50.0, 1), ((1.0, -2.0, 7.5), 200.0, 3)])
def test_team_equals_one_thread(handle, field, h_max, n_iter, nonzero, objective):  # noqa: F811
    ev = dict(synth.make_event(synth.scaled(synth.WORKLOADS["uneven30_1m"], 333)))
    ev["bfield"] = np.array(field)
    S = ev["center"].shape[1]
    rng = np.random.default_rng(6)
    align = np.zeros((6, S))
    if nonzero:
        align[:3, 1:] = rng.normal(size=(3, S - 1)) * 0.05
        align[3:, 1:] = rng.normal(size=(3, S - 1)) * 5e-4
    v, W = _smoother_weights(ev) if objective == "whole" else (None, None)
    w = rng.uniform(0.5, 1.5, size=333)
    opt = dict(h_max=h_max, n_iter=n_iter)
    one = _whole(handle, ev, align, w, v, W, opt=kf.kf_default_options(block=64, **opt))
    team = _whole(handle, ev, align, w, v, W, opt=kf.kf_default_options(block=0, **opt))
    for k in VALUES + ("gs",):
        assert np.array_equal(one[k], team[k], equal_nan=True), k
    assert np.isfinite(one["gs"]).any() and np.isfinite(one["ga"]).all()
    assert np.allclose(team["ga"], one["ga"], rtol=1e-12, atol=1e-12 * np.abs(one["ga"]).max())
    if not nonzero:
        f = gpu_fit(handle, ev, FP64, team_warps=1, **opt)
        ok = f["status"] == 0
        for k in VALUES:
            assert np.array_equal(f[k][..., ok], team[k][..., ok]), k
            assert np.isnan(team[k][..., ~ok]).all(), k
