"""Rounding errors of the FP64 fit, against the fit in extended precision: the
closed-form transport, the fixed-point smoother and the fast helpers lose
nothing against a plain double-precision evaluation of the method (the oracle,
stage by stage, with the backward smoother).  The root mean square errors of
parameters, covariances and chi2 over the tracks (metrics in tests/metrics.py)
are held to those of the oracle, which has the same inputs and the same 53
bits."""
import numpy as np
import pytest

import oracle
from paper_2105_01796_gb300 import synth
from tests import extended
from tests.metrics import chi2_err, cov_err, param_err
from tests.test_gpu_parity import FP64, gpu_fit, handle  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return extended.build(str(tmp_path_factory.mktemp("extended")))


def _errors(g, ref):
    ok = ref["status"] == 0
    e = (param_err(g["params"], ref["params"], ref["cov"]), cov_err(g["cov"], ref["cov"]),
         chi2_err(g["chi2"], ref["chi2"]))
    return [float(np.sqrt(np.mean(np.square(x[..., ok])))) for x in e]


@pytest.mark.parametrize("form", [dict(team_warps=1), dict(team_warps=4), dict(energy_loss=1)],
                         ids=["one_thread", "team", "energy_loss"])
@pytest.mark.parametrize("wl,field", [("tel10_1k", (0.0, 0.0, 2.0)), ("tel30_100k", (0.0, 0.0, 2.0)),
                                      ("uneven30_1m", (0.4, -0.8, 1.7)), ("align20_100k", (0.0, 0.0, 2.0))])
def test_errors_no_larger_than_a_plain_evaluation(handle, lib, wl, field, form):  # noqa: F811
    ev = dict(synth.make_event(synth.scaled(synth.WORKLOADS[wl], 400)))
    ev["bfield"] = np.array(field)
    eloss = "energy_loss" in form
    ref = extended.fit_batch(lib, ev, energy_loss=eloss)
    plain = oracle.fit_batch(ev, method=dict(energy_loss=True) if eloss else None)
    g = gpu_fit(handle, ev, FP64, **form)
    assert (ref["status"] == 0).mean() > 0.9
    assert np.array_equal(g["status"], ref["status"]) and np.array_equal(plain["status"], ref["status"])
    kernel, bound = _errors(g, ref), _errors(plain, ref)
    assert all(k <= b for k, b in zip(kernel, bound)), (kernel, bound)


@pytest.mark.parametrize("form", [dict(team_warps=1), dict(team_warps=4), dict(energy_loss=1)],
                         ids=["one_thread", "team", "energy_loss"])
@pytest.mark.parametrize("field", [(0.0, 0.0, 2.0), (0.4, -0.8, 1.7)])
def test_loose_prior_and_precise_hits(handle, lib, field, form):  # noqa: F811
    """A seed that knows one angle to 0.3 rad and hits of 1 um in axes turned by
    45 degrees: both coordinates of a hit see that angle, so the innovation's
    covariance is ill-conditioned (81 mm^2 against 1e-6 at the first plane) and
    the smoothed variances are 1e-7 of the prior's.  A stable update loses what
    rounding at the prior's size costs: 100 roundings (about ten in each of the
    ten updates) of the largest ratio of prior to smoothed variance."""
    ev = dict(synth.make_event(synth.scaled(synth.WORKLOADS["tel10_1k"], 97)))
    ev["bfield"] = np.array(field)
    R = ev["rot"].reshape(3, 3, -1).copy()
    u, v = R[:, 0].copy(), R[:, 1].copy()
    s = np.sqrt(0.5)
    R[:, 0], R[:, 1] = s * (u + v), s * (v - u)
    ev["rot"] = np.ascontiguousarray(R.reshape(9, -1))
    turn = np.array([[s, s], [-s, s]])
    ev["loc"] = turn @ ev["loc"]
    ev["cov"] = np.repeat(np.array([[1e-6], [0.0], [1e-6]]), ev["loc"].shape[1], 1)
    ev["seed_params"] = ev["seed_params"].copy()
    ev["seed_params"][:2] = turn @ ev["seed_params"][:2]
    c = np.zeros_like(ev["seed_cov"])
    c[[0, 2, 5, 9, 14, 20]] = np.array([1.0, 1.0, 0.09, 1e-8, 1e-2, 1.0])[:, None]
    ev["seed_cov"] = c
    eloss = "energy_loss" in form
    ref = extended.fit_batch(lib, ev, energy_loss=eloss)
    g = gpu_fit(handle, ev, FP64, **form)
    assert (ref["status"] == 0).all() and (g["status"] == 0).all()
    diag = [0, 2, 5, 9, 14, 20]
    bound = 100 * 2.0 ** -53 * (c[diag] / ref["cov"][diag].astype(np.float64)).max(0)
    assert bound.min() > 1e-10 and bound.max() < 1e-4
    err = cov_err(g["cov"], ref["cov"]).max(0)
    assert np.all(err < bound), float((err / bound).max())
