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
import paper_2105_01796_gb300 as kf
from paper_2105_01796_gb300 import synth
from tests import extended
from tests.metrics import DIAG, chi2_err, cov_err, param_err
from tests.test_gpu_adjoint import _whole
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


def _loose_prior(field):
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
    c[DIAG] = np.array([1.0, 1.0, 0.09, 1e-8, 1e-2, 1.0])[:, None]
    ev["seed_cov"] = c
    return ev


def _roundings(ev, ref):
    return 100 * 2.0 ** -53 * (ev["seed_cov"][DIAG] / ref["cov"][DIAG].astype(np.float64)).max(0)


@pytest.mark.parametrize("form", [dict(team_warps=1), dict(team_warps=4), dict(energy_loss=1)],
                         ids=["one_thread", "team", "energy_loss"])
@pytest.mark.parametrize("field", [(0.0, 0.0, 2.0), (0.4, -0.8, 1.7)])
def test_loose_prior_and_precise_hits(handle, lib, field, form):  # noqa: F811
    ev = _loose_prior(field)
    ref = extended.fit_batch(lib, ev, energy_loss="energy_loss" in form)
    g = gpu_fit(handle, ev, FP64, **form)
    assert (ref["status"] == 0).all() and (g["status"] == 0).all()
    bound = _roundings(ev, ref)
    assert bound.min() > 1e-10 and bound.max() < 1e-4
    err = cov_err(g["cov"], ref["cov"]).max(0)
    assert np.all(err < bound), float((err / bound).max())


@pytest.mark.parametrize("team", [1, 2])
@pytest.mark.parametrize("whole", [False, True], ids=["chi2", "whole"])
@pytest.mark.parametrize("field", [(0.0, 0.0, 2.0), (0.4, -0.8, 1.7)])
def test_gradients_of_a_loose_prior(handle, lib, field, whole, team):  # noqa: F811
    """The seed gradients of the same tracks against central differences of the
    extended fit (step 1e-12: with 113 bits their own error is below 1e-12): the
    gradients' contract, 1e-5, of the track's largest one."""
    if np.finfo(np.longdouble).nmant < 100:
        pytest.skip("long double is too short for the differences on this host")
    ev = _loose_prior(field)
    v, W = (np.ones((6, 97)), np.ones((21, 97))) if whole else (None, None)

    def objective(seed):
        r = extended.fit_batch(lib, dict(ev, seed_params=seed))
        assert (r["status"] == 0).all()
        return r["chi2"] + (r["params"].sum(0) + r["cov"].sum(0) if whole else 0)

    h = np.longdouble(1e-12)
    fd = np.zeros((6, 97))
    for i in range(6):
        up, dn = (ev["seed_params"].astype(np.longdouble) for _ in range(2))
        up[i] += h
        dn[i] -= h
        fd[i] = (objective(up) - objective(dn)) / (2 * h)
    g = _whole(handle, ev, np.zeros((6, ev["center"].shape[1])), None, v, W,
               opt=kf.kf_default_options(block=0, team_warps=team))
    err = np.abs(g["gs"] - fd).max(0) / np.abs(fd).max(0)
    assert err.max() < 1e-5, err.max()
