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
