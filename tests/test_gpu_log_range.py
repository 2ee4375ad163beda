"""The logarithm in the scattering width over thicknesses for which its fast
form holds and for which it does not (subnormal), against the oracle: FP64
fits with and without energy loss.  Tolerance: the FP64 contract (1e-9
relative, metrics in tests/metrics.py); the function itself is checked by
kf_selftest."""
import numpy as np
import pytest

import oracle
import paper_2105_01796_gb300 as kf
from paper_2105_01796_gb300 import synth
from tests.test_gpu_parity import FP64, compare, gpu_fit, handle  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("team", [0, 4])
@pytest.mark.parametrize("xx0", [0.0, 4e-320, 3e-308, 1e-40, 1e-9, 0.9, 40.0])
def test_scattering_width_over_thicknesses(handle, team, xx0):  # noqa: F811
    ev = dict(synth.make_event(synth.scaled(synth.WORKLOADS["tel10_1k"], 65)))
    ev["x_over_x0"] = ev["x_over_x0"].copy()
    ev["x_over_x0"][1::2] = xx0
    g = gpu_fit(handle, ev, FP64, team_warps=team)
    r = oracle.fit_batch(ev)
    assert (r["status"] == 0).all()
    compare(g, r, FP64)


def test_fast_functions_within_their_bounds():
    assert kf.kf_selftest(1 << 18)[5] == 0
