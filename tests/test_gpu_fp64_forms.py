"""One thread per track, and teams of 2 and 4 warps, over the edge cases of the
FP64 path: the one-thread kernel against the oracle (the FP64 contract, 1e-9),
the teams equal to it bit for bit, with and without smoothed states.  (A batch
of this size goes to teams when the launch shape is left to the library:
team_warps = 1 names the one-thread kernel.)"""
import numpy as np
import pytest

import oracle
from tests.metrics import state_sigmas, states_err
from tests.test_gpu_fp64_path import _event
from tests.test_gpu_parity import FP64, _edge_event, compare, gpu_fit, handle  # noqa: F401

pytestmark = pytest.mark.gpu

I44, I54, I55 = 14, 19, 20


def _strong_field(field):
    ev = _event()
    ev["bfield"] = np.array(field)
    hole = ev["is_hole"].reshape(-1, 11).copy()
    hole[:, 3:] = 1  # the hits belong to 2 T
    ev["is_hole"] = hole.reshape(-1)
    return ev


def _turned():
    ev = _event()
    s = ev["seed_params"].copy()
    s[2, 0::3] += 2 * np.pi
    s[3, 1::3] = -s[3, 1::3]
    s[2, 1::3] += np.pi
    s[3, 2::3] += 2 * np.pi
    ev["seed_params"] = s
    return ev


def _verdict():
    ev = _event(64)
    c = ev["seed_cov"].copy()
    c[I54] = np.where(np.arange(64) % 2 == 0, 1.0 - 1e-7, 1.5) * np.sqrt(c[I44] * c[I55])
    ev["seed_cov"] = c
    return ev


def _small_time_error():
    ev = _event()
    c = ev["seed_cov"].copy()
    c[I55, 0::3] = 1e-12
    ev["seed_cov"] = c
    return ev


def _thickness(xx0):
    ev = _event(65)
    ev["x_over_x0"] = ev["x_over_x0"].copy()
    ev["x_over_x0"][1::2] = xx0
    return ev


CASES = {
    "8T along z, long corrections": (lambda: _strong_field((0.0, 0.0, 8.0)), dict(h_max=200.0, n_iter=3)),
    "8T along z, one correction": (lambda: _strong_field((0.0, 0.0, 8.0)), dict(h_max=200.0, n_iter=1)),
    "8T along no axis, long corrections": (lambda: _strong_field((1.0, -2.0, 7.5)), dict(h_max=200.0, n_iter=3)),
    "8T along no axis, sub-steps": (lambda: _strong_field((1.0, -2.0, 7.5)), dict(h_max=7.0, n_iter=2)),
    "no field, sub-steps": (lambda: _strong_field((0.0, 0.0, 0.0)), dict(h_max=7.0, n_iter=2)),
    "start angles out of range": (_turned, {}),
    "positivity left to the FP64 pivots": (_verdict, {}),
    "time carried along": (_small_time_error, {}),
    "short tracks, holes, bad input": (_edge_event, {}),
    "subnormal thickness": (lambda: _thickness(4e-320), {}),
    "thick planes": (lambda: _thickness(40.0), {}),
}


@pytest.mark.parametrize("name", CASES)
def test_forms_agree(handle, name):  # noqa: F811
    make, opt = CASES[name]
    ev = make()
    r = oracle.fit_batch(ev, with_states=True, **opt)
    assert (r["status"] == 0).mean() >= 0.5
    for states in (False, True):
        one = gpu_fit(handle, ev, FP64, with_states=states, team_warps=1, **opt)
        compare(one, r, FP64)
        if states:
            ok = np.repeat(r["status"] == 0, np.diff(ev["offsets"].astype(np.int64)))
            err = states_err(one["states"][:, ok], r["states"][:, ok], state_sigmas(ev, **opt)[:, ok])
            assert err.max() < 1e-9, err.max()
        for team in (2, 4):
            g = gpu_fit(handle, ev, FP64, with_states=states, team_warps=team, **opt)
            for k in one:
                if one[k] is not None:
                    assert np.array_equal(one[k], g[k], equal_nan=True), (team, states, k)
