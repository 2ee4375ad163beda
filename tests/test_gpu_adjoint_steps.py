"""The adjoint's reverse through the path's steps and corrections away from
the default stepping, against the oracle's central differences with the same
stepping (element-wise 1e-5 above the differences' own resolution, as in
test_gpu_adjoint): sub-steps, 0 to 5 corrections, corrections too long to be
summed (a strong field), a field along no axis and none, uneven tracks with
holes, a measured state 0, every register variant."""
import functools

import numpy as np
import pytest

import oracle
import paper_2105_01796_gb300 as kf
from paper_2105_01796_gb300 import synth
from tests.test_gpu_adjoint import _check_grads, _fd2, _smoother_weights, _whole, handle  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = [  # workload, field, h_max, n_iter, options
    ("align20_100k", (0.0, 0.0, 2.0), 7.0, 3, {}),
    ("align20_100k", (0.4, -0.8, 1.7), 50.0, 2, {}),
    ("align20_100k", (0.4, -0.8, 1.7), 7.0, 1, dict(min_blocks=3)),
    ("align20_100k", (0.0, 0.0, 2.0), 50.0, 0, {}),
    ("align20_100k", (0.0, 0.0, 0.0), 50.0, 5, dict(min_blocks=4)),
    ("tel10_1k", (0.0, 0.0, 8.0), 200.0, 3, {}),
    ("tel10_1k", (1.0, -2.0, 7.5), 200.0, 2, {}),
    ("uneven30_1m", (0.0, 0.0, 2.0), 50.0, 3, {}),
]


@pytest.mark.parametrize("wl,field,h_max,n_iter,opt", CASES)
def test_stepping(handle, monkeypatch, wl, field, h_max, n_iter, opt):  # noqa: F811
    n = 24
    ev = dict(synth.make_event(synth.scaled(synth.WORKLOADS[wl], n)))
    ev["bfield"] = np.array(field)
    if wl == "tel10_1k":  # the hits belong to 2 T: only the first planes measure
        hole = ev["is_hole"].reshape(-1, 11).copy()
        hole[:, 4:] = 1
        ev["is_hole"] = hole.reshape(-1)
    if wl == "uneven30_1m":  # the seed's plane measures too
        first = ev["offsets"][:-1]
        ev["is_hole"] = ev["is_hole"].copy()
        ev["is_hole"][first] = 0
        ev["loc"] = ev["loc"].copy()
        ev["loc"][:, first] = ev["seed_params"][:2] + 0.05
        ev["cov"] = ev["cov"].copy()
        ev["cov"][:, first] = np.array([[0.04], [0.01], [0.09]])
    S = ev["center"].shape[1]
    rng = np.random.default_rng(4)
    align = np.zeros((6, S))
    align[:3, 1:] = rng.normal(size=(3, S - 1)) * 0.05
    align[3:, 1:] = rng.normal(size=(3, S - 1)) * 5e-4
    monkeypatch.setattr(oracle, "fit_batch", functools.partial(oracle.fit_batch, h_max=h_max, n_iter=n_iter))
    v, W = _smoother_weights(ev)
    w = rng.uniform(0.5, 1.5, size=n)
    for vv, WW in ((None, None), (v, W)):
        g = _whole(handle, ev, align, w, vv, WW, opt=kf.kf_default_options(block=0, h_max=h_max, n_iter=n_iter, **opt))
        fd = _fd2(oracle.objective_gradient_fd, ev=ev, align=align, weights=w, dl_dparams=vv, dl_dcov=WW)
        _, l_abs = oracle.objective_per_track(ev, align, weights=w, dl_dparams=vv, dl_dcov=WW)
        _check_grads(g["gs"], g["ga"], fd[0], fd[1], ev["seed_params"], l_abs, min_resolved=0.2)
