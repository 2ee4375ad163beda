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


@pytest.mark.parametrize("objective", ["chi2", "whole"])
def test_the_form_is_the_caller_s(handle, objective):  # noqa: F811
    """team_warps 1 and 2 each start the form they name: on a batch that leaves
    the GPU idle a team takes well under the time of one thread per track
    (device times, best of ten), also with a block given; 0 starts the team
    there, and one thread per track with a block given."""
    import torch
    ev = synth.make_event(synth.scaled(synth.WORKLOADS["align20_100k"], 320))
    dev = kf.event_to_device(ev)
    S = ev["center"].shape[1]
    v, W = _smoother_weights(ev) if objective == "whole" else (None, None)
    cu = lambda a: None if a is None else torch.from_numpy(a).cuda()  # noqa: E731
    v, W = cu(v), cu(W)
    gs = torch.empty((6, 320), dtype=torch.float64, device="cuda")
    ga = torch.empty((6, S), dtype=torch.float64, device="cuda")

    def best(**opt):
        o, t = kf.kf_default_options(**opt), []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            kf.kf_grad(handle, dev, dl_dparams=v, dl_dcov=W, grad_seed=gs, grad_align=ga, opt=o)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        return min(t[2:])

    one, team = best(block=0, team_warps=1), best(block=0, team_warps=2)
    assert team < 0.8 * one, (team, one)
    assert best(block=64, team_warps=2) < 0.8 * one
    assert best(block=0) < 0.8 * one < best(block=64)


def test_more_teams_than_sms(handle):  # noqa: F811
    import torch
    n = 32 * torch.cuda.get_device_properties(0).multi_processor_count + 33
    ev = synth.make_event(synth.scaled(synth.WORKLOADS["tel10_1k"], n))
    S = ev["center"].shape[1]
    v, W = np.full((6, n), 0.5), np.full((21, n), 2.0)
    one, team, auto = (_whole(handle, ev, np.zeros((6, S)), None, v, W,
                              opt=kf.kf_default_options(block=0, team_warps=t)) for t in (1, 2, 0))
    for k in VALUES + ("gs",):
        assert np.array_equal(one[k], team[k]) and np.array_equal(one[k], auto[k]), k
    assert np.allclose(team["ga"], one["ga"], rtol=1e-11, atol=1e-11 * np.abs(one["ga"]).max())


@pytest.mark.parametrize("prec", ["fp64", "mixed", "grad"])
def test_largest_surface_table(handle, prec):  # noqa: F811
    """1024 surfaces, of which the tracks cross the last ones: the staged tables
    at their largest, beside the teams' buffers."""
    ev = dict(synth.make_event(synth.scaled(synth.WORKLOADS["tel10_1k"], 65)))
    small = ev
    S = ev["center"].shape[1]
    pad = lambda a: np.concatenate([np.repeat(a[..., :1], 1024 - S, -1), a], -1)  # noqa: E731
    ev = dict(ev, center=pad(ev["center"]), rot=pad(ev["rot"]), x_over_x0=pad(ev["x_over_x0"]),
              surface_id=(ev["surface_id"] + (1024 - S)).astype(np.int32))
    if prec == "grad":
        v, W = np.full((6, 65), 0.5), np.full((21, 65), 2.0)
        a, b = (_whole(handle, e, np.zeros((6, e["center"].shape[1])), None, v, W,
                       opt=kf.kf_default_options(block=0, team_warps=t)) for e, t in ((small, 1), (ev, 2)))
        for k in VALUES + ("gs",):
            assert np.array_equal(a[k], b[k]), k
        assert np.allclose(b["ga"][:, -S:], a["ga"], rtol=1e-12, atol=1e-12 * np.abs(a["ga"]).max())
        assert not b["ga"][:, :-S].any()
        return
    from tests.test_gpu_parity import MIXED
    for team in (1, 2, 4) if prec == "fp64" else (0,):
        a, b = (gpu_fit(handle, e, FP64 if prec == "fp64" else MIXED, team_warps=team) for e in (small, ev))
        for k in VALUES:
            assert np.array_equal(a[k], b[k]), (team, k)
