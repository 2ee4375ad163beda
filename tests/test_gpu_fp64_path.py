"""The FP64 path's branches away from the telescope workloads, against the
oracle: long plane corrections and sub-steps in a strong field, start angles
outside their principal range, predicted covariances the float positivity
certificate does not settle, tracks of one and two states.  Tolerance: the
FP64 contract (1e-9 relative, metrics in tests/metrics.py)."""
import numpy as np
import pytest

import oracle
import paper_2105_01796_gb300 as kf
from paper_2105_01796_gb300 import synth
from tests.metrics import state_sigmas, states_err
from tests.test_gpu_parity import FP64, compare, gpu_fit, handle  # noqa: F401

pytestmark = pytest.mark.gpu

TEAMS = [0, 2, 4]


def _event(n=97):
    return dict(synth.make_event(synth.scaled(synth.WORKLOADS["tel10_1k"], n)))


@pytest.mark.parametrize("team", TEAMS)
@pytest.mark.parametrize("field", [(0.0, 0.0, 8.0), (1.0, -2.0, 7.5), (0.0, 0.0, 0.0)])
@pytest.mark.parametrize("h_max,n_iter", [(200.0, 3), (200.0, 1), (7.0, 2)])
def test_strong_field_and_substeps(handle, team, field, h_max, n_iter):  # noqa: F811
    # 8 T bends a 1 GeV track by 0.07 rad per gap: corrections of a
    # millimetre, far beyond the summed-correction range; only the first two
    # planes measure, so the later states are the propagated prediction
    ev = _event()
    ev["bfield"] = np.array(field)
    hole = ev["is_hole"].reshape(-1, 11).copy()
    hole[:, 3:] = 1
    ev["is_hole"] = hole.reshape(-1)
    opt = dict(h_max=h_max, n_iter=n_iter)
    g = gpu_fit(handle, ev, FP64, with_states=True, team_warps=team, **opt)
    r = oracle.fit_batch(ev, with_states=True, **opt)
    assert (r["status"] == 0).mean() > 0.5
    compare(g, r, FP64)
    ok = np.repeat(r["status"] == 0, 11)
    err = states_err(g["states"][:, ok], r["states"][:, ok], state_sigmas(ev, **opt)[:, ok])
    assert err.max() < 1e-9, err.max()


@pytest.mark.parametrize("team", TEAMS)
def test_start_angles_outside_the_principal_range(handle, team):  # noqa: F811
    ev = _event()
    s = ev["seed_params"].copy()
    s[2, 0::3] += 2 * np.pi
    s[3, 1::3] = -s[3, 1::3]
    s[2, 1::3] += np.pi
    s[3, 2::3] += 2 * np.pi
    ev["seed_params"] = s
    g = gpu_fit(handle, ev, FP64, with_states=True, team_warps=team)
    r = oracle.fit_batch(ev, with_states=True)
    assert (r["status"] == 0).all()
    compare(g, r, FP64)
    err = states_err(g["states"], r["states"], state_sigmas(ev))
    assert err.max() < 1e-9, err.max()


@pytest.mark.parametrize("team", TEAMS)
def test_positive_definiteness_verdict(handle, team):  # noqa: F811
    """Correlation of q/p and t (which no noise touches) of 1 - 1e-7: the
    certificate cannot decide and the FP64 pivots accept; of 1.5: not
    positive definite."""
    ev = _event(64)
    c = ev["seed_cov"].copy()
    i44, i55, i54 = 14, 20, 19
    rho = np.where(np.arange(64) % 2 == 0, 1.0 - 1e-7, 1.5)
    c[i54] = rho * np.sqrt(c[i44] * c[i55])
    ev["seed_cov"] = c
    g = gpu_fit(handle, ev, FP64, team_warps=team)
    r = oracle.fit_batch(ev)
    assert (r["status"][0::2] == oracle.OK).all() and (r["status"][1::2] == oracle.NON_SPD).all()
    compare(g, r, FP64)


@pytest.mark.parametrize("team", TEAMS)
@pytest.mark.parametrize("length", [1, 2, 3])
def test_short_tracks(handle, team, length):  # noqa: F811
    ev = _event(33)
    keep = (np.arange(33)[:, None] * 11 + np.arange(length)).ravel()
    ev["offsets"] = (np.arange(34) * length).astype(np.int32)
    for k in ("loc", "cov", "truth_states"):
        ev[k] = np.ascontiguousarray(ev[k][:, keep])
    for k in ("surface_id", "is_hole"):
        ev[k] = np.ascontiguousarray(ev[k][keep]).copy()
    ev["is_hole"][:] = 0  # the seed's own plane measures too
    g = gpu_fit(handle, ev, FP64, with_states=True, team_warps=team)
    r = oracle.fit_batch(ev, with_states=True)
    compare(g, r, FP64)
    err = states_err(g["states"], r["states"], state_sigmas(ev))
    assert err.max() < 1e-9, err.max()


@pytest.mark.parametrize("field", [(0.0, 0.0, 2.0), (0.3, -0.2, 2.0)])
@pytest.mark.parametrize("states", [False, True])
def test_library_shape_gives_the_same_bits(handle, field, states):  # noqa: F811
    """The default launch shape (teams of 4 or 2 warps for a part-filled last
    round of one warp per sub-partition) against one thread per track: small
    batches, and full rounds with a remainder of one unit, of under and over
    one team per SM, and of more than two."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rnd = 32 * 4 * sms
    sizes = [1, 97, 32 * sms, 32 * sms + 1, 64 * sms, 64 * sms + 1, rnd, rnd + 1, rnd + 33 * sms]
    ev = dict(synth.make_event(synth.scaled(synth.WORKLOADS["uneven30_1m"], max(sizes))))
    ev["bfield"] = np.array(field)
    for n in sizes:
        sub = dict(ev)
        m = int(ev["offsets"][n])
        sub["n_tracks"], sub["offsets"] = n, ev["offsets"][:n + 1]
        for k in ("seed_params", "seed_cov"):
            sub[k] = np.ascontiguousarray(ev[k][:, :n])
        for k in ("loc", "cov", "truth_states"):
            if k in ev:
                sub[k] = np.ascontiguousarray(ev[k][:, :m])
        for k in ("surface_id", "is_hole"):
            sub[k] = ev[k][:m]
        a = gpu_fit(handle, sub, FP64, with_states=states)
        b = gpu_fit(handle, sub, FP64, with_states=states, team_warps=1)
        for k in a:
            if a[k] is not None:
                assert np.array_equal(a[k], b[k], equal_nan=True), (n, k)


@pytest.mark.parametrize("team", TEAMS)
def test_time_carried_or_not(handle, team):  # noqa: F811
    """The fit leaves the time row out where the seed settles its pivot: seeds
    with correlated times, and with time errors so small (1e-6 ns) that the
    row is carried, give the oracle's results and the bits of the fit that
    keeps every state (which always carries it)."""
    ev = _event(97)
    c = ev["seed_cov"].copy()
    sd = np.sqrt(c[[0, 2, 5, 9, 14, 20]])
    sd[5, 0::3] = 1e-6
    for e, (i, j) in enumerate((i, j) for i in range(6) for j in range(i + 1)):
        rho = 1.0 if i == j else 0.3 if (i, j) in ((5, 0), (5, 3), (2, 0)) else 0.0
        c[e] = rho * sd[i] * sd[j]
    ev["seed_cov"] = c
    g = gpu_fit(handle, ev, FP64, team_warps=team)
    compare(g, oracle.fit_batch(ev), FP64)
    s = gpu_fit(handle, ev, FP64, with_states=True, team_warps=team)
    for k in ("params", "cov", "chi2", "status"):
        assert np.array_equal(g[k], s[k]), k
