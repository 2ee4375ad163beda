"""The library's own launch shape of the FP64 kernels for equally long tracks
(full waves, a last wave, teams) against the plain grid of 64-thread CTAs, at
batch sizes on both sides of the waves' edges: every track is fitted by the
same operations in the same order, so the outputs are equal bit for bit."""
import numpy as np
import pytest
import torch

import paper_2105_01796_gb300 as kf
from paper_2105_01796_gb300 import synth
from tests.test_gpu_parity import FP64, gpu_fit, handle  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [dict(), dict(energy_loss=1)])
@pytest.mark.parametrize("warps_per_sm,extra", [(0, 1), (1, -1), (2, 1), (4, 1), (5, 1), (7, 0), (8, 1), (10, 33),
                                                (20, 33)])
def test_waves_fit_every_track_alike(handle, variant, warps_per_sm, extra):  # noqa: F811
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 32 * sms * warps_per_sm + extra
    ev = dict(synth.make_event(synth.scaled(synth.WORKLOADS["tel10_1k"], 97)))
    rep = np.arange(n) % 97
    states = (rep[:, None] * 11 + np.arange(11)).reshape(-1)
    big = dict(ev, n_tracks=n, offsets=(np.arange(n + 1) * 11).astype(ev["offsets"].dtype))
    for k in ("seed_params", "seed_cov"):
        big[k] = np.ascontiguousarray(ev[k][:, rep])
    for k in ("loc", "cov"):
        big[k] = np.ascontiguousarray(ev[k][:, states])
    for k in ("surface_id", "is_hole"):
        big[k] = np.ascontiguousarray(ev[k][states])
    for k in ("truth_params", "truth_states"):
        big.pop(k)
    a = gpu_fit(handle, big, FP64, **variant)
    b = gpu_fit(handle, big, FP64, schedule=kf.KF_SCHEDULE_GRID, block=64, **variant)
    for k in ("params", "cov", "chi2", "ndf", "status"):
        assert np.array_equal(a[k], b[k], equal_nan=True), k
