"""The mixed path's double-float update and smoother at their edges, against
the oracle with the mixed contract's tolerances (1e-4 on parameters and chi2,
1e-3 on covariances): the FP64 update of a measured state 0, short tracks,
measurements with correlated and very unequal errors, a singular prediction."""
import numpy as np
import pytest

import oracle
import paper_2105_01796_gb300 as kf
from tests.test_gpu_fp64_path import _event
from tests.test_gpu_parity import MIXED, compare, gpu_fit, handle  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPES = [dict(), dict(block=128, min_blocks=3), dict(block=256, min_blocks=4)]


@pytest.mark.parametrize("shape", SHAPES, ids=["255", "168", "128"])
@pytest.mark.parametrize("length", [1, 2, 3, 11])
def test_measured_first_state_and_short_tracks(handle, length, shape):  # noqa: F811
    ev = _event(97)
    keep = (np.arange(97)[:, None] * 11 + np.arange(length)).ravel()
    ev["offsets"] = (np.arange(98) * length).astype(np.int32)
    for k in ("loc", "cov"):
        ev[k] = np.ascontiguousarray(ev[k][:, keep])
    for k in ("surface_id", "is_hole"):
        ev[k] = np.ascontiguousarray(ev[k][keep]).copy()
    ev["is_hole"][0::length] = 0
    ev["loc"][:, 0::length] += ev["seed_params"][:2]
    compare(gpu_fit(handle, ev, MIXED, **shape), oracle.fit_batch(ev), MIXED)


@pytest.mark.parametrize("field", [(0.0, 0.0, 2.0), (0.3, -0.6, 1.9)])
def test_unequal_correlated_hits(handle, field):  # noqa: F811
    ev = _event(333)
    ev["bfield"] = np.array(field)
    rng = np.random.default_rng(3)
    s = 0.05 * 10.0 ** rng.uniform(-0.7, 0.7, (2, ev["loc"].shape[1]))
    rho = rng.uniform(-0.95, 0.95, ev["loc"].shape[1])
    ev["cov"] = np.stack([s[0] ** 2, rho * s[0] * s[1], s[1] ** 2])
    compare(gpu_fit(handle, ev, MIXED), oracle.fit_batch(ev), MIXED)


def test_not_positive_definite(handle):  # noqa: F811
    ev = _event(64)
    c = ev["seed_cov"].copy()
    c[19] = np.where(np.arange(64) % 2, 1.5, 0.5) * np.sqrt(c[14] * c[20])  # (q/p, t)
    ev["seed_cov"] = c
    r = oracle.fit_batch(ev)
    assert (r["status"][1::2] == oracle.NON_SPD).all() and (r["status"][0::2] == oracle.OK).all()
    compare(gpu_fit(handle, ev, MIXED), r, MIXED)
