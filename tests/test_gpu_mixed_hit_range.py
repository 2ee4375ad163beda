"""The mixed path's update over the range of hit variances, against the oracle
with the mixed contract's tolerances: hits that carry no information (variances
of 1e13 to 1e38 mm^2 in one coordinate or in both, as a reconstruction program
marks a coordinate that was not measured), with ordinary and with large
residuals, correlated, and hits far more precise than the prediction."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_fp64_path import _event
from tests.test_gpu_mixed_path import SHAPES
from tests.test_gpu_parity import FP64, MIXED, compare, gpu_fit, handle  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coords", [(0,), (1,), (0, 1)], ids=["loc0", "loc1", "both"])
@pytest.mark.parametrize("var", [1e-13, 1e13, 1e20, 1e30, 1e38])
@pytest.mark.parametrize("shape", SHAPES, ids=["255", "168", "128"])
def test_hit_variances(handle, var, coords, shape):  # noqa: F811
    ev = _event(97)
    ev["cov"], ev["loc"] = ev["cov"].copy(), ev["loc"].copy()
    rho = 0.5 if len(coords) == 2 else 0.0
    for plane in (1, 4, 10):  # the first measurement, one in the middle, the last
        at = slice(plane, None, 11)
        for c in coords:
            ev["cov"][2 * c, at] = var
        ev["cov"][1, at] = rho * var
        if plane == 4 and var > 1.0:
            ev["loc"][coords[0], at] += 1e-3 * np.sqrt(var)
    r = oracle.fit_batch(ev)
    assert (r["status"] == 0).all()
    compare(gpu_fit(handle, ev, MIXED, **shape), r, MIXED)


@pytest.mark.parametrize("coords", [(0,), (1,), (0, 1)], ids=["loc0", "loc1", "both"])
@pytest.mark.parametrize("prec,opt", [(FP64, dict(team_warps=1)), (FP64, dict(team_warps=4)), (FP64, dict(energy_loss=1)),
                                      (MIXED, {})], ids=["one_thread", "team", "energy_loss", "mixed"])
def test_infinite_variance_is_refused(handle, prec, opt, coords):  # noqa: F811
    """An infinite variance fails its track, in either precision; the others fit."""
    ev = _event(64)
    ev["cov"] = ev["cov"].copy()
    for c in coords:
        ev["cov"][2 * c, 4::22] = np.inf  # every second track
    g = gpu_fit(handle, ev, prec, **opt)
    assert (g["status"][0::2] != 0).all() and (g["status"][1::2] == 0).all()
    assert np.isnan(g["params"][:, 0::2]).all() and np.isnan(g["chi2"][0::2]).all()
