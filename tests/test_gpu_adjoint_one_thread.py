"""The adjoint's one-thread kernel (a block given, or team_warps = 1) against
the oracle's central differences on the stepping cases of
test_gpu_adjoint_steps, which the library gives to the team kernel when the
launch shape is left to it."""
import numpy as np
import pytest

import paper_2105_01796_gb300 as kf
from tests import test_gpu_adjoint_steps as steps
from tests.test_gpu_adjoint import handle  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [dict(block=64), dict(block=0, team_warps=1)], ids=["block64", "team1"])
@pytest.mark.parametrize("case", [c for c in steps.CASES if not c[4]], ids=lambda c: "%s-%s-%g-%d" % c[:4])
def test_stepping(handle, monkeypatch, case, shape):  # noqa: F811
    seen = []
    make = kf.kf_default_options

    def options(*a, **k):
        o = make(*a, **dict(k, **shape))
        seen.append((o.block, o.team_warps))
        return o

    monkeypatch.setattr(kf, "kf_default_options", options)
    steps.test_stepping(handle, monkeypatch, *case)
    assert seen and set(seen) == {(shape["block"], shape.get("team_warps", 0))}, np.unique(seen, axis=0)
