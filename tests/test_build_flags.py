"""The warps of a track team never exchange the state: each computes it with
its own instance of the team code and must round alike and decide alike.  Every
source that holds that code is therefore compiled without contraction of
products and sums beyond the fused operations written in it; so are the
one-thread kernels that promise the same bits."""
import os
import re

from paper_2105_01796_gb300 import _build


def _includes(name, seen):
    if name in seen:
        return seen
    seen.add(name)
    with open(os.path.join(_build.CSRC, name)) as f:
        for inc in re.findall(r'#include "(kf_[^"]+)"', f.read()):
            _includes(inc, seen)
    return seen


def test_team_code_is_compiled_without_contraction():
    users = [s for s in _build.SOURCES if "kf_team.cuh" in _includes(s, set())]
    assert "kf_team.cu" in users and "kf_adjoint.cu" in users
    for src in users + ["kf_kernels.cu"]:
        assert "-fmad=false" in _build.FILE_FLAGS.get(src, []), src
