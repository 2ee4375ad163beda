"""The gradient's device scratch is what its kernels use: 22 doubles per state
and track, 52 with the smoother's adjoint, beside the surface tables (2 MiB of
slack for them and for the allocator's granules)."""
import pytest

import paper_2105_01796_gb300 as kf
from paper_2105_01796_gb300 import synth
from tests.test_gpu_parity import handle  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("whole", [False, True])
def test_scratch_is_what_is_used(handle, whole):  # noqa: F811
    import torch
    n = 20_000
    ev = synth.make_event(synth.scaled(synth.WORKLOADS["tel10_1k"], n))
    dev = kf.event_to_device(ev)
    gs = torch.empty((6, n), dtype=torch.float64, device="cuda")
    v = torch.ones((6, n), dtype=torch.float64, device="cuda") if whole else None
    kf.kf_grad(handle, dev, dl_dparams=v, grad_seed=gs)  # module and local memory in place
    torch.cuda.synchronize()
    h = kf.Handle()
    before = torch.cuda.mem_get_info()[0]
    kf.kf_grad(h, dev, dl_dparams=v, grad_seed=gs)
    torch.cuda.synchronize()
    taken = before - torch.cuda.mem_get_info()[0]
    h.close()
    used = 8 * (52 if whole else 22) * 11 * n
    assert used <= taken + (2 << 20) and taken <= used + (4 << 20), (taken, used)
