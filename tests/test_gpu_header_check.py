"""Separate pack and apply on the compensated path, whose header check runs inside the pass over the factor rows: a buffer
with another header leaves W as it is (all bits), the right one is applied as sfb_step applies it; one launch (K <= 1024)
and several, J and D at the edges of the 64-value groups of that pass.
"""
import pytest
import torch

from sfbgen import make_inputs, scaled
from tests.test_gpu_parity import _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("J,D,P,B", [(3, 64, 1, 5), (64, 68, 2, 33), (65, 128, 3, 400), (130, 260, 17, 64)])
def test_header_is_checked_before_the_update(J, D, P, B):
    from paper_1511_08486_b200 import binding
    cfg = scaled("C1", J=J, D=D, P=P, B=B)
    wl = _workload(cfg, make_inputs(cfg), "tf32x3")
    try:
        wl.compute_factors(0)
        wl.pack(0)
        wl.sf_buf[20] ^= 64                                  # J field of the header
        wl.apply(0.5)
        assert wl.ctx.status() == binding.SFB_DEV_BAD_HEADER
        assert torch.equal(wl.W, wl.W0)
        wl.sf_buf[20] ^= 64
        wl.apply(0.5)
        assert wl.ctx.status() == 0
        applied = wl.W.clone()
        wl.W.copy_(wl.W0)
        wl.ctx.invalidate()
        wl.step(0, 0.5)
        assert torch.equal(applied, wl.W) and not torch.equal(applied, wl.W0)
    finally:
        wl.close()
