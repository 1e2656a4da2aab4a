"""DML factors without the factor v (V = None): the reduction is cut as it is with v, so u has the same bits."""
import pytest
import torch

from sfbgen import make_inputs, scaled
from tests.test_gpu_parity import _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("J,D,P,B", [(64, 4096, 2, 32), (65, 1003, 5, 13), (129, 2050, 3, 65), (20, 60, 2, 8), (600, 4000, 4, 128),
                                     (300, 500, 7, 100)])
def test_u_does_not_depend_on_whether_v_is_kept(J, D, P, B):
    cfg = scaled("C2", J=J, D=D, P=P, B=B)
    wl = _workload(cfg, make_inputs(cfg), "f32", guard=True)
    try:
        t = wl.batches[0]
        wl.compute_factors(0)
        with_v = wl.U.clone()
        wl.U.fill_(7.0)
        wl.ctx.compute_factors(wl.W, t["X"], t["aux"], wl.U, None)
        assert wl.ctx.status() == 0 and wl.guards_intact()
        assert torch.equal(wl.U, with_v)
    finally:
        wl.close()
