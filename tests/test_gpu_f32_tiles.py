"""fp32 GEMMs on 64 x 64 tiles at tile and range edges, against the oracle, with guard bands around every output.

One tile and many ranges, rows and columns one beyond a tile, feature counts that are no multiple of four (and of the
16 steps of a stage), samples that straddle workers, and the list of kept pairs of a compacted buffer.
"""
import pytest

from sfbgen import scaled
from tests.test_gpu_parity import check_config

pytestmark = pytest.mark.gpu

SHAPES = [(20, 9001, 2, 10), (64, 4096, 2, 32), (65, 1003, 5, 13), (10, 513, 4, 12), (129, 70, 3, 65), (300, 777, 7, 27),
          (500, 700, 4, 16), (33, 2050, 1, 200)]


@pytest.mark.parametrize("J,D,P,B", SHAPES)
def test_mlr(J, D, P, B):
    check_config(scaled("C1", J=J, D=D, P=P, B=B, pool=1), "f32", eta=0.5, steps=2, guard=True)


@pytest.mark.parametrize("compact", [0, 1])
@pytest.mark.parametrize("J,D,P,B", SHAPES[2:6])
def test_dml(J, D, P, B, compact):
    cfg = scaled("C2", J=J, D=D, P=P, B=B)
    if not compact:
        check_config(cfg, "f32", eta=1e-3, steps=2, guard=True)
        return
    import torch
    from sfbgen import make_inputs
    from tests.test_gpu_parity import _workload
    inputs = make_inputs(cfg)
    full, comp = _workload(cfg, inputs, "f32"), _workload(dict(cfg, compact=1), inputs, "f32", guard=True)
    try:
        for t in range(2):
            full.step(t, eta=1e-3)
            comp.step(t, eta=1e-3)
        torch.cuda.synchronize()
        assert torch.equal(full.W, comp.W) and comp.guards_intact()      # zero pairs left out: the same sums
        assert full.ctx.status() == 0 and comp.ctx.status() == 0
    finally:
        full.close()
        comp.close()
