"""Compaction at the edges of its waves of 256 pairs and 128-byte column slices: the oracle's bytes, W unchanged by it."""
import numpy as np
import pytest
import torch

from oracle import sfb_oracle as orc
from sfbgen import make_inputs, scaled
from tests.test_gpu_parity import _workload
from tests.util import MODEL_ID

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", ["f32", "tf32", "tf32x3"])
@pytest.mark.parametrize("J,D,P,B,similar", [
    (33, 36, 1, 1, 0.0), (32, 64, 2, 256, 0.3), (31, 100, 2, 257, 0.6), (65, 132, 1, 700, 0.1), (40, 96, 3, 255, 1.0),
])
def test_compacted_buffer_is_the_oracles(path, J, D, P, B, similar):
    cfg = scaled("C2", J=J, D=D, P=P, B=B)
    cfg["path"] = path
    cfg["w_std"] = 1.0                                  # dissimilar pairs lie beyond the margin: u = 0
    inputs = make_inputs(cfg)
    rng = np.random.default_rng(P * B)
    inputs["similar"] = (rng.random(P * B) < similar).astype(np.uint8)
    full, comp = _workload(cfg, inputs, path), _workload(dict(cfg, compact=1), inputs, path, guard=True)
    try:
        full.step(0, eta=0.0)
        comp.step(0, eta=0.0)
        torch.cuda.synchronize()
        _, U, V = orc.unpack(full.sf_buf.cpu().numpy())
        ref = orc.pack(MODEL_ID["dml"], orc.DTYPE_F32, J, D, P, B, U, V, clock=0, compact=True)
        assert np.array_equal(comp.sf_buf.cpu().numpy(), ref)
        assert comp.ctx.active_pairs() == int(np.any(U != 0, axis=1).sum()) == int(inputs["similar"].sum())
        staged = comp.sf_buf.clone()
        comp.compute_factors(0)
        comp.pack(0, clock=0)                           # flags found by a pass of their own
        torch.cuda.synchronize()
        assert torch.equal(comp.sf_buf, staged)
        assert full.ctx.status() == 0 and comp.ctx.status() == 0 and comp.guards_intact()
    finally:
        full.close()
        comp.close()
