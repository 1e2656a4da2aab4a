"""Column projection of sparse coding (sfb_prox) at the edges of its slabs and CTA shares, and what it leaves cached.

A slab is 32 columns wide; a CTA holds 512 rows of it, a cluster up to 8 CTAs; longer columns are read twice.
"""
import numpy as np
import pytest
import torch

from oracle import sfb_oracle as orc
from sfbgen import make_inputs, scaled
from tests.test_gpu_parity import _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("J,D", [(1, 4), (31, 33), (32, 32), (65, 1), (512, 100), (513, 35), (4096, 64), (4097, 31), (9000, 40)])
def test_prox_matches_the_oracle(J, D):
    from paper_1511_08486_b200 import binding as B
    rng = np.random.default_rng(J + D)
    W = rng.standard_normal((J, D)) / np.sqrt(J)
    W = (W * rng.choice([0.4, 2.5], D)[None, :]).astype(np.float32)
    if J == 1:
        W = np.where(np.abs(W) < 0.5, 0.25, 3.0).astype(np.float32)
    ctx = B.Context(B.make_desc("sc", "f32", J, D, 1, 1, v_sparse=1, nnz_capacity=32))
    try:
        raw = torch.full((J * D + 256,), 7.0, device="cuda")       # guard bands: a stray store shows there
        got = raw[128:128 + J * D].view(J, D)
        got.copy_(torch.from_numpy(W))
        ctx.prox(got)
        assert ctx.status() == 0
        assert (raw[:128] == 7.0).all() and (raw[128 + J * D:] == 7.0).all()
        out = got.cpu().numpy()
        inside = np.linalg.norm(W.astype(np.float64), axis=0) <= 1.0
        assert np.array_equal(out[:, inside], W[:, inside])
        # a sum of J squares in fp32 and two more roundings: relative error below (J / 32 + 64) 2^-24 by far
        assert orc.rel_fro(out, orc.prox_unit_columns(W)) <= 2e-6
    finally:
        ctx.destroy()


@pytest.mark.parametrize("J,D", [(70, 332), (600, 1000)])
def test_prox_keeps_the_compensated_operand_of_w_in_step(J, D):
    """The projection rewrites the cached correction operand with W: the next step gives the bits of a step that
    rebuilds the operand from scratch."""
    cfg = scaled("C3", J=J, D=D, P=3, B=20, density=0.1)
    cfg["path"] = "tf32x3"
    inputs = make_inputs(cfg)
    a, b = _workload(cfg, inputs, "tf32x3"), _workload(cfg, inputs, "tf32x3")
    try:
        for t in range(3):
            a.step(t, eta=0.05)
            a.ctx.prox(a.W)
            b.step(t, eta=0.05)
            b.ctx.prox(b.W)
            b.ctx.invalidate()
            torch.cuda.synchronize()
            assert torch.equal(a.W, b.W) and torch.equal(a.sf_buf, b.sf_buf)
        assert (a.W.double().norm(dim=0) <= 1.0 + 1e-5).all()
    finally:
        a.close()
        b.close()
