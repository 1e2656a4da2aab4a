"""The single-launch step of small dense fp32 problems: the separate calls' W, SF buffer and dual variables, bit for bit.

Sizes go from one pair and one row of W to the largest the single launch takes (K J D = 65536, J = 128, D = 1024) and beyond.
"""
import numpy as np
import pytest
import torch

from sfbgen import make_inputs, scaled
from tests.test_gpu_parity import _workload, check_config

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1, 1), (10, 64, 4, 8), (3, 7, 2, 5), (5, 301, 3, 4), (128, 16, 4, 8), (127, 17, 3, 10), (128, 64, 2, 4),
          (16, 64, 8, 8), (16, 65, 8, 8), (4, 1023, 2, 8), (4, 1024, 2, 8), (33, 100, 1, 19)]


def _bits_agree(cfg, inputs, K=None, dual=False, bad_label=False):
    from paper_1511_08486_b200 import binding as B
    a, b = _workload(cfg, inputs, "f32", guard=True), _workload(cfg, inputs, "f32", guard=True)
    try:
        duals = []
        for w in (a, b):
            t = w.batches[0]
            if bad_label:
                t["labels"][0] = cfg["J"]
                t["labels"][-1] = -1
            d = torch.full((cfg["K"], (cfg["J"] + 3) // 4 * 4), 0.25, device="cuda") if dual else None
            duals.append(d)
            if dual:
                t["aux"] = B.make_aux(labels=t["labels"], dual=d, sdca_step=0.5)
        for t in range(2):
            n0 = a.ctx.launch_count()
            a.step(t, eta=0.3, K=K)
            n1 = a.ctx.launch_count()
            b.compute_factors(t)
            b.pack(t, clock=t)
            b.apply(0.3, K)
            torch.cuda.synchronize()
            assert (n1 - n0 == 1) == (cfg["K"] * cfg["J"] * cfg["D"] <= 65536)
            assert torch.equal(a.W, b.W) and torch.equal(a.sf_buf, b.sf_buf)
            if dual:
                assert torch.equal(duals[0], duals[1])
        want = B.SFB_DEV_BAD_LABEL if bad_label else 0
        assert a.ctx.status() == want and b.ctx.status() == want
        assert a.guards_intact() and b.guards_intact()
    finally:
        a.close()
        b.close()


@pytest.mark.parametrize("J,D,P,B", SHAPES)
def test_small_step_has_the_bits_of_the_separate_calls(J, D, P, B):
    for name in ("C0", "C2"):
        cfg = scaled(name, J=J, D=D, P=P, B=B)
        _bits_agree(cfg, make_inputs(cfg))


def test_small_step_options():
    cfg = scaled("C0", J=13, D=37, P=4, B=6)
    inputs = make_inputs(cfg)
    _bits_agree(cfg, inputs, K=12)            # the first two workers' pairs only
    _bits_agree(cfg, inputs, dual=True)
    _bits_agree(cfg, inputs, bad_label=True)
    _bits_agree(cfg, inputs, dual=True, bad_label=True)


def test_small_step_against_the_oracle():
    check_config(scaled("C0", J=100, D=64, P=2, B=5), "f32", eta=1.0, steps=3)
    check_config(scaled("C2", J=24, D=120, P=3, B=6), "f32", eta=1e-2, steps=3)


def test_a_bad_header_found_before_keeps_w_as_it_is():
    from paper_1511_08486_b200 import binding as B
    cfg = scaled("C0")
    w = _workload(cfg, make_inputs(cfg), "f32")
    try:
        w.step(0)
        w.sf_buf[0] = 0
        w.apply(0.1)                           # finds the bad header; the status bit stays until it is read
        before = w.W.clone()
        w.step(1)
        torch.cuda.synchronize()
        assert torch.equal(w.W, before)
        assert w.ctx.status() & B.SFB_DEV_BAD_HEADER
        w.step(2)
        torch.cuda.synchronize()
        assert not torch.equal(w.W, before) and w.ctx.status() == 0
        assert np.isfinite(w.W.cpu().numpy()).all()
    finally:
        w.close()
