"""A buffer whose header does not match the descriptor: nothing behind the header is read, W and the context stay sound."""
import pytest
import torch

from sfbgen import make_inputs, scaled
from tests.test_gpu_parity import _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", ["f32", "tf32", "tf32x3"])
def test_codes_of_a_refused_buffer_are_not_read(path):
    """Its codes hold atoms that do not exist (every read stays inside the buffer): reading them would set BAD_INDEX."""
    from paper_1511_08486_b200 import binding as B
    cfg = scaled("C3", J=36, D=100, P=3, B=7, density=0.2)
    cfg["path"] = path
    wl = _workload(cfg, make_inputs(cfg), path)
    try:
        wl.compute_factors(0)
        wl.pack(0)
        good = wl.sf_buf.clone()
        off, stride = B.sfb_sf_buffer_layout(wl.desc)
        pad = lambda n: (n + 127) // 128 * 128
        idx = off + pad(cfg["B"] * wl.ldu * 4) + pad((cfg["B"] + 1) * 4)
        cap = wl.desc.nnz_capacity // cfg["P"]
        for p in range(cfg["P"]):
            wl.sf_buf[idx + p * stride:idx + p * stride + cap * 4] = 0xFF
        wl.sf_buf[20] ^= 64                                  # J field of the header
        wl.apply(0.5)
        assert wl.ctx.status() == B.SFB_DEV_BAD_HEADER
        assert torch.equal(wl.W, wl.W0)
        # a right buffer afterwards is applied as if nothing had happened
        wl.sf_buf.copy_(good)
        wl.apply(1e-2)
        assert wl.ctx.status() == 0
        applied = wl.W.clone()
        wl.reset()
        wl.compute_factors(0)
        wl.pack(0)
        wl.apply(1e-2)
        assert torch.equal(applied, wl.W) and not torch.equal(applied, wl.W0)
    finally:
        wl.close()


@pytest.mark.parametrize("path,name,over", [
    ("bf16", "C4", dict(J=130, D=264, P=2, B=40, pool=1, labels="uniform")), ("tf32x3", "C1", dict(J=130, D=260, P=2, B=40)),
    ("tf32x3", "C2", dict(J=70, D=132, P=2, B=40)), ("tf32x3", "C3", dict(J=70, D=132, P=2, B=40, density=0.2))])
def test_a_refused_update_leaves_no_stale_copy_of_w(path, name, over):
    """The context has not seen W yet, or W has changed since: after a refused update its copy is rebuilt, not trusted."""
    from paper_1511_08486_b200 import binding as B
    cfg = scaled(name, **over)
    cfg["path"] = path
    inputs = make_inputs(cfg)
    a, b = _workload(cfg, inputs, path), _workload(cfg, inputs, path)
    try:
        for wl in (a, b):                       # b never sees the bad buffer
            wl.W.mul_(0.5)
        a.apply(0.5)                            # header of zeros
        assert a.ctx.status() == B.SFB_DEV_BAD_HEADER and torch.equal(a.W, b.W)
        for _ in range(2):
            a.step(0, eta=1e-3)
            b.step(0, eta=1e-3)
            assert a.ctx.status() == 0 and torch.equal(a.W, b.W) and torch.equal(a.sf_buf, b.sf_buf)
            a.sf_buf[20] ^= 64
            a.apply(0.5)
            assert a.ctx.status() == B.SFB_DEV_BAD_HEADER
            a.sf_buf[20] ^= 64
            for wl in (a, b):
                wl.W.mul_(0.9)
                wl.ctx.invalidate()
            a.sf_buf[20] ^= 64
            a.apply(0.5)
            assert a.ctx.status() == B.SFB_DEV_BAD_HEADER
    finally:
        a.close()
        b.close()


@pytest.mark.parametrize("name,over", [
    ("C1", dict(J=1000, D=2003, P=8, B=100, pool=1)), ("C2", dict(J=257, D=1025, P=3, B=300)), ("C2", dict(J=257, D=1025, P=3, B=300, compact=1))])
def test_large_fp32_update_of_a_refused_buffer(name, over):
    """Dense fp32 on the tensor cores.  The streams hold NaN (every read stays inside the buffer); afterwards the right buffer is
    applied, and a step taken, as by a context that never saw the refused one."""
    from paper_1511_08486_b200 import binding as B
    cfg = scaled(name, **over)
    inputs = make_inputs(cfg)
    wl, fresh = _workload(cfg, inputs, "f32", guard=True), _workload(cfg, inputs, "f32")
    try:
        for w in (wl, fresh):
            w.compute_factors(0)
            w.pack(0)
        good = wl.sf_buf.clone()
        off, _ = B.sfb_sf_buffer_layout(wl.desc)
        wl.sf_buf[20] ^= 64                                  # J field of the header
        wl.sf_buf[off:] = 0xFF
        bad = wl.sf_buf.clone()
        wl.apply(0.5)
        assert wl.ctx.status() == B.SFB_DEV_BAD_HEADER
        assert torch.equal(wl.W, wl.W0) and torch.equal(wl.sf_buf, bad)
        wl.sf_buf.copy_(good)
        for w in (wl, fresh):
            w.apply(1e-4)
            w.step(0, eta=1e-4)
            assert w.ctx.status() == 0
        assert torch.equal(wl.W, fresh.W) and torch.equal(wl.sf_buf, fresh.sf_buf)
        assert not torch.equal(wl.W, wl.W0) and wl.guards_intact()
    finally:
        wl.close()
        fresh.close()
