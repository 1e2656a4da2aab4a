"""Edge cases and the host-buffer entry point, through the C ABI on the GPU."""
import numpy as np
import pytest
import torch

from oracle import sfb_oracle as orc
from sfbgen import get_config, make_inputs, scaled
from tests.test_gpu_parity import _workload, check_config
from tests.util import to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,path,over", [
    ("C0", "f32", {}),
    ("C2", "f32", dict(J=40, D=300, P=2, B=6)),
    ("C3", "f32", dict(J=64, D=400, P=2, B=4, density=0.1)),
    ("C4", "bf16", dict(J=256, D=512, P=2, B=64, pool=1, labels="uniform")),
])
def test_step_host_equals_step(name, path, over):
    """sfb_step_host (minibatch in pinned host memory) leaves exactly the W and SF buffer of sfb_step."""
    from paper_1511_08486_b200 import binding as B
    cfg = scaled(name, **over) if over else get_config(name)
    cfg["path"] = path
    inputs = make_inputs(cfg)
    wl = _workload(cfg, inputs, path)
    try:
        wl.step(0, eta=0.05)
        torch.cuda.synchronize()
        W_ref, buf_ref = wl.W.clone(), wl.sf_buf.clone()
        wl.reset()
        wl.sf_buf.zero_()
        t = wl.batches[0]
        host = {k: v.cpu().pin_memory() for k, v in t.items() if isinstance(v, torch.Tensor)}
        aux = B.make_aux(**{k: v for k, v in host.items() if k != "X"})
        header = torch.zeros(128, dtype=torch.uint8).pin_memory()
        wl.ctx.step_host(wl.W, host.get("X"), aux, wl.sf_buf, 0.05, clock=0, header_host=header)
        assert wl.ctx.status() == 0                      # synchronises
        assert torch.equal(wl.W, W_ref) and torch.equal(wl.sf_buf, buf_ref)
        h = orc.parse_header(header.numpy())
        assert h["magic"] == orc.MAGIC and h["J"] == cfg["J"] and h["P"] == cfg["P"]
    finally:
        wl.close()


def test_single_worker_single_sample_and_single_class():
    check_config(scaled("C0", J=10, D=64, P=1, B=1), "f32", eta=1.0, steps=1)
    # J = 1: softmax is identically 1, so u = 1 - 1 = 0 and W must not move
    cfg = scaled("C0", J=1, D=16, P=2, B=3)
    inputs = make_inputs(cfg)
    wl = _workload(cfg, inputs, "f32")
    try:
        wl.step(0, eta=1.0)
        torch.cuda.synchronize()
        assert torch.equal(wl.W, wl.W0)
        _, U, _ = orc.unpack(wl.sf_buf.cpu().numpy())
        assert not U.any()
    finally:
        wl.close()


def test_dml_all_pairs_beyond_the_margin_leaves_dissimilar_rows_zero():
    cfg = scaled("C2", J=24, D=200, P=2, B=4)
    cfg["w_std"] = 1.0                                    # |L d|^2 >> margin: every dissimilar pair inactive
    inputs = make_inputs(cfg)
    wl = _workload(cfg, inputs, "f32")
    try:
        wl.compute_factors(0)
        torch.cuda.synchronize()
        U = to_f64(wl.U)
        sim = inputs["similar"].astype(bool)
        assert not U[~sim].any() and U[sim].any()
    finally:
        wl.close()


def test_sparse_codes_with_empty_rows_and_an_empty_worker():
    cfg = scaled("C3", J=48, D=300, P=3, B=4, density=0.1)
    inputs = make_inputs(cfg)
    rp, ix, vl = inputs["rowptr"][0].astype(np.int64), inputs["idx"][0], inputs["val"][0]
    # empty the codes of sample 1 and of every sample of worker 2 (samples 8..11)
    keep = np.ones(ix.size, bool)
    for i in [1] + list(range(8, 12)):
        keep[rp[i]:rp[i + 1]] = False
    counts = np.diff(rp)
    counts[[1, 8, 9, 10, 11]] = 0
    inputs["rowptr"][0] = np.concatenate([[0], np.cumsum(counts)]).astype(np.uint32)
    inputs["idx"][0], inputs["val"][0] = ix[keep], vl[keep]
    wl = _workload(cfg, inputs, "f32")
    try:
        wl.step(0, eta=0.05)
        torch.cuda.synchronize()
        W_or, U_or, _ = orc.step(orc.MODEL_SC, inputs["W"], dict(rowptr=inputs["rowptr"][0], idx=inputs["idx"][0],
                                                                  val=inputs["val"][0], Xdata=inputs["Xdata"][0]), 0.05)
        W0 = inputs["W"].astype(np.float64)
        err = np.linalg.norm((to_f64(wl.W) - W0) - (W_or - W0)) / np.linalg.norm(W_or - W0)
        assert err <= 1e-5 + 2.0 ** -24 * np.linalg.norm(W0) / np.linalg.norm(W_or - W0)
        h, U, (rp2, ix2, vl2) = orc.unpack(wl.sf_buf.cpu().numpy())
        assert np.array_equal(rp2, inputs["rowptr"][0]) and np.array_equal(ix2, inputs["idx"][0])
        assert np.allclose(U[1], -inputs["Xdata"][0][1], atol=0)       # empty code: u = -x exactly
        assert wl.ctx.status() == 0
    finally:
        wl.close()


def test_sparse_capacity_overflow_sets_status():
    from paper_1511_08486_b200 import binding as B
    cfg = scaled("C3", J=32, D=200, P=2, B=4, density=0.2)
    inputs = make_inputs(cfg)
    inputs["nnz_capacity"] = 2 * 32                         # far below the real nonzero count per worker
    wl = _workload(cfg, inputs, "f32")
    try:
        wl.compute_factors(0)
        wl.pack(0)
        assert wl.ctx.status() & B.SFB_DEV_CAPACITY
    finally:
        wl.close()


@pytest.mark.parametrize("path,over", [
    ("f32", dict(J=300, D=512, P=2, B=64)),
    ("tf32", dict(J=1000, D=1024, P=4, B=128)),
    ("bf16", dict(J=1000, D=1024, P=4, B=128)),
])
def test_saturated_softmax(path, over):
    """Logits of magnitude ~30 (W ~ N(0, 1)): most exponentials underflow, the partial maxima of the fused
    epilogue differ by tens of units between tiles, and u is close to +-1 on one or two classes per sample."""
    name = "C4" if path == "bf16" else "C1"
    cfg = scaled(name, pool=1, **over)
    cfg["path"] = path
    cfg["w_std"] = 1.0
    if name == "C4":
        cfg["labels"] = "uniform"
    inputs = make_inputs(cfg)
    wl = _workload(cfg, inputs, path)
    try:
        wl.compute_factors(0)
        torch.cuda.synchronize()
        assert wl.ctx.status() == 0
        U = to_f64(wl.U)[:, :cfg["J"]]
        # the oracle gets the operands as the tensor cores see them (tf32: low 13 mantissa bits dropped; bf16:
        # W rounded to nearest even, X is bf16 already), so that what is compared is the kernel's arithmetic and
        # not the sensitivity of a saturated softmax to operand rounding
        W_used, X_used = inputs["W"], inputs["X"][0]
        if path == "tf32":
            trunc = lambda a: (np.ascontiguousarray(a).view(np.uint32) & np.uint32(0xFFFFE000)).view(np.float32)
            W_used, X_used = trunc(W_used), trunc(X_used)
        elif path == "bf16":
            from sfbgen import bf16_bits_to_f32, bf16_round_bits
            W_used, X_used = bf16_bits_to_f32(bf16_round_bits(W_used)), bf16_bits_to_f32(inputs["X_bits"][0])
        U_or, _ = orc.mlr_factors(W_used, X_used, inputs["labels"][0])
        assert np.isfinite(U).all()
        assert np.abs(U.sum(axis=1)).max() <= (1e-4 if path == "f32" else 2e-2)       # rows of u still sum to zero
        from tests.util import TOL
        assert orc.rel_fro(U, U_or) <= TOL[path]
    finally:
        wl.close()


def test_dml_step_leaves_out_inactive_pairs_bit_identically():
    """The fp32 DML step applies only the pairs with u != 0 (an ordered list built on the device from the finishing pass's
    flags); the result must equal, bit for bit, that of the staged calls, which find these pairs in the buffer's rows, and
    both the sum over all K pairs."""
    cfg = scaled("C2", J=300, D=8192, P=4, B=96)
    inputs = make_inputs(cfg)
    wl = _workload(cfg, inputs, "f32")
    try:
        wl.step(0, eta=1e-4)
        torch.cuda.synchronize()
        W_step, buf_step = wl.W.clone(), wl.sf_buf.clone()
        _, U, _ = orc.unpack(buf_step.cpu().numpy())
        inactive = int((~U.any(axis=1)).sum())
        assert 0 < inactive < cfg["K"]                        # the case really has pairs beyond the margin
        assert wl.ctx.active_pairs() == cfg["K"] - inactive   # what the step's apply multiplied through
        wl.reset()
        wl.sf_buf.zero_()
        wl.compute_factors(0)
        wl.pack(0, clock=0)
        wl.apply(1e-4)
        assert wl.ctx.status() == 0
        assert torch.equal(wl.sf_buf, buf_step) and torch.equal(wl.W, W_step)
        U, V = (x.astype(np.float64) for x in orc.unpack(buf_step.cpu().numpy())[1:])
        dW, dW_or = to_f64(W_step) - inputs["W"].astype(np.float64), -1e-4 * (U.T @ V)
        assert np.linalg.norm(dW - dW_or) <= 1e-6 * np.linalg.norm(dW_or) + 2.0 ** -24 * np.linalg.norm(inputs["W"])
        # partial apply inside the step: only the first two workers' streams
        wl.reset()
        wl.step(0, eta=1e-4, K=2 * cfg["B"])
        torch.cuda.synchronize()
        W_part = wl.W.clone()
        wl.reset()
        wl.compute_factors(0)
        wl.pack(0, clock=0)
        wl.apply(1e-4, K=2 * cfg["B"])
        torch.cuda.synchronize()
        assert torch.equal(wl.W, W_part)
    finally:
        wl.close()


def test_bf16_two_classes_step_size_and_the_rounding_contract():
    """MLR with J = 2, D = 760, K = 260 on the bf16 path, the one shape a randomised sweep found above 1e-2
    (1.1e-2 after two steps with eta = 0.3, i.e. eta * |x|^2 = 228: the first step throws the logits of the
    second to +-300).  The cause is the path's contract, not its kernels: W enters the forward pass rounded to
    bf16 and u goes on the wire in bf16, and a softmax at |z| ~ 300 amplifies those roundings.  Checked both ways:
    (a) with a step ten times smaller the same shape is inside the stated tolerance against the plain oracle;
    (b) at eta = 0.3 the GPU agrees to 1e-3 with the oracle run on operands rounded the way the contract says
        (bf16 W for the forward, bf16 u for the update, fp32 storage of W between steps)."""
    from sfbgen import bf16_bits_to_f32, bf16_round_bits
    cfg = scaled("C4", J=2, D=760, P=2, B=130, pool=1, labels="uniform")
    cfg["path"] = "bf16"
    check_config(cfg, "bf16", eta=0.03, steps=2)
    inputs = make_inputs(cfg)
    X, y = bf16_bits_to_f32(inputs["X_bits"][0]), inputs["labels"][0]
    rb = lambda a: bf16_bits_to_f32(bf16_round_bits(np.ascontiguousarray(a, dtype=np.float32)))
    eta = 0.3
    W = inputs["W"].astype(np.float32)
    for _ in range(2):
        U, V = orc.mlr_factors(rb(W), X, y)
        W = orc.apply_dense(W, rb(U.astype(np.float32)), V, eta).astype(np.float32)
    wl = _workload(cfg, inputs, "bf16")
    try:
        for t in range(2):
            wl.step(t, eta=eta)
        torch.cuda.synchronize()
        assert wl.ctx.status() == 0
        W0 = inputs["W"].astype(np.float64)
        got, want = to_f64(wl.W) - W0, W.astype(np.float64) - W0
        err = np.linalg.norm(got - want) / np.linalg.norm(want)
        assert err <= 1e-3, f"{err:.3e} against the oracle on contract-rounded operands"
    finally:
        wl.close()
