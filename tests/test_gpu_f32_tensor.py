"""The fp32 path of large dense problems, whose products run on the tensor cores as three bf16 parts per operand.

Shapes at the edges of its tiles (256 x 256 and 256 x 128 per CTA pair) and of its chunks of 64 reduction steps, ragged rows, few
classes and one sample beyond a tile, against the oracle with guard bands; its error against the CUDA cores' own; operands that
are not finite, which fall back to the CUDA cores for that call only.
"""
import numpy as np
import pytest
import torch

from oracle import sfb_oracle as orc
from sfbgen import make_inputs, scaled
from tests.test_gpu_parity import _workload, check_config
from tests.util import to_f64

pytestmark = pytest.mark.gpu

# J, D, P, B
MLR = [(1000, 2003, 8, 100), (257, 5121, 3, 171), (256, 4096, 4, 128), (385, 3333, 5, 103), (129, 8193, 1, 513), (100, 16841, 16, 42), (10, 9174, 10, 254),
       (3000, 641, 3, 333), (513, 191, 9, 229)]
DML = [(129, 8193, 1, 513), (600, 2001, 8, 64), (257, 1025, 3, 300), (40, 11625, 14, 85)]


@pytest.mark.parametrize("J,D,P,B", MLR)
def test_mlr(J, D, P, B):
    cfg = scaled("C1", J=J, D=D, P=P, B=B, pool=1)
    wl = _workload(cfg, make_inputs(cfg), "f32")
    try:
        assert wl.ctx.on_tensor_cores()
    finally:
        wl.close()
    check_config(cfg, "f32", eta=0.5, steps=2, guard=True)


@pytest.mark.parametrize("J,D,P,B", DML)
def test_dml(J, D, P, B):
    cfg = scaled("C2", J=J, D=D, P=P, B=B)
    check_config(cfg, "f32", eta=1e-3, steps=2, guard=True)
    inputs = make_inputs(cfg)
    full, comp = _workload(cfg, inputs, "f32"), _workload(dict(cfg, compact=1), inputs, "f32", guard=True)
    try:
        assert full.ctx.on_tensor_cores() and comp.ctx.on_tensor_cores()
        for t in range(2):
            full.step(t, eta=1e-3)
            comp.step(t, eta=1e-3)
        torch.cuda.synchronize()
        assert torch.equal(full.W, comp.W) and comp.guards_intact()      # the sums depend on the nonzero pairs alone
        _, U, _ = orc.unpack(full.sf_buf.cpu().numpy())
        assert full.ctx.active_pairs() == comp.ctx.active_pairs() == int(U.any(axis=1).sum()) < cfg["K"]
    finally:
        full.close()
        comp.close()


def test_error_is_below_that_of_fp32_multiply_adds():
    """u = L d of similar pairs, 300 x 8192: a chain of n fp32 multiply-adds rounds n times, about sqrt(n) 2^-25 of a sum of
    random signs (8192 / 9 ranges: 9e-7 at worst, 4e-7 measured on the CUDA cores); the chunk sums here are good to 2^-24."""
    cfg = scaled("C2", J=300, D=8192, P=4, B=96)
    inputs = make_inputs(cfg)
    inputs["similar"] = np.ones_like(inputs["similar"])
    wl = _workload(cfg, inputs, "f32")
    try:
        wl.compute_factors(0)
        assert wl.ctx.status() == 0
        d = to_f64(wl.V)[:, :8192]
        assert orc.rel_fro(to_f64(wl.U)[:, :300], d @ inputs["W"].astype(np.float64).T) <= 2.0 ** -22
    finally:
        wl.close()


@pytest.mark.parametrize("exponent", [-100, -113, -126, -140])
def test_small_operands_keep_all_their_bits(exponent):
    """W, then u, of about 2^exponent (fp32's own subnormals at -140) against samples of about 2^30: every operand's 24 bits count,
    so the errors are those of ordinary operands (the bound is the one above)."""
    cfg = scaled("C2", J=300, D=8192, P=4, B=96)
    inputs = make_inputs(cfg)
    inputs["similar"] = np.ones_like(inputs["similar"])
    rng = np.random.default_rng(5)
    wl = _workload(cfg, inputs, "f32")
    try:
        assert wl.ctx.on_tensor_cores()
        wl.batches[0]["X"].mul_(2.0 ** 30)
        wl.batches[0]["Xb"].mul_(2.0 ** 30)
        small = lambda *shape: torch.from_numpy(np.ldexp(rng.standard_normal(shape), exponent).astype(np.float32)).cuda()
        wl.W.copy_(small(300, 8192))
        wl.compute_factors(0)
        d, w = to_f64(wl.V)[:, :8192], to_f64(wl.W)
        assert orc.rel_fro(to_f64(wl.U)[:, :300], d @ w.T) <= 2.0 ** -22
        wl.U[:, :300] = small(384, 300)
        wl.pack(0)
        wl.W.zero_()
        wl.apply(-1.0)
        assert wl.ctx.status() == 0
        assert orc.rel_fro(to_f64(wl.W), to_f64(wl.U)[:, :300].T @ d) <= 2.0 ** -22
    finally:
        wl.close()


@pytest.mark.parametrize("where", ["w", "x", "big", "none"])
def test_operands_that_are_not_finite(where):
    """Operands that are not finite or so large that products overflow.  A weight of -inf that meets positive features only is a logit of -inf: class probability 0, everything else finite.  An
    infinite feature makes its sample's u NaN, and with it W; a finite weight whose product overflows is a logit of -inf too (its
    first two bf16 parts have different signs: their products would be -inf and +inf).  The next call, on finite values, is again that of a fresh context."""
    cfg = scaled("C1", J=257, D=2051, P=4, B=128, pool=1)
    inputs = make_inputs(cfg)
    wl, fresh = _workload(cfg, inputs, "f32", guard=True), _workload(cfg, inputs, "f32")
    try:
        assert fresh.ctx.on_tensor_cores()
        t = wl.batches[0]
        x = t["X"].clone()
        t["X"][:, 7] = t["X"][:, 7].abs() + 0.1
        W = wl.W.clone()
        if where == "w":
            wl.W[31, 7] = -float("inf")
        elif where == "big":
            t["X"][:, 7] = 2.0 ** 40
            wl.W[:, 7] = 0.0
            wl.W[31, 7] = -(2.0 ** 101) * (1 - 2.0 ** -12)
        elif where == "x":
            t["X"][100, 9] = float("inf")
        X64, W64 = to_f64(t["X"]), to_f64(wl.W)
        wl.step(0, eta=0.25)
        assert wl.ctx.status() == 0 and wl.guards_intact()
        h, U, V = orc.unpack(wl.sf_buf.cpu().numpy())
        with np.errstate(invalid="ignore"):
            U_or, _ = orc.mlr_factors(W64, X64, t["labels"].cpu().numpy())
            W_or = W64 - 0.25 * (U_or.T @ X64)
        assert np.array_equal(np.isnan(U), np.isnan(U_or))
        ok = np.isfinite(U_or)
        assert np.linalg.norm((U - U_or)[ok]) <= 1e-5 * np.linalg.norm(U_or[ok])
        got = to_f64(wl.W)
        ok = np.isfinite(W_or)
        assert np.array_equal(np.isfinite(got), ok) and (where == "x") == (not ok.any())
        if ok.any():
            assert np.linalg.norm(got[ok] - W_or[ok]) <= 1e-5 * np.linalg.norm(W_or[ok] - W64[ok]) + 2.0 ** -24 * np.linalg.norm(W64[ok])
        wl.W.copy_(W)
        t["X"].copy_(x)
        wl.step(0, eta=0.25)
        fresh.W.copy_(W)
        fresh.step(0, eta=0.25)
        assert wl.ctx.status() == 0
        assert torch.equal(wl.W, fresh.W) and torch.equal(wl.sf_buf, fresh.sf_buf)
    finally:
        wl.close()
        fresh.close()


@pytest.mark.parametrize("J,D,P,B", [(300, 8192, 4, 96), (600, 2001, 8, 64)])
def test_inactive_pairs_that_are_not_finite(J, D, P, B):
    """A dissimilar pair with a NaN or an infinite feature is beyond the margin (no comparison with NaN holds): its u is zero and
    the step leaves it out, with and without compaction.  W is that of the same pairs with finite features far apart."""
    cfg = scaled("C2", J=J, D=D, P=P, B=B)
    inputs = make_inputs(cfg)
    apart = np.nonzero(inputs["similar"] == 0)[0]
    full, comp, ref = _workload(cfg, inputs, "f32", guard=True), _workload(dict(cfg, compact=1), inputs, "f32"), _workload(cfg, inputs, "f32")
    try:
        for wl, values in ((full, ("nan", "inf", "-inf")), (comp, ("nan", "inf", "-inf")), (ref, (1e4, 1e4, -1e4))):
            for i, x in zip((apart[0], apart[7], apart[-1]), values):
                wl.batches[0]["X"][int(i), 5 + int(i) % 7] = float(x)
            wl.step(0, eta=1e-4)
            assert wl.ctx.status() == 0
        assert bool(torch.isfinite(full.W).all()) and torch.equal(full.W, comp.W) and full.guards_intact()
        assert full.ctx.active_pairs() == comp.ctx.active_pairs() == ref.ctx.active_pairs()
        dw, want = to_f64(full.W) - inputs["W"].astype(np.float64), to_f64(ref.W) - inputs["W"].astype(np.float64)
        # two roundings of the sums, and of W, per side
        assert np.linalg.norm(dw - want) <= 2e-6 * np.linalg.norm(want) + 2.0 ** -23 * np.linalg.norm(inputs["W"])
    finally:
        full.close()
        comp.close()
        ref.close()


@pytest.mark.parametrize("compact", [0, 1])
@pytest.mark.parametrize("n", [1, 5, 6])
def test_update_by_few_pairs(n, compact):
    """Fewer than six rows with nonzero u: the CUDA cores' multiply-adds, bit for bit those of a context (96 columns) that has only
    these; from six on the tensor cores.  A v that is not finite makes NaN where its u is zero, too, unless the pair is left out."""
    J, D, P, B = 300, 8192, 4, 96
    cfg = scaled("C2", J=J, D=D, P=P, B=B, compact=compact)
    small = scaled("C2", J=J, D=96, P=P, B=B, compact=compact)
    wide, narrow = _workload(cfg, make_inputs(cfg), "f32", guard=True), _workload(small, make_inputs(small), "f32")
    rng = np.random.default_rng(3)
    try:
        assert wide.ctx.on_tensor_cores() and not narrow.ctx.on_tensor_cores()
        wide.V.copy_(torch.from_numpy(rng.standard_normal((P * B, D)).astype(np.float32)))
        narrow.V.copy_(wide.V[:, :96])
        rows = torch.from_numpy(rng.permutation(P * B)[:n])
        for wl in (wide, narrow):
            wl.U.zero_()
            wl.W.zero_()
        wide.U[rows, :J] = torch.from_numpy(rng.standard_normal((n, J)).astype(np.float32)).cuda()
        narrow.U.copy_(wide.U)
        for wl in (wide, narrow):
            wl.pack(0)
            wl.apply(-1.0)
            assert wl.ctx.status() == 0
        assert torch.equal(wide.W[:, :96], narrow.W) == (n < 6)
        assert orc.rel_fro(to_f64(wide.W), to_f64(wide.U)[:, :J].T @ to_f64(wide.V)) <= 2.0 ** -24
        other = next(i for i in range(P * B) if i not in rows)
        wide.V[other, 70] = float("nan")
        W = wide.W.clone()
        wide.W.zero_()
        wide.pack(0)
        wide.apply(-1.0)
        assert wide.ctx.status() == 0 and wide.guards_intact()
        if compact:
            assert torch.equal(wide.W, W)
        else:
            assert bool(wide.W[:, 70].isnan().all()) and int(wide.W.isnan().sum()) == J
    finally:
        wide.close()
        narrow.close()


@pytest.mark.parametrize("where", ["u", "v", "v of a zero u"])
def test_separate_update_of_values_that_are_not_finite(where):
    """Separate calls: the update finds them itself, in listed rows and in a v whose u is zero (0 times infinity is a NaN of
    that column).  The next update, of finite rows, is that of a fresh context."""
    cfg = scaled("C1", J=257, D=2051, P=4, B=128, pool=1)
    inputs = make_inputs(cfg)
    wl, fresh = _workload(cfg, inputs, "f32", guard=True), _workload(cfg, inputs, "f32")
    try:
        assert wl.ctx.on_tensor_cores()
        for w in (wl, fresh):
            w.compute_factors(0)
            w.U[300] = 0.0
        U, V = wl.U.clone(), wl.V.clone()
        if where == "u":
            wl.U[17, 5] = float("inf")
        elif where == "v":
            wl.V[17, 9] = float("nan")
        else:
            wl.V[300, 9] = -float("inf")
        wl.pack(0)
        wl.apply(0.25)
        assert wl.ctx.status() == 0 and wl.guards_intact()
        with np.errstate(invalid="ignore"):
            u, v = to_f64(wl.U)[:, :257], to_f64(wl.V)[:, :2051]
            W_or = inputs["W"].astype(np.float64) - 0.25 * (u.T @ v)
        got, ok = to_f64(wl.W), np.isfinite(W_or)
        assert not ok.all() and np.array_equal(np.isnan(got), np.isnan(W_or)) and np.array_equal(np.isfinite(got), ok)
        # a chain of 512 multiply-adds rounds 512 times: sqrt(512) 2^-25 = 6.7e-7 of a change of random signs; then W's own rounding
        dw = np.linalg.norm(W_or[ok] - inputs["W"].astype(np.float64)[ok])
        assert np.linalg.norm(got[ok] - W_or[ok]) <= 2.0 ** -20 * dw + 2.0 ** -24 * np.linalg.norm(W_or[ok])
        wl.U.copy_(U)
        wl.V.copy_(V)
        wl.W.copy_(wl.W0)
        for w in (wl, fresh):
            w.pack(0)
            w.apply(0.25)
            assert w.ctx.status() == 0
        assert torch.equal(wl.W, fresh.W) and bool(torch.isfinite(wl.W).all())
    finally:
        wl.close()
        fresh.close()
