"""fp32 factors of so many samples that their tiles exceed the 65535 blocks of a launch grid's second dimension:
4 194 240 samples on 64-row tiles, 8 388 480 on 128-row tiles."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("J,D,K", [(3, 5, 4194241), (2, 4, 8388481), (5, 64, 4194305)])
def test_factors_of_very_many_samples(J, D, K):
    from paper_1511_08486_b200 import binding as B
    g = torch.Generator(device="cuda")
    g.manual_seed(K)
    W = torch.randn(J, D, device="cuda", generator=g)
    X = torch.randn(K, D, device="cuda", generator=g)
    labels = torch.randint(0, J, (K,), device="cuda", generator=g, dtype=torch.int32)
    ctx = B.Context(B.make_desc("mlr", "f32", J, D, 1, K))
    try:
        U = torch.full((K, ctx.ldu), 7.0, device="cuda")
        V = torch.full((K, ctx.ldv), 7.0, device="cuda")
        ctx.compute_factors(W, X, B.make_aux(labels=labels), U, V)
        assert ctx.status() == 0
        ref = torch.softmax(X.double() @ W.double().T, dim=1)
        ref[torch.arange(K, device="cuda"), labels.long()] -= 1.0
        # |z| below 60: sums of D products and the exponential, both to a few 2^-24 of |z|
        assert (U[:, :J].double() - ref).abs().max().item() <= 60 * (D + 4) * 2.0 ** -24
        assert torch.equal(V[:, :D], X) and not U[:, J:].any() and not V[:, D:].any()
    finally:
        ctx.destroy()
