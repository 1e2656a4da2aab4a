"""The work a program has this library do, as timed cases over the range of shapes it is used at.

A case is one iteration of a training loop on one minibatch, through the public entry points of
`paper_1511_08486_b200.binding.Context`: `sfb_step` (factors, commit to the SF buffer, rank-K apply), the same as the
three separate calls a sender and a receiver make (`sfb_compute_factors`, `sfb_pack`, `sfb_apply`), the sparse-coding
step with its proximal operator, SDCA factors, and compacted buffers, on all four arithmetic paths.

Fields of a case: model, path, J x D (size of W), P workers of B samples each, call ("step" | "separate"), eta, and
per model  mlr: normalise (unit-norm features, else N(0,1)), zipf (label distribution), dual (SDCA factors);
dml: compact (pairs with u = 0 leave the buffer);  sc: density of the codes, prox (column projection after the step).
"""
import math

import torch

from paper_1511_08486_b200 import binding as B

W_STD = 0.01          # MLR: W ~ N(0, 0.01)
SDCA_LAMBDA, SDCA_STEP = 1.0, 0.2
CODE_NOISE = 0.01     # sparse coding: x = W_true a + N(0, 0.01)


def _mlr(path, J, D, P, batch, eta, normalise, zipf=False, dual=False, call="step"):
    return dict(model="mlr", path=path, J=J, D=D, P=P, B=batch, call=call, eta=eta, normalise=normalise, zipf=zipf,
                dual=dual)


def _dml(path, J, D, P, batch, compact=False, call="step"):
    return dict(model="dml", path=path, J=J, D=D, P=P, B=batch, call=call, eta=1e-2 / D, compact=compact)


def _sc(path, J, D, P, batch, density, prox, call="step"):
    return dict(model="sc", path=path, J=J, D=D, P=P, B=batch, call=call, eta=1e-4, density=density, prox=prox)


def listed():
    return [
        # the smallest problem: a few classes over a few dozen features, where launches and host time are everything
        dict(_mlr("f32", 10, 64, 4, 8, 1e-2, False), name="mlr_tiny_f32"),
        # a small ragged problem (no dimension a multiple of a tile, short worker streams) on the dual side: SDCA
        dict(_mlr("tf32", 257, 1000, 2, 100, 1.0 / (SDCA_LAMBDA * 200), True, dual=True), name="mlr_small_sdca_tf32"),
        # the large multiclass problem of the benchmark on each of the paths that take fp32 samples
        dict(_mlr("f32", 1000, 20000, 8, 128, 1e-2, True), name="mlr_large_f32"),
        dict(_mlr("tf32", 1000, 20000, 8, 128, 1e-2, True), name="mlr_large_tf32"),
        dict(_mlr("tf32x3", 1000, 20000, 8, 128, 1e-2, True), name="mlr_large_tf32x3"),
        # distance metric learning: the reference arithmetic, and the reduced one with inactive pairs left out
        dict(_dml("f32", 600, 10000, 8, 256), name="dml_f32"),
        dict(_dml("tf32", 600, 10000, 8, 256, compact=True), name="dml_compact_tf32"),
        # a mid-sized metric whose factors travel: computed, packed and applied by separate calls
        dict(_dml("tf32x3", 600, 2000, 8, 32, call="separate"), name="dml_mid_separate_tf32x3"),
        # dictionary update of sparse coding, with the projection that ends every iteration: sparse and dense routes
        dict(_sc("f32", 4096, 10000, 16, 64, 0.05, True), name="sc_prox_f32"),
        dict(_sc("tf32x3", 4096, 10000, 16, 64, 0.05, True), name="sc_prox_tf32x3"),
        # bf16 samples: a mid-sized ragged problem with the paper's 100 samples per worker, and the largest one
        dict(_mlr("bf16", 4000, 2056, 10, 100, 1e-5, False, zipf=True), name="mlr_mid_bf16"),
        dict(_mlr("bf16", 32768, 8192, 16, 256, 1e-5, False, zipf=True), name="mlr_scale_bf16"),
    ]


# Most multiply-adds (J * D * K) of a drawn case per path, and the cap on K: what the listed cases of the path hold.
_MOST = {"f32": 2.1e10, "tf32": 4.2e10, "tf32x3": 4.2e10, "bf16": 1.1e12}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    model, path = rng.choice([("mlr", "f32"), ("mlr", "tf32"), ("mlr", "tf32x3"), ("mlr", "bf16"), ("mlr", "bf16"),
                              ("dml", "f32"), ("dml", "tf32"), ("dml", "tf32x3"), ("sc", "f32"), ("sc", "tf32"),
                              ("sc", "tf32x3")])
    while True:
        big = path == "bf16"
        J = _log(rng, 64, 4096) if model == "sc" else _log(rng, 32, 800) if model == "dml" else _log(
            rng, 10, 32768 if big else 4000)
        D = _log(rng, 256, 10000) if model == "sc" else _log(rng, 64, 20000)
        P, batch = rng.randint(1, 16), _log(rng, 5, 256)
        # rows of samples are whole 16-byte units on the tensor-core paths; any length on the fp32 path
        unit = {"f32": 1, "tf32": 4, "tf32x3": 4, "bf16": 8}[path]
        D = max(unit, D // unit * unit)
        if J * D * P * batch <= _MOST[path] and J * D <= 2.7e8:
            break
    call = "separate" if rng.random() < 0.2 else "step"
    if model == "dml":
        return _dml(path, J, D, P, batch, compact=rng.random() < 0.4, call=call)
    if model == "sc":
        return _sc(path, J, D, P, batch, rng.choice([0.01, 0.02, 0.05]), rng.random() < 0.5, call=call)
    if big:
        return _mlr(path, J, D, P, batch, 1e-5, False, zipf=rng.random() < 0.5, call=call)
    if rng.random() < 0.25:
        return _mlr(path, J, D, P, batch, 1.0 / (SDCA_LAMBDA * P * batch), True, dual=True, call=call)
    return _mlr(path, J, D, P, batch, 1e-2, True, call=call)


# ------------------------------------------------------------------------------------------ what the program has in hand
def _unit_columns(m):
    return m / m.norm(dim=0, keepdim=True)


def _nnz_capacity(case):
    """CSR room per worker: the expected count of nonzeros plus eight standard deviations, whole 32-entry units."""
    n = case["B"] * case["D"]
    room = n * case["density"] + 8.0 * math.sqrt(n * case["density"]) + 32
    return int(min(n, room) + 31) // 32 * 32 * case["P"]


def prepare(case, seed):
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    model, J, D, P, batch = case["model"], case["J"], case["D"], case["P"], case["B"]
    K = P * batch
    s = dict(case=case, K=K, clock=0)

    def normal(*shape):
        return torch.randn(*shape, device=dev, generator=g)

    nnz_capacity = 0
    if model == "mlr":
        W = normal(J, D).mul_(W_STD)
        X = normal(K, D)
        if case["normalise"]:
            X /= X.norm(dim=1, keepdim=True)
        if case["zipf"]:
            p = torch.arange(1, J + 1, device=dev, dtype=torch.float32).pow(-1.1)
            labels = torch.multinomial(p, K, replacement=True, generator=g).int()
        else:
            labels = torch.randint(0, J, (K,), device=dev, generator=g, dtype=torch.int32)
        s["X"] = X.bfloat16() if case["path"] == "bf16" else X
        s["side"] = dict(labels=labels)
        if case["dual"]:
            s["dual"] = torch.zeros(K, (J + 3) // 4 * 4, device=dev)
            s["side"].update(dual=s["dual"], sdca_step=SDCA_STEP)
    elif model == "dml":
        # E |L d|^2 is 1, the margin, for a pair of independent points.  Similar pairs lie close together; of the
        # dissimilar ones every other is a hard one (well inside the margin), the rest are far apart.
        W = normal(J, D).mul_(1.0 / math.sqrt(2.0 * J * D))
        i = torch.arange(K, device=dev)
        apart = torch.tensor([0.5, 0.4, 0.5, 2.5], device=dev)[i % 4] * math.sqrt(2.0)
        s["X"] = normal(K, D)
        Xb = normal(K, D).mul_(apart[:, None]).add_(s["X"])
        s["side"] = dict(Xb=Xb, similar=(i % 2 == 0).to(torch.uint8))
    else:
        true = _unit_columns(normal(J, D))
        W = _unit_columns(true + 0.5 * _unit_columns(normal(J, D)))
        u = torch.rand(K, D, device=dev, generator=g) - 0.5
        codes = -torch.sign(u) * torch.log1p(-2.0 * u.abs().clamp_(max=0.4999999))      # Laplace(0, 1)
        codes *= torch.rand(K, D, device=dev, generator=g) < case["density"]
        data = codes @ true.T + CODE_NOISE * normal(K, J)
        at = codes.nonzero()
        counts = torch.bincount(at[:, 0], minlength=K)
        nnz_capacity = _nnz_capacity(case)
        s["X"] = None
        s["side"] = dict(rowptr=torch.nn.functional.pad(counts.cumsum(0), (1, 0)).int(), idx=at[:, 1].int().contiguous(),
                         val=codes[at[:, 0], at[:, 1]].contiguous(), Xdata=data)
    s["W"] = W
    s["aux"] = B.make_aux(**s["side"])
    desc = B.make_desc(model, case["path"], J, D, P, batch, v_sparse=model == "sc", margin=1.0, nnz_capacity=nnz_capacity,
                       compact=int(case.get("compact", False)))
    ctx = s["ctx"] = B.Context(desc)
    buf = s["buf"] = torch.zeros(ctx.sf_buffer_bytes, dtype=torch.uint8, device=dev)
    if case["call"] == "separate":
        dtype = torch.bfloat16 if case["path"] == "bf16" else torch.float32
        s["U"] = torch.zeros(K, ctx.ldu, dtype=dtype, device=dev)
        s["V"] = None if model == "sc" else torch.zeros(K, ctx.ldv, dtype=dtype, device=dev)
    s["out"] = _outputs(s, desc, buf)
    return s


def _outputs(s, desc, buf):
    """W and everything in the SF buffer, as views: header and directory, the u rows, the v rows or the CSR codes."""
    case, ctx = s["case"], s["ctx"]
    P, batch = case["P"], case["B"]
    dtype, es = (torch.bfloat16, 2) if case["path"] == "bf16" else (torch.float32, 4)
    off, stride = B.sfb_sf_buffer_layout(desc)
    pad = lambda n: (n + 127) // 128 * 128
    v_off = off + pad(batch * ctx.ldu * es)
    vals, words = buf.view(dtype), buf.view(torch.int32)
    out = dict(W=s["W"], head=buf[:off],
               U=vals.as_strided((P, batch, ctx.ldu), (stride // es, ctx.ldu, 1), off // es))
    if case["model"] == "sc":
        cap = desc.nnz_capacity // P
        idx_off = v_off + pad((batch + 1) * 4)
        out["rowptr"] = words.as_strided((P, batch + 1), (stride // 4, 1), v_off // 4)
        out["idx"] = words.as_strided((P, cap), (stride // 4, 1), idx_off // 4)
        out["val"] = vals.as_strided((P, cap), (stride // 4, 1), (idx_off + pad(cap * 4)) // 4)
    else:
        out["V"] = vals.as_strided((P, batch, ctx.ldv), (stride // es, ctx.ldv, 1), v_off // es)
    if "dual" in s:
        out["dual"] = s["dual"]
    return out


# ------------------------------------------------------------------------------------------ one iteration
def run(s):
    case, ctx, W, X, aux, buf, clock = s["case"], s["ctx"], s["W"], s["X"], s["aux"], s["buf"], s["clock"]
    s["clock"] = clock + 1
    if case["call"] == "step":
        ctx.step(W, X, aux, buf, case["eta"], clock=clock)
    else:
        ctx.compute_factors(W, X, aux, s["U"], s["V"])
        ctx.pack(s["U"], s["V"], aux, buf, clock)
        ctx.apply(W, buf, case["eta"])
    if case.get("prox"):
        ctx.prox(W)
    return s["out"]


def work(case):
    """Samples (and labels, codes, data) in, W in and out, the committed buffer out; 2 J D K multiply-adds' worth of
    flops for the factors and as many for the apply (for sparse codes: per nonzero)."""
    J, D, K = case["J"], case["D"], case["P"] * case["B"]
    es = 2 if case["path"] == "bf16" else 4
    n = 8.0 * J * D
    if case["model"] == "sc":
        nnz = K * D * case["density"]
        n += 2 * 8 * nnz + 2 * 4.0 * K * J
        return dict(bytes=n, flops=4.0 * J * nnz)
    n += K * D * es * (2 if case["model"] == "dml" else 1)          # the samples
    n += K * (J + D) * es                                           # the factors
    if case.get("dual"):
        n += 8.0 * K * J
    return dict(bytes=n, flops=4.0 * J * D * K)


def tolerance(case):
    # fp32 sums of up to 20000 terms, and fp32-grade compensated ones, agree with a 64-bit evaluation to 1e-6 .. 4e-6
    # on u; operands of 11 significant bits (tf32) to about 1e-3 on u = W d, of 8 (bf16) to a few 1e-3 on W's change.
    return {"rel": {"f32": 1e-5, "tf32x3": 1e-5, "tf32": 3e-3, "bf16": 1e-2}[case["path"]]}
