"""Code rows that repeat an atom behind a smaller one (5, 3, 5) or descend: forward and apply take the same entries, on
every path and every call, and the result is reproducible.  The rule: an entry counts if its atom exists and exceeds its
predecessor's; values of an atom that counts twice add up."""
import numpy as np
import pytest
import torch

from oracle import sfb_oracle as orc
from sfbgen import make_inputs, scaled
from tests.test_gpu_parity import _workload
from tests.util import TOL

pytestmark = pytest.mark.gpu


def _merged(rp, ix, vl, D):
    """The same codes as well-formed rows."""
    rows, idx, val = [0], [], []
    for i in range(rp.size - 1):
        a = {}
        for k in range(rp[i], rp[i + 1]):
            if ix[k] < D and not (k > rp[i] and ix[k - 1] >= ix[k]):
                a[int(ix[k])] = a.get(int(ix[k]), 0.0) + float(vl[k])
        idx += sorted(a)
        val += [a[d] for d in sorted(a)]
        rows.append(len(idx))
    return np.array(rows, np.uint32), np.array(idx, np.uint32), np.array(val, np.float32)


@pytest.mark.parametrize("path,J,D,P,B,density", [("f32", 70, 120, 2, 20, 0.15), ("tf32", 70, 120, 2, 20, 0.15), ("tf32x3", 70, 120, 2, 20, 0.15),
                                                  ("f32", 40, 3000, 1, 5, 0.5), ("f32", 12, 72, 4, 4101, 0.1)])
def test_repeated_and_descending_atoms(path, J, D, P, B, density):
    from paper_1511_08486_b200 import binding
    cfg = scaled("C3", J=J, D=D, P=P, B=B, density=density)
    cfg["path"], cfg["pool"] = path, 1
    inputs = make_inputs(cfg)
    rp = inputs["rowptr"][0].astype(np.int64)
    ix, vl = inputs["idx"][0].copy(), inputs["val"][0]
    changed = 0
    for i in (0, 3, cfg["K"] // 2, cfg["K"] - 1):
        n = rp[i + 1] - rp[i]
        if n < 4:
            continue
        changed += 1
        row = ix[rp[i]:rp[i + 1]]
        row[-1] = row[-3]                 # ..., a, b, a with b < a, or (all but the first) a row that falls and rises again
        row[-2] = 0
        if i and n > 6:
            row[1], row[2] = row[n // 2], row[0]
    assert changed >= 2
    inputs["idx"][0] = ix
    wl = _workload(cfg, inputs, path, guard=True)
    try:
        eta = 1e-2
        wl.step(0, eta=eta)
        assert wl.ctx.status() & binding.SFB_DEV_BAD_INDEX
        W1, buf = wl.W.clone(), wl.sf_buf.clone()
        rows, idx, val = _merged(rp, ix, vl, D)
        W_or, U_or, _ = orc.step(orc.MODEL_SC, inputs["W"], dict(rowptr=rows, idx=idx, val=val, Xdata=inputs["Xdata"][0]), eta)
        W0 = inputs["W"].astype(np.float64)
        err = np.linalg.norm((W1.cpu().numpy() - W0) - (W_or - W0)) / np.linalg.norm(W_or - W0)
        assert err <= TOL[path] + 2.0 ** -24 * np.linalg.norm(W0) / np.linalg.norm(W_or - W0), f"{err:.3e}"
        _, U_wire, _ = orc.unpack(buf.cpu().numpy())
        assert orc.rel_fro(U_wire, U_or) <= TOL[path]
        for _ in range(2):                # again, and by the separate calls
            wl.reset()
            wl.step(0, eta=eta)
            assert torch.equal(wl.W, W1)
            wl.reset()
            wl.compute_factors(0)
            wl.pack(0)
            wl.apply(eta)
            assert wl.ctx.status() & binding.SFB_DEV_BAD_INDEX
            assert torch.equal(wl.W, W1)
        assert wl.guards_intact()
    finally:
        wl.close()
