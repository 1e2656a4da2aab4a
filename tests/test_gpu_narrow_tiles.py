"""Tensor-core tiles of 64 columns (small problems, singles only) at their edges, against the oracle with guard bands: rows and
columns one unit around a tile, samples that straddle workers, fewer samples than a tile has rows, reductions of one atom and
of several ranges.  All of these shapes take such tiles in the update, most of them in the forward too.
"""
import re

import pytest
import torch

from sfbgen import make_inputs, scaled
from tests.test_gpu_parity import _workload, check_config

pytestmark = pytest.mark.gpu

SHAPES = [(63, 56, 2, 9), (64, 64, 1, 32), (129, 72, 3, 43), (257, 1000, 2, 100), (128, 200, 5, 130), (20, 2056, 7, 5)]   # J, D, P, B


@pytest.mark.parametrize("path", ["tf32", "bf16", "tf32x3"])
@pytest.mark.parametrize("J,D,P,B", SHAPES)
def test_mlr(path, J, D, P, B):
    name, over = ("C4", dict(labels="uniform")) if path == "bf16" else ("C1", {})
    check_config(scaled(name, J=J, D=D, P=P, B=B, pool=1, **over), path, eta=0.05 if path == "bf16" else 0.5, steps=2, guard=True)


@pytest.mark.parametrize("path", ["tf32", "tf32x3"])
@pytest.mark.parametrize("J,D,P,B", SHAPES[2:4])
def test_dml_and_sparse_coding(path, J, D, P, B):
    # two steps: the second sees the first's error times 1 + eta |v|^2, |v|^2 about 2 D (pair differences) or D / 5 (codes, a tenth
    # of them nonzero with variance 2); these eta keep that factor below 1.25, so that one step's tolerance does for both
    check_config(scaled("C2", J=J, D=D, P=P, B=B), path, eta=1e-4, steps=2, guard=True)
    check_config(scaled("C3", J=J, D=D, P=P, B=B // 4, density=0.1), path, eta=1e-3, steps=2, guard=True)


def _tile_widths(path, J, D, P, B):
    """Widths of the forward's and the update's tiles of one step, from the names of the kernels that ran."""
    from torch.profiler import ProfilerActivity, profile
    name, over = ("C4", dict(labels="uniform")) if path == "bf16" else ("C1", {})
    cfg = scaled(name, J=J, D=D, P=P, B=B, pool=1, **over)
    wl = _workload(cfg, make_inputs(cfg), path)
    try:
        wl.step(0, eta=0.0)
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            wl.step(0, eta=0.0)
            torch.cuda.synchronize()
    finally:
        wl.close()
    # umma_gemm_kernel<bytes of a value, update?, tile width, ...>
    found = [re.search(r"umma_gemm_kernel<\d+, (true|false), (\d+),", e.name) for e in prof.events()]
    found = [(m[1] == "true", int(m[2])) for m in found if m]
    return [w for update, w in found if not update], [w for update, w in found if update]


@pytest.mark.parametrize("path", ["tf32", "bf16", "tf32x3"])
def test_the_shapes_above_take_narrow_tiles(path):
    widths = [_tile_widths(path, *shape) for shape in SHAPES]
    if not any(update for _, update in widths):
        pytest.skip("no kernel names from the profiler here")
    assert all(update == [64] for _, update in widths), widths
    assert 2 * sum(forward == [64] for forward, _ in widths) > len(SHAPES), widths


@pytest.mark.parametrize("J,D,P,B", [(256, 2048, 5, 128), (300, 1280, 10, 33)])
def test_long_compensated_updates_on_pairs_keep_wide_tiles(J, D, P, B):
    """More than 14 reduction blocks of up to 32 pairs, rows of whole 128-byte units: narrow tiles lose."""
    _, update = _tile_widths("tf32x3", J, D, P, B)
    if not update:
        pytest.skip("no kernel names from the profiler here")
    assert 64 not in update, update
