"""Tensor-core tiles of 64 columns (small problems, singles only) at their edges, against the oracle with guard bands: rows and
columns one unit around a tile, samples that straddle workers, fewer samples than a tile has rows, reductions of one atom and
of several ranges.  All of these shapes take such tiles in the update, most of them in the forward too.
"""
import pytest

from sfbgen import scaled
from tests.test_gpu_parity import check_config

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
