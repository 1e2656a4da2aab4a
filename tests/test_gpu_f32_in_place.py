"""The one-launch fp32 forward on 128 x 128 tiles, and the finishing passes of many rows, at their edges, against the oracle
with guard bands: classes one beyond a tile, ragged and short feature rows, samples that straddle workers (the first three are
taken in place with and without pairs, the next two thirds with pairs); 512 / 513 / 1024 / 1025 classes; directories of more
than one block (more than 512 workers).
"""
import pytest

from sfbgen import scaled
from tests.test_gpu_parity import check_config

pytestmark = pytest.mark.gpu

SHAPES = [(257, 70, 50, 250), (65, 33, 100, 366), (385, 61, 73, 128), (200, 17, 13, 500), (512, 20, 5, 300), (513, 64, 30, 90), (1024, 12, 3, 420),
          (1025, 100, 4, 400), (10, 64, 1300, 1), (70, 100, 513, 3)]


@pytest.mark.parametrize("J,D,P,B", SHAPES)
def test_mlr(J, D, P, B):
    check_config(scaled("C1", J=J, D=D, P=P, B=B, pool=1), "f32", eta=0.5, steps=2, guard=True)


@pytest.mark.parametrize("J,D,P,B", SHAPES)
def test_dml(J, D, P, B):
    check_config(scaled("C2", J=J, D=D, P=P, B=B), "f32", eta=1e-3, steps=2, guard=True)


@pytest.mark.parametrize("path,J,D,P,B", [("tf32", 40, 64, 1300, 1), ("tf32x3", 70, 100, 700, 2), ("bf16", 520, 64, 620, 3)])
def test_large_directories(path, J, D, P, B):
    name, over = ("C4", dict(labels="uniform")) if path == "bf16" else ("C1", {})
    check_config(scaled(name, J=J, D=D, P=P, B=B, pool=1, **over), path, eta=0.05, steps=1, guard=True)
