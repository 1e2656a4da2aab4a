"""Tile shapes and reduction ranges of the tensor-core GEMMs where they change over, against the oracle.

Few tiles (up to 16 ranges, the last one shorter), row units that straddle workers (samples are tiled across workers),
a lone row unit, pair tiles whose last pair is half empty, and shapes just below and above a full wave of pair tiles.
"""
import pytest

from sfbgen import scaled
from tests.test_gpu_parity import check_config

pytestmark = pytest.mark.gpu

SHAPES = [
    (257, 1000, 2, 100),     # 6 tiles, ranges; samples of two workers in one row unit
    (20, 9000, 3, 43),       # one tile, sixteen ranges
    (129, 2104, 7, 37),      # rows 0..258: three units, the last of three rows
    (1000, 520, 2, 50),      # a lone row unit
    (2304, 1032, 9, 57),     # pair tiles: 513 rows, an odd number of row units
]


@pytest.mark.parametrize("path", ["tf32", "bf16", "tf32x3"])
@pytest.mark.parametrize("J,D,P,B", SHAPES)
def test_mlr_at_tile_changes(path, J, D, P, B):
    cfg = scaled("C4" if path == "bf16" else "C1", J=J, D=D, P=P, B=B, pool=1, labels="uniform")
    cfg["path"] = path
    check_config(cfg, path, eta=0.3 if path != "bf16" else 0.05, steps=2)


@pytest.mark.parametrize("path", ["tf32", "tf32x3"])
@pytest.mark.parametrize("name,over,eta", [
    ("C2", dict(J=140, D=2008, P=5, B=53), 1e-4),               # operand rows in the buffer's streams: per worker
    ("C3", dict(J=300, D=1500, P=7, B=21, density=0.05), 1e-3),  # dense code rows: across workers
])
def test_other_models_at_tile_changes(path, name, over, eta):
    cfg = scaled(name, **over)
    cfg["path"] = path
    check_config(cfg, path, eta=eta, steps=2)
