"""The sparse-v apply at the edges of its slices of samples, blocks of atoms and blocks of rows, against the oracle.

1408 samples fill one slice of u in shared memory, 1409 take two; the codes are sorted in chunks of 32 samples; blocks
are 32 rows of W by 8 atoms; columns are streamed in groups of four entries, 128 at a time
(density 1: every column holds every sample).
"""
import pytest

from sfbgen import scaled
from tests.test_gpu_parity import check_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("J,D,P,B,density", [
    (3, 9, 1, 2, 1.0), (64, 8, 1, 4, 1.0), (65, 7, 3, 11, 1.0), (63, 17, 8, 87, 0.3), (130, 33, 17, 41, 0.3),
    (70, 1003, 5, 300, 0.02), (200, 400, 2, 16, 0.004), (4100, 40, 2, 20, 0.2),
    (32, 9, 8, 176, 0.3), (33, 8, 1, 1409, 0.3), (31, 200, 20, 142, 0.05), (97, 15, 1, 12, 1.0),
    (40, 8200, 1, 32, 0.01), (40, 64, 3, 11, 0.5),
])
def test_sparse_steps_match_the_oracle(J, D, P, B, density):
    cfg = scaled("C3", J=J, D=D, P=P, B=B, density=density)
    cfg["path"] = "f32"
    check_config(cfg, "f32", eta=1e-2, steps=2)
