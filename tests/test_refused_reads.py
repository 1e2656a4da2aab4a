"""A buffer whose header was refused is not read behind it, by any kernel of an update, read from the sources (no GPU needed).

The buffer may have been made for fewer workers, samples, classes or features, so that rows at this descriptor's offsets lie
outside of it.  Every kernel that sfb_apply launches on the buffer behind the header check has to look at the check's outcome
before its first access to rows, codes or the directory.
"""
import re

import pytest

from tests.test_chained_kernels import _kernels, _sources

ROWS = r"\.row\(|csr_row2?\("
# kernel: what its first access to the buffer looks like
READS = {
    "row_nonzero_kernel": ROWS, "kept_rows_kernel": r"\(buf \+", "planes_kernel": r"make_planes\(",
    "umma_f32_kernel": r"tma_load", "sgemm_pipe_kernel": ROWS, "sgemm_small_kernel": ROWS, "densify_kernel": ROWS,
    "csc_mask_kernel": ROWS, "csc_fill_kernel": ROWS, "csc_apply_kernel": ROWS, "sc_malformed_kernel": ROWS, "sc_apply_kernel": ROWS,
    "split_mn_kernel": r"\*reinterpret_cast<const float4\*>\(x\)", "umma_gemm_kernel": r"p\.dir\[",
}


@pytest.mark.parametrize("kernel", sorted(READS))
def test_refusal_is_looked_at_before_the_first_row(kernel):
    bodies = [b for _, text in _sources() for n, _, b in _kernels(text) if n == kernel]
    assert len(bodies) == 1, kernel
    look = re.search(r"is_refused\(|SFB_DEV_BAD_HEADER", bodies[0])
    read = re.search(READS[kernel], bodies[0])
    assert read and look and look.start() < read.start(), kernel
