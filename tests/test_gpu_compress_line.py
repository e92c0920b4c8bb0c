"""The compression has a kernel for matrices of few blocks and one for the others: the edges of test_gpu_compress_cells.py, whose
matrices are all for the first, at sizes for the second, and the last size of one beside the first of the other.  The largest
two are fused with the pruning by the second also at 16-byte boundaries."""
import pytest

import test_gpu_compress_cells as cells

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("pad,shift", [(0, 0), (16, 0), (0, 16), (8, 8)])
@pytest.mark.parametrize("dtype,M,K", [("bf16", 14220, 16), ("bf16", 7113, 144), ("bf16", 7072, 256), ("bf16", 7073, 256),
                                       ("bf16", 4750, 272), ("bf16", 3560, 512), ("i8", 14220, 48), ("i8", 7072, 512),
                                       ("i8", 7073, 512), ("i8", 4750, 528), ("i8", 4751, 768)])
def test_both_sides_of_the_line(dtype, M, K, pad, shift, layout):
    cells.test_units_against_the_oracle(dtype, M, K, pad, shift, layout)


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("dtype,M,K", [("bf16", 16001, 2064), ("i8", 20001, 3216)])
def test_large_at_16_byte_boundaries(dtype, M, K, layout):
    cells.test_units_against_the_oracle(dtype, M, K, 8, 8, layout)
