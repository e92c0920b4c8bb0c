"""Matrices with more rows than the blocks of the compression's launch cover in one step (8 blocks an SM, which then loop over
the rows), with the last step ragged: bytes against the oracle, both layouts, alone and fused with the pruning."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import to_device, to_host_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("dtype,K", [("bf16", 1024), ("f16", 272), ("i8", 2048), ("i8", 528)])
@pytest.mark.parametrize("M", [9601, 20000])
def test_against_the_oracle(dtype, K, M, layout):
    from paper_2104_08378_b200 import binding as sp
    rng = np.random.default_rng(M + K)
    x = rng.integers(-128, 128, (M, K), dtype=np.int8) if dtype == "i8" else rng.integers(0, 1 << 16, (M, K), dtype=np.uint16)
    v_ref, m_ref, _ = oracle.compress(x, dtype)
    xd = to_device(x, dtype)
    vals, meta, dropped = sp.compress(xd, layout=layout, count_dropped=True)
    pruned, vals2, meta2, dropped2 = sp.prune_compress(xd, layout=layout, count_dropped=True)
    assert np.array_equal(to_host_bits(vals), v_ref) and torch.equal(vals.view(torch.uint8), vals2.view(torch.uint8))
    assert torch.equal(meta, meta2) and torch.equal(dropped, dropped2)
    if layout == sp.META_CANONICAL:
        assert np.array_equal(meta.cpu().numpy(), np.asarray(m_ref).reshape(-1))
    assert np.array_equal(to_host_bits(pruned), oracle.prune(x, dtype))
    back = sp.decompress(vals, meta, layout=layout)
    assert np.array_equal(to_host_bits(back), to_host_bits(pruned))
