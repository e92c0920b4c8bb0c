"""The compression's work units (32 bytes of two rows, eight apart) where they can go wrong: half a unit at the end of a row,
rows of as many units as a warp takes and one more, row groups that end half-way, operands at 16-byte but not 32-byte
boundaries.  Values, metadata, pruned matrix and dropped count against the oracle, both layouts."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import to_host_bits

pytestmark = pytest.mark.gpu
STORE = {"bf16": (torch.int16, torch.bfloat16), "i8": (torch.int8, torch.int8)}


def _strided(x, dtype, pad, shift):
    """The matrix on the GPU in rows that are `pad` elements longer, its first element `shift` elements into a buffer."""
    M, K = x.shape
    raw, kind = STORE[dtype]
    flat = torch.zeros(M * (K + pad) + shift, dtype=raw, device="cuda")
    view = flat[shift:].view(M, K + pad)[:, :K]
    view.copy_(torch.from_numpy(x.view(np.int16) if dtype == "bf16" else x))
    return view.view(kind)


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("pad,shift", [(0, 0), (16, 0), (0, 16), (8, 8)])
@pytest.mark.parametrize("dtype,M,K", [("bf16", 1, 16), ("bf16", 9, 128), ("bf16", 24, 144), ("bf16", 128, 256), ("bf16", 200, 272),
                                       ("bf16", 128, 512), ("i8", 1, 16), ("i8", 17, 48), ("i8", 40, 256), ("i8", 128, 512),
                                       ("i8", 130, 528), ("i8", 128, 768)])
def test_units_against_the_oracle(dtype, M, K, pad, shift, layout):
    from paper_2104_08378_b200 import binding as sp
    if dtype == "i8":  # (the same bytes as for 16-bit types)
        pad, shift = 2 * pad, 2 * shift
    rng = np.random.default_rng(M * K + pad + shift)
    pool = [-128, -127, -2, -1, 0, 1, 2, 127] if dtype == "i8" else [0, 0x8000, 1, 0x8001, 0x3F80, 0xBF80, 0x7F80, 0xFFC0, 0x7FFF]
    x = np.array(pool, dtype=np.int8 if dtype == "i8" else np.uint16)[rng.integers(0, len(pool), (M, K))]
    v_ref, m_ref, d_ref = oracle.compress(x, dtype)
    expect = np.asarray(m_ref).ravel() if layout == sp.META_CANONICAL else oracle.meta_to_operand_order(m_ref, dtype)
    xd = _strided(x, dtype, pad, shift)
    vals, meta, dropped = sp.compress(xd, layout=layout, count_dropped=True)
    pruned = _strided(np.zeros_like(x), dtype, pad, shift)
    _, vals2, meta2, dropped2 = sp.prune_compress(xd, layout=layout, count_dropped=True, pruned=pruned)
    for v, m, d in ((vals, meta, dropped), (vals2, meta2, dropped2), sp.compress(xd, layout=layout)):
        assert np.array_equal(to_host_bits(v), v_ref) and np.array_equal(m.cpu().numpy(), expect)
        assert d is None or int(d) == d_ref
    assert np.array_equal(to_host_bits(pruned.contiguous()), oracle.prune(x, dtype))
    assert np.array_equal(to_host_bits(sp.prune(xd).contiguous()), oracle.prune(x, dtype))
