"""Rows whose offsets pass 32 bits: from 2^28 columns in the operand-order metadata, from 4 GiB in the matrix itself.  Bytes,
block by block, against a restatement in torch."""
import pytest
import torch

pytestmark = pytest.mark.gpu

TORCH = {"bf16": torch.bfloat16, "i8": torch.int8, "e5m2": torch.float8_e5m2}
BLOCK = 1 << 24   # columns compared at a time


def _bits(t):
    return t.view(torch.int16 if t.element_size() == 2 else torch.int8)


def _matrix(dtype, K, g):
    """One row of K columns, every bit pattern among them."""
    x = torch.empty((1, K), dtype=TORCH[dtype], device="cuda")
    for c in range(0, K, BLOCK):
        part = _bits(x)[0, c:c + BLOCK]
        part.copy_(torch.randint(-128, 128, (part.numel() * x.element_size(),), dtype=torch.int8, device="cuda",
                                 generator=g).view(part.dtype))
    return x


def _first_row(meta, es):
    """Operand-order metadata as 16-bit words and the places in a 128-column block of row 0's eight of them."""
    return meta.view(torch.int16).view(-1, 1024), [(128 * (c & 1) + 4 * (c >> 1) if es == 2 else 2 * c) // 2 for c in range(8)]


@pytest.mark.parametrize("dtype,K,layout", [("bf16", 2**28 + 4096, 1), ("i8", 2**28 + 4096, 1), ("bf16", 2**31 + 4096, 0),
                                            ("i8", 2**32 + 4096, 0)])
def test_apply_mask(dtype, K, layout):
    from paper_2104_08378_b200 import binding as sp
    g = torch.Generator(device="cuda").manual_seed(41)
    w = _matrix(dtype, K, g)
    pairs = torch.tensor([0x4, 0x8, 0xC, 0x9, 0xD, 0xE], dtype=torch.uint8, device="cuda")   # the six ascending pairs
    row = torch.empty(K // 8, dtype=torch.uint8, device="cuda")
    for c in range(0, K // 8, BLOCK):
        n = min(BLOCK, K // 8 - c)
        lo, hi = (pairs[torch.randint(0, 6, (n,), device="cuda", generator=g)] for _ in range(2))
        row[c:c + n] = lo | (hi << 4)
    if layout == sp.META_TCGEN05:
        meta = torch.full((sp.meta_bytes(dtype, 1, K, layout),), 0x44, dtype=torch.uint8, device="cuda")
        blocks, at = _first_row(meta, w.element_size())
        blocks[:, at] = row.view(torch.int16).view(-1, 8)
    else:
        meta = row
    got = sp.apply_mask(w, meta, layout=layout, out=torch.empty_like(w))
    byte = torch.arange(256, device="cuda")
    keep = torch.zeros((256, 8), dtype=torch.bool, device="cuda")
    for group in range(2):
        for position in range(2):
            keep[byte, 4 * group + ((byte >> (4 * group + 2 * position)) & 3)] = True
    for c in range(0, K, BLOCK):
        kept = keep[row[c // 8:(c + BLOCK) // 8].long()].view(-1)
        assert torch.equal(_bits(got)[0, c:c + BLOCK], torch.where(kept, _bits(w)[0, c:c + BLOCK], 0)), c
