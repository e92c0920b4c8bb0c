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


@pytest.mark.parametrize("dtype,K,layout", [("bf16", 2**28 + 4096, 1), ("e5m2", 2**28 + 4096, 1), ("i8", 2**32 + 4096, 0)])
def test_prune_and_compress(dtype, K, layout):
    """One long row is, group by group, the matrix of its pieces: values, canonical metadata and pruned matrix of both are the
    same bytes in the same order, and the operand order holds the same bits."""
    from paper_2104_08378_b200 import binding as sp
    x = _matrix(dtype, K, torch.Generator(device="cuda").manual_seed(42))
    pieces = x.view(-1, 4096)
    want_pruned, want_vals, want_meta, want_dropped = sp.prune_compress(pieces, layout=sp.META_CANONICAL, count_dropped=True)
    vals, meta, dropped = sp.compress(x, layout=layout, count_dropped=True)
    for v, m, d in ((vals, meta, dropped), sp.prune_compress(x, layout=layout, count_dropped=True)[1:]):
        assert torch.equal(_bits(v).view(-1), _bits(want_vals).view(-1)) and torch.equal(d, want_dropped)
        if layout == sp.META_CANONICAL:
            assert torch.equal(m.view(-1), want_meta.view(-1))
        else:
            blocks, at = _first_row(m, x.element_size())
            assert torch.equal(blocks[:, at], want_meta.view(torch.int16).view(-1, 8))
            assert (blocks[:, [i + 8 for i in at]] == 0x4444).all()              # row 1: padding
    assert torch.equal(_bits(sp.prune(x)).view(-1), _bits(want_pruned).view(-1))
    assert torch.equal(_bits(sp.decompress(vals, meta, layout=layout)).view(-1), _bits(want_pruned).view(-1))


def test_pairs_of_float32():
    from paper_2104_08378_b200 import binding as sp
    K = 2**27 + 4096                     # the operand order of the 1:2 pattern: 64 columns to a 2048-byte block
    x = torch.randn((1, K), device="cuda", generator=torch.Generator(device="cuda").manual_seed(43))
    want_vals, want_meta, _ = sp.compress(x.view(-1, 4096), layout=sp.META_CANONICAL)
    vals, meta, _ = sp.compress(x)
    blocks, at = _first_row(meta, 2)
    assert torch.equal(vals.view(-1), want_vals.view(-1)) and torch.equal(blocks[:, at], want_meta.view(torch.int16).view(-1, 8))
    assert torch.equal(sp.decompress(vals, meta).view(-1), sp.prune(x.view(-1, 4096)).view(-1))
