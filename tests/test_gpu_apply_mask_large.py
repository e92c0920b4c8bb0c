"""apply_mask on matrices large enough to leave the kernels' usual road: more row groups than blocks are launched for, so that the
cells' row loop takes a second step, and either side of the size from which whole cells go by 16-byte units.  Any two positions,
both layouts, in place; every row against the elements that the metadata names."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("dtype,M,K", [("i8", 524288 + 37, 1024), ("bf16", 10240, 4096), ("bf16", 10241, 4096), ("i8", 10405, 8064)])
def test_every_row(dtype, M, K, in_place, layout):
    from paper_2104_08378_b200 import binding as sp
    g = torch.Generator(device="cuda").manual_seed(M + K)
    kind = torch.int8 if dtype == "i8" else torch.bfloat16
    kept = torch.randint(0, 6, (M, K // 4), device="cuda", generator=g)          # which two of a group's four positions
    pairs = torch.tensor([[1, 1, 0, 0], [1, 0, 1, 0], [1, 0, 0, 1], [0, 1, 1, 0], [0, 1, 0, 1], [0, 0, 1, 1]], dtype=torch.int8, device="cuda")
    mask = pairs[kept].view(M, K)
    _, meta, _ = sp.compress(mask if dtype == "i8" else mask.bfloat16(), layout=layout)
    w = torch.randint(1, 127, (M, K), dtype=torch.int8, device="cuda", generator=g)
    want = w * mask
    src = w.to(kind)
    out = src if in_place else torch.full_like(src, 7)
    sp.apply_mask(src, meta, layout=layout, out=out)
    assert torch.equal(out, want.to(kind))
