"""apply_mask on rows of whole 32-byte cells: 8, 16 and 32 cells of a row to a warp and one more or fewer, row groups that end
half-way, rows at 32-byte and at 16-byte boundaries (another kernel), any two positions, both layouts, in place."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import to_device, to_host_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("dtype,M,K", [("bf16", 16, 128), ("bf16", 9, 144), ("bf16", 40, 256), ("bf16", 33, 272), ("bf16", 128, 512),
                                       ("bf16", 70, 528), ("bf16", 24, 11632), ("i8", 16, 256), ("i8", 25, 288), ("i8", 130, 512),
                                       ("i8", 48, 1024), ("i8", 7, 1056)])
def test_cells(dtype, M, K, layout):
    from paper_2104_08378_b200 import binding as sp
    rng = np.random.default_rng(M * K)
    raw, kind = (np.int16, torch.bfloat16) if dtype == "bf16" else (np.int8, torch.int8)
    w = rng.integers(np.iinfo(raw).min, np.iinfo(raw).max + 1, (M, K)).astype(raw)
    x = rng.integers(np.iinfo(raw).min, np.iinfo(raw).max + 1, (M, K)).astype(raw)
    bits = x.view(np.uint16) if dtype == "bf16" else x
    _, meta_ref, _ = oracle.compress(np.ascontiguousarray(bits), dtype)
    want = oracle.apply_mask(w.view(np.uint16) if dtype == "bf16" else w, meta_ref, dtype)
    _, meta, _ = sp.compress(to_device(np.ascontiguousarray(bits), dtype), layout=layout)
    for shift in (0, 8 if dtype == "bf16" else 16):  # elements: 16 bytes
        for in_place in (False, True):
            src, dst = (torch.full((M * K + 64,), 7, dtype=torch.int16 if dtype == "bf16" else torch.int8, device="cuda") for _ in range(2))
            a, b = (t[shift:shift + M * K].view(M, K) for t in (src, dst))
            a.copy_(torch.from_numpy(w))
            out = a if in_place else b
            got = sp.apply_mask(a.view(kind), meta, layout=layout, out=out.view(kind))
            assert np.array_equal(to_host_bits(got), want)
            whole = src if in_place else dst
            assert (whole[:shift] == 7).all() and (whole[shift + M * K:] == 7).all()
