"""apply_mask's vector kernel where its launch geometry can go wrong: one unit to a row, rows that end inside an unrolled
step, more rows than a block covers, both metadata layouts, padded rows, in place, and metadata whose two positions are
equal or in falling order (the positions named are kept, whatever they are).  Bytes, against the oracle and a numpy
restatement."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import to_device, to_host_bits

pytestmark = pytest.mark.gpu


def _rand(dtype, rows, cols, seed):
    rng = np.random.default_rng(seed)
    if dtype == "i8":
        return rng.integers(-128, 128, (rows, cols), dtype=np.int8)
    return rng.integers(0, 1 << 16, (rows, cols), dtype=np.uint16)


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("dtype", ["bf16", "i8"])
@pytest.mark.parametrize("shape", [(1, 16), (9, 48), (130, 1040), (257, 272), (37, 4112), (300, 8208)])
def test_against_the_oracle(dtype, shape, layout):
    from paper_2104_08378_b200 import binding as sp
    M, K = shape
    x, w = _rand(dtype, M, K, 1), _rand(dtype, M, K, 2)
    _, meta_ref, _ = oracle.compress(x, dtype)
    want = oracle.apply_mask(w, meta_ref, dtype)
    _, meta, _ = sp.compress(to_device(x, dtype), layout=layout)
    for pad in (0, 32):
        wide = to_device(np.full((M, K + pad), 7, dtype=w.dtype), dtype)
        wide[:, :K] = to_device(w, dtype)
        out = torch.zeros_like(wide)
        assert np.array_equal(to_host_bits(sp.apply_mask(wide[:, :K], meta, layout=layout, out=out[:, :K])), want)
        assert not out[:, K:].any()
        sp.apply_mask(wide[:, :K], meta, layout=layout, out=wide[:, :K])
        assert np.array_equal(to_host_bits(wide[:, :K]), want) and (wide[:, K:] == to_device(np.full((1, 1), 7, dtype=w.dtype), dtype)).all()


@pytest.mark.parametrize("dtype", ["f16", "i8"])
def test_any_two_positions(dtype):
    from paper_2104_08378_b200 import binding as sp
    M, K = 64, 512
    w = _rand(dtype, M, K, 3)
    meta = np.random.default_rng(4).integers(0, 256, (M, K // 8), dtype=np.uint8)
    nibbles = np.stack([meta & 15, meta >> 4], -1).reshape(M, K // 4)
    keep = np.zeros((M, K // 4, 4), bool)
    for p in (nibbles & 3, nibbles >> 2):
        np.put_along_axis(keep, p[..., None].astype(np.int64), True, -1)
    got = sp.apply_mask(to_device(w, dtype), torch.from_numpy(meta).cuda().view(-1), layout=0)
    assert np.array_equal(to_host_bits(got), np.where(keep.reshape(M, K), w, 0).astype(w.dtype))
