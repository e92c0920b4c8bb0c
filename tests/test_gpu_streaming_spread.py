"""The streaming kernels behind a product, whose launches of up to four blocks to an SM leave room for an even spread only: sizes on
either side of each number of blocks, the product's result and every output against the oracle, also in a captured graph."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import to_device, to_host_bits

pytestmark = pytest.mark.gpu
K = 512


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("rows", [16, 2352, 2368, 2384, 4720, 4736, 4752, 7104, 7120, 9472, 9488])
def test_behind_a_product(rows, captured):
    """(bf16: 148 blocks of apply_mask and of the compression for each 2368 rows)"""
    from paper_2104_08378_b200 import binding as sp
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    M = rows * sms // 148 // 16 * 16
    rng = np.random.default_rng(rows)
    x = rng.integers(0, 0x7F80, (M, K)).astype(np.uint16) | (rng.integers(0, 2, (M, K)) << 15).astype(np.uint16)   # finite bf16
    v_ref, m_ref, _ = oracle.compress(x, "bf16")
    pruned_ref, meta_ref = oracle.prune(x, "bf16"), oracle.meta_to_operand_order(m_ref, "bf16")
    xd, a, b = to_device(x, "bf16"), torch.randn(1536, 512, device="cuda").bfloat16(), torch.randn(96, 512, device="cuda").bfloat16()
    va, ma, _ = sp.compress(a)
    want = sp.gemm(va, ma, b)
    vals, meta, pruned, masked, again = (torch.zeros_like(t) for t in (xd[:, :K // 2].contiguous(), to_device(meta_ref.view(np.int8), "i8").view(torch.uint8), xd, xd, xd))
    d = torch.zeros_like(want)

    def step():
        for f in (lambda: sp.prune_compress(xd, pruned=pruned, vals=vals, meta=meta), lambda: sp.apply_mask(xd, meta, out=masked),
                  lambda: sp.compress_into(masked, vals, meta), lambda: sp.prune(xd, out=again)):
            sp.gemm(va, ma, b, out=d)
            f()

    if captured:
        step()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            step()
        for t in (vals, meta, pruned, masked, again, d):
            t.zero_()
        graph.replay()
    else:
        step()
    torch.cuda.synchronize()
    assert torch.equal(d.view(torch.int16), want.view(torch.int16))
    assert np.array_equal(to_host_bits(vals), v_ref) and np.array_equal(meta.cpu().numpy(), meta_ref)
    for t in (pruned, masked, again):
        assert np.array_equal(to_host_bits(t), pruned_ref)
