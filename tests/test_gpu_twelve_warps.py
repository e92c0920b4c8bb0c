"""Dequantised products on a short K in several rounds of tiles, whose kernels for int8 results have twelve epilogue warps: ragged rows, columns and
tiles of fewer boxes than warps, one k-block to one more than the rule takes, against the exact integer product."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import to_device

pytestmark = pytest.mark.gpu


# (test_split_choice_cpu.py holds them to twelve warps and the one of seven k-blocks to eight)
SHAPES = [(5920, 960, 256), (3104, 4128, 768), (2080, 9248, 1504), (4640, 3424, 1568), (19232, 224, 32)]


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_against_the_exact_product(M, N, K):
    from paper_2104_08378_b200 import binding as sp
    rng = np.random.default_rng(M + N + K)
    a, bt = (rng.integers(-128, 128, s, dtype=np.int8) for s in ((M, K), (N, K)))
    vals, meta, _ = sp.compress(to_device(a, "i8"))
    scale, bias = (rng.normal(size=M) / (40 * K ** .5)).astype(np.float32), rng.normal(size=M).astype(np.float32)
    sd, bd = torch.from_numpy(scale).cuda(), torch.from_numpy(bias).cuda()
    acc = (oracle.prune(a, "i8").astype(np.float32) @ bt.astype(np.float32).T).astype(np.int32)  # exact: sums below 2^24
    value, code = oracle.dequant(acc, scale, bias, relu=True, out_scale=0.02)
    for cols in (False, True):
        form = (lambda t: t.t()) if cols else (lambda t: t)
        for cd in ("i8", "bf16"):
            wide = torch.full((N, M + 32) if cols else (M, N + 32), 7, device="cuda").to(sp.TORCH_DTYPE[cd])
            out = wide[:, :M if cols else N]
            sp.gemm_i8_dequant(vals, meta, to_device(bt, "i8"), sd, bias=bd, relu=True, out_scale=0.02, cd=cd, cd_col_major=cols, out=out)
            got = form(out).cpu()
            assert (wide[:, M if cols else N:] == 7).all()
            if cd == "i8":
                assert np.array_equal(got.numpy(), code)
            else:  # a rounding in FP32, and that to the type
                assert (np.abs(got.double().numpy() - value) <= (2.0 ** -8 + 2.0 ** -22) * (np.abs(value) + np.abs(bias[:, None]))).all()
