"""INT32 accumulators whose k-blocks a cluster of 2, 4 or 8 CTAs shares: every form of the result at ragged rows, columns and
k-blocks, bit for bit against the exact integer product, and an expired wait in such a cluster."""
import os
import re
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
from gpu_util import to_device

pytestmark = pytest.mark.gpu

# M, N, K, the CTAs that share a tile's k-blocks and the tile's columns (test_split_choice_cpu.py holds the choice to these)
SHAPES = [(3072, 32, 4096, 4, 32), (416, 96, 2592, 4, 32), (160, 32, 8224, 8, 32), (32, 32, 4128, 8, 32), (672, 320, 10720, 4, 64),
          (6432, 32, 4128, 2, 32), (192, 608, 10688, 4, 64), (2944, 192, 10016, 2, 64), (736, 416, 10176, 4, 96),
          (672, 1024, 7520, 2, 96), (608, 1760, 11488, 2, 128)]
EXPIRED_WAIT = (1024, 32, 4096, 8, 32)


@pytest.fixture(scope="module")
def sp():
    from paper_2104_08378_b200 import binding
    return binding


def _operands(sp, M, N, K):
    rng = np.random.default_rng(M + N + K)
    a, bt = (rng.integers(-128, 128, s, dtype=np.int8) for s in ((M, K), (N, K)))
    vals, meta, _ = sp.compress(to_device(a, "i8"))
    # exact in float64: every partial sum is below K / 2 * 2^14
    acc = (oracle.prune(a, "i8").astype(np.float64) @ bt.astype(np.float64).T).astype(np.int32)
    return vals, meta, to_device(bt, "i8"), acc, rng


@pytest.mark.parametrize("M,N,K,parts,columns", SHAPES)
def test_every_form_of_the_result(sp, M, N, K, parts, columns):
    vals, meta, x, acc, rng = _operands(sp, M, N, K)
    c = rng.integers(-1 << 30, 1 << 30, (M, N), dtype=np.int32)
    scale, bias = (rng.normal(size=M) / (40 * K ** .5)).astype(np.float32), rng.normal(size=M).astype(np.float32)
    sd, bd = torch.from_numpy(scale).cuda(), torch.from_numpy(bias).cuda()
    value, code = oracle.dequant(acc, scale, bias, relu=False, out_scale=0.02)
    for cols in (False, True):
        form = (lambda t: t.t().contiguous()) if cols else (lambda t: t)
        wide = torch.full((N, M + 32) if cols else (M, N + 32), 7, dtype=torch.int32, device="cuda")
        out = wide[:, :M if cols else N]
        sp.gemm(vals, meta, x, cd="i32", out=out, cd_col_major=cols)
        assert np.array_equal(form(out).cpu().numpy(), acc) and (wide[:, M if cols else N:] == 7).all()
        got = sp.gemm(vals, meta, x, cd="i32", beta=1, C=form(torch.from_numpy(c).cuda()), cd_col_major=cols)
        assert np.array_equal(form(got).cpu().numpy(), acc + c)
        for cd, eps in (("i8", None), ("bf16", 2.0 ** -8), ("f16", 2.0 ** -11), ("f32", 2.0 ** -23)):
            got = form(sp.gemm_i8_dequant(vals, meta, x, sd, bias=bd, out_scale=0.02, cd=cd, cd_col_major=cols)).cpu()
            if cd == "i8":
                assert np.array_equal(got.numpy(), code)
            else:  # a rounding of the accumulator and one of scale * accumulator + bias in FP32, and that to the type
                bound = (eps + 2.0 ** -22) * (np.abs(value) + np.abs(bias[:, None])) + 2.0 ** -24
                assert (np.abs(got.double().numpy() - value) <= bound).all()


def test_the_device_takes_them():
    """What the library says of its choices here; a part with fewer clusters may choose other numbers than the ones above."""
    code = ("import sys, torch; sys.path[:0] = sys.argv[1:]\n"
            "from paper_2104_08378_b200 import binding as sp\n"
            "from test_gpu_split_k_blocks import SHAPES\n"
            "for M, N, K, *_ in SHAPES:\n"
            "    vals, meta, _ = sp.compress(torch.ones(M, K, dtype=torch.int8, device='cuda'))\n"
            "    d = sp.gemm(vals, meta, torch.ones(N, K, dtype=torch.int8, device='cuda'), cd='i32')\n"
            "    assert (d == K // 2).all()\n")
    here = os.path.dirname(os.path.abspath(__file__))
    said = subprocess.run([sys.executable, "-c", code, os.path.dirname(here), here], env={**os.environ, "SP24_LOG": "1"},
                          capture_output=True, text=True, check=True).stderr
    parts = [int(n) for n in re.findall(r"split=(\d+)", said)]
    assert len(parts) == len(SHAPES) and min(parts) > 1, said


def _expired(sp, skip, M, N, K):
    """(D, status record) of a product on an untouched D of sevens, with the hook's k-blocks left out."""
    vals, meta, x, acc, _ = _operands(sp, M, N, K)
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    out = torch.full((M, N), 7, dtype=torch.int32, device="cuda")
    sp.set_fault_hooks(20000000, skip)  # ~10 ms of SM clock per wait
    try:
        sp.gemm(vals, meta, x, cd="i32", ws=ws, out=out)
        torch.cuda.synchronize()
    finally:
        sp.set_fault_hooks(0, False)
    words = ws.view(torch.int32)[:2].tolist()
    assert sp.gemm_status(ws) != 0 and sp.gemm_status(ws) == 0
    for _ in range(3):
        assert np.array_equal(sp.gemm(vals, meta, x, cd="i32", ws=ws).cpu().numpy(), acc)
    assert sp.gemm_status(ws) == 0
    return out, words


@pytest.mark.parametrize("M,N,K,parts,columns", [EXPIRED_WAIT, SHAPES[0]])
def test_one_cta_of_a_cluster_gives_up(sp, M, N, K, parts, columns):
    """One k-block of rank r is left out.  The other CTAs have all of theirs, and their waits for the sums of rank r, which itself
    waits longer, are the first to expire: nothing of D is written, and every CTA of every cluster has given up."""
    for rank in range(parts):
        out, (code, expired) = _expired(sp, 2 + rank, M, N, K)
        assert (out == 7).all()
        assert code == 6                           # the others' sums
        assert expired >= parts * ((M + 127) // 128)


def test_expired_wait(sp):
    """One k-block of each part left out."""
    out, (code, _) = _expired(sp, True, *EXPIRED_WAIT[:3])
    assert (out == 7).all() and code in (1, 3, 4)  # ring, operands, accumulators
