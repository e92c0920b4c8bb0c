"""Column-major results are the row-major ones transposed, bit for bit, for every output type and tile shape.

Both orders convert the same accumulators with the same operations; they differ in how a 32 x 32 box leaves the
registers (transposing buffer, ldmatrix, direct stores).  Row-major results are compared with the oracle elsewhere.
The outputs are slices of wider buffers whose remaining columns must keep their fill."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

TORCH = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32, "i32": torch.int32, "i8": torch.int8}
# (operand kind, output type); dq: the dequantising epilogue
KINDS = [("bf16", "bf16"), ("f16", "f16"), ("bf16", "f32"), ("tf32", "f32"), ("e4m3", "bf16"), ("i8", "i32"),
         ("dq", "i8"), ("dq", "bf16"), ("dq", "f32")]
TILES = [None, "1x128x1", "2x224x1", "2x224x2", "2x240x1", "2x256x1"]
SHAPES = [(32, 32, 64), (160, 96, 288), (544, 480, 128), (1056, 736, 256)]   # partial boxes, quarters, m-blocks, tiles


@pytest.fixture(scope="module")
def sp():
    from paper_2104_08378_b200 import binding
    return binding


def _operands(kind, M, N, K):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + 7 * N + K)
    if kind in ("i8", "dq"):
        return [torch.randint(-128, 128, s, dtype=torch.int8, device="cuda", generator=g) for s in ((M, K), (N, K))]
    dt = {"bf16": torch.bfloat16, "f16": torch.float16, "tf32": torch.float32, "e4m3": torch.float8_e4m3fn}[kind]
    return [torch.randn(s, device="cuda", generator=g).to(dt) for s in ((M, K), (N, K))]


def _padded(rows, cols, dt, extra=32):
    """A slice [rows, cols] of a wider buffer filled with 7s."""
    return torch.full((rows, cols + extra), 7, device="cuda", dtype=torch.float32).to(dt)


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("kind,cd", KINDS)
def test_column_major_is_the_transpose(sp, force_tile, kind, cd, tile):
    if tile == "2x240x1" and (kind not in ("bf16", "f16") or cd == "f32"):
        pytest.skip("240-column tiles are built for the 16-bit kinds with 16-bit results")
    for M, N, K in SHAPES:
        A, Bt = _operands(kind, M, N, K)
        vals, meta, _ = sp.compress(A)
        row, col = _padded(M, N, TORCH[cd]), _padded(N, M, TORCH[cd])
        if tile:
            force_tile(tile)
        if kind == "dq":
            scale = torch.linspace(0.5, 1.5, M, device="cuda") / (100.0 * K ** 0.5)
            bias = torch.linspace(-1.0, 1.0, M, device="cuda")
            for relu in (False, True):
                for out, flag in ((row[:, :N], False), (col[:, :M], True)):
                    sp.gemm_i8_dequant(vals, meta, Bt, scale, bias=bias, relu=relu, out_scale=0.5, cd=cd, out=out,
                                       cd_col_major=flag)
                assert torch.equal(row[:, :N].t(), col[:, :M])
            if cd == "i8":     # and the codes are the oracle's
                v_ref, m_ref, _ = oracle.compress(A.cpu().numpy(), "i8")
                acc = oracle.gemm_sparse(v_ref, m_ref, Bt.cpu().numpy(), "i8")
                _, q = oracle.dequant(acc, scale.cpu().numpy(), bias.cpu().numpy(), relu=True, out_scale=0.5)
                assert np.array_equal(row[:, :N].cpu().numpy(), q)
        else:
            C = torch.arange(M * N, device="cuda").remainder(251).sub(125).to(TORCH[cd]).view(M, N)
            Ct = C.t().contiguous()
            for beta in (0, 1) if cd == "i32" else (0.0, -1.5):
                kw = dict(beta=beta, cd=cd)
                sp.gemm(vals, meta, Bt, C=C if beta else None, out=row[:, :N], **kw)
                sp.gemm(vals, meta, Bt, C=Ct if beta else None, out=col[:, :M], cd_col_major=True, **kw)
                assert torch.equal(row[:, :N].t(), col[:, :M])
                if beta:   # C and D may be the same buffer
                    inplace = Ct.clone()
                    sp.gemm(vals, meta, Bt, C=inplace, out=inplace, cd_col_major=True, **kw)
                    assert torch.equal(inplace, col[:, :M])
        assert (row[:, N:].float() == 7).all() and (col[:, M:].float() == 7).all()
        assert sp.gemm_status(device=A.device) == 0
