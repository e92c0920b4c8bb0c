"""4-byte row-major results of at most 32 columns on pairs of CTAs: a row of boxes is one box, which two warps share out, so
that the second warp's first box is in the second m-block, or nowhere.  Bit for bit the results of 128 x 128 tiles (an
element's sum runs over K in the same order with the same instructions), and against the product in 64 bits."""
import pytest
import torch

pytestmark = pytest.mark.gpu

TORCH = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32, "e4m3": torch.float8_e4m3fn}
# kind, dense, N-contiguous B, M, N, K, the tile this takes
CASES = [("bf16", True, False, 229376, 32, 64, "2x256x2"), ("bf16", True, False, 229376 + 272, 16, 64, "2x256x2"),
         ("bf16", False, False, 57344, 32, 6144, "2x224x2"), ("f32", False, False, 57344, 16, 4096, "2x224x2"),
         ("bf16", True, False, 8192, 32, 512, "2x224x1"), ("f32", True, False, 8208, 16, 256, "2x224x1"),
         ("f16", False, True, 8192, 32, 512, "2x224x1"), ("i8", True, False, 8192, 32, 512, "2x224x1"),
         ("i8", False, True, 8224, 32, 512, "2x224x1"), ("e4m3", False, True, 8192, 32, 512, "2x224x1"),
         ("i8", False, False, 76800, 32, 12288, "2x224x1")]


@pytest.mark.parametrize("kind,dense,b_rows,M,N,K,tile", CASES)
def test_same_bits_as_128_columns(force_tile, kind, dense, b_rows, M, N, K, tile):
    from paper_2104_08378_b200 import binding as sp
    g = torch.Generator(device="cuda").manual_seed(5)

    def rand(rows, cols):
        if kind == "i8":
            return torch.randint(-128, 128, (rows, cols), dtype=torch.int8, device="cuda", generator=g)
        return torch.randn((rows, cols), device="cuda", generator=g).to(TORCH[kind])

    cd = "i32" if kind == "i8" else "f32"
    A, x = rand(M, K), rand(*((K, N) if b_rows else (N, K)))
    vals, meta = (A, None) if dense else sp.compress(A)[:2]
    desc = sp.make_desc(kind, cd, M, N, K, vals.stride(0), x.stride(0), N, N, dense, b_rows)
    assert sp.gemm_plan(desc) == tile                       # else this test does not show what it is for
    C = torch.randint(-9, 10, (M, N), device="cuda", generator=g).to(sp.TORCH_DTYPE[cd])
    for beta in (0.0, 1.0):
        got = []
        for forced in (None, "1x128x1"):
            force_tile(forced)
            got.append(sp.gemm(vals, meta, x, beta=beta, C=C if beta else None, cd=cd, b_row_major=b_rows, a_is_dense=dense))
        assert torch.equal(*got)
        weights = A if dense else sp.prune(A)
        for r in (0, 128, 256, M - 128):                    # both m-blocks of the first tile, the last rows
            want = weights[r:r + 128].double() @ (x.double() if b_rows else x.double().t()) + beta * C[r:r + 128].double()
            # FP32 sums of K products (TF32 operands: 10 bits, rounded by 2^-11 each): well below 1 % of the norm
            err = (got[0][r:r + 128].double() - want).norm() / want.norm()
            assert err <= (0 if kind == "i8" else 2e-3)
    assert sp.gemm_status(device="cuda") == 0
