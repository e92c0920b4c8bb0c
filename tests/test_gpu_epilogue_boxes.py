"""Every form of the result at the edges of the epilogue's boxes: 16 rows or columns left of a box, tiles with fewer
boxes than there are warps for them, more boxes with C than are fetched ahead.  Operands and C are small whole numbers
(sums of at most 32 kept products of up to 4, plus 1.5 * 4, stay below 256), so that every result is exact in every
type and equal to the product in 64 bits."""
import pytest
import torch

pytestmark = pytest.mark.gpu

TORCH = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32, "i32": torch.int32, "i8": torch.int8,
         "e4m3": torch.float8_e4m3fn, "e5m2": torch.float8_e5m2, "tf32": torch.float32}
SHAPES = [(16, 16), (48, 80), (144, 464), (592, 48), (800, 240)]


@pytest.fixture(scope="module")
def sp():
    from paper_2104_08378_b200 import binding
    return binding


@pytest.mark.parametrize("tile", ["1x128x1", "1x128x3", "2x224x1", "2x224x2", "2x256x1"])
@pytest.mark.parametrize("kind,cd", [("bf16", "bf16"), ("f16", "f32"), ("tf32", "f32"), ("e4m3", "f16"), ("i8", "i32")])
def test_exact_results(sp, force_tile, kind, cd, tile):
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    unit = 32 if kind in ("e4m3", "i8") else 16
    K, ab = 64, "f32" if kind == "tf32" else kind

    def whole(rows, cols, limit, dt):
        return torch.randint(-limit, limit + 1, (rows, cols), device="cuda", generator=g).float().to(TORCH[dt])

    force_tile(tile)
    for M, N in SHAPES:
        M, N = (M + unit - 1) // unit * unit, (N + unit - 1) // unit * unit
        A, x = sp.prune(whole(M, K, 2, kind)), whole(N, K, 2, kind)
        vals, meta, _ = sp.compress(A)
        C = (2 * whole(M, N, 2, "f32")).to(TORCH[cd])
        product = A.double() @ x.double().t()
        for beta in (0, 1 if kind == "i8" else -1.5):
            want = (product + beta * C.double()).to(TORCH[cd])
            for cols in (False, True):
                c = C.t().contiguous() if cols else C.clone()
                out = torch.full((N, M) if cols else (M, N), 99, device="cuda").to(TORCH[cd])
                kw = dict(beta=beta, cd=cd, ab=ab, cd_col_major=cols)
                sp.gemm(vals, meta, x, C=c if beta else None, out=out, **kw)
                assert torch.equal(out.t() if cols else out, want)
                if beta:   # C and D may be the same buffer
                    sp.gemm(vals, meta, x, C=c, out=c, **kw)
                    assert torch.equal(c.t() if cols else c, want)
    assert sp.gemm_status(device="cuda") == 0
