"""Small problems take narrower tiles than their shape's widest (more SMs, fewer columns each): their results are, bit for
bit, those of 128 x 128 tiles, which other tests compare with the oracle.  An element's sum runs over K in the same order
with the same instructions whatever the width, so that no tolerance is needed."""
import pytest
import torch

pytestmark = pytest.mark.gpu

TORCH = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32, "tf32": torch.float32, "i32": torch.int32,
         "e4m3": torch.float8_e4m3fn, "e5m2": torch.float8_e5m2}
# less than one block of rows, widths that leave 16 or 32 columns over, enough tiles for two rounds, a K of one and of two
# k-blocks ...
SHAPES = [(16, 16, 64), (160, 48, 288), (256, 256, 512), (320, 1104, 128), (512, 208, 1344), (1184, 736, 1008), (1024, 2080, 256),
          (2784, 1312, 272), (64, 96, 1408), (304, 64, 2304)]
# ... and those that, with them, take every width of single CTAs and of pairs in every kind and order of B, and, two k-blocks
# to a stage, an odd and an even number of them (test_tile_choice_cpu.py)
SHAPES += [(800, 704, 320), (320, 3744, 288), (448, 3616, 288), (2464, 960, 288), (1376, 2048, 288), (3744, 832, 288),
           (288, 3520, 1120), (3392, 1280, 288), (320, 1632, 1376), (2784, 1568, 288), (128, 32, 1152), (576, 3168, 320),
           (832, 768, 768), (3168, 192, 896), (2336, 2816, 288), (448, 1216, 832)]
KINDS = [("bf16", "bf16"), ("f16", "f32"), ("tf32", "f32"), ("e4m3", "bf16"), ("e5m2", "f32"), ("i8", "i32")]


def shapes(kind):
    unit = 32 if kind in ("e4m3", "e5m2", "i8") else 16
    return [tuple((v + unit - 1) // unit * unit for v in shape) for shape in SHAPES]


@pytest.fixture(scope="module")
def sp():
    from paper_2104_08378_b200 import binding
    return binding


def _matrix(kind, rows, cols, g, pad):
    if kind == "i8":
        return torch.randint(-128, 128, (rows, cols + pad), dtype=torch.int8, device="cuda", generator=g)[:, :cols]
    return torch.randn((rows, cols + pad), device="cuda", generator=g).to(TORCH[kind])[:, :cols]


@pytest.mark.parametrize("b_rows", [False, True])
@pytest.mark.parametrize("kind,cd", KINDS)
def test_same_bits_as_128_columns(sp, force_tile, kind, cd, b_rows):
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    for M, N, K in shapes(kind):
        for dense in (False, True):
            A, x = _matrix(kind, M, K, g, 0), _matrix(kind, *((K, N) if b_rows else (N, K)), g, 32)
            vals, meta = (A, None) if dense else sp.compress(A)[:2]
            C = _matrix("i8" if cd == "i32" else cd, M, N, g, 0).to(TORCH[cd]).contiguous()
            for cols in (False, True):
                for beta in (0, 1 if kind == "i8" else -1.5):
                    got = []
                    for tile in (None, "1x128x1"):
                        force_tile(tile)
                        out = torch.full((N, M + 32) if cols else (M, N + 32), 7, device="cuda").to(TORCH[cd])
                        sp.gemm(vals, meta, x, beta=beta, C=(C.t().contiguous() if cols else C) if beta else None, cd=cd,
                                ab="f32" if kind == "tf32" else kind, out=out[:, : M if cols else N], b_row_major=b_rows,
                                cd_col_major=cols, a_is_dense=dense)
                        got.append(out)
                    assert torch.equal(got[0], got[1]), (M, N, K, dense, cols, beta)
    assert sp.gemm_status(device="cuda") == 0


@pytest.mark.parametrize("cd", ["i8", "bf16", "f32"])
def test_dequantising_form(sp, force_tile, cd):
    g = torch.Generator(device="cuda")
    g.manual_seed(12)
    for M, N, K in ((32, 32, 64), (256, 256, 512), (1024, 1056, 320), (4096, 96, 4096)):
        vals, meta, _ = sp.compress(_matrix("i8", M, K, g, 0))
        x = _matrix("i8", N, K, g, 0)
        scale, bias = torch.rand(M, device="cuda", generator=g) * 0.01, torch.randn(M, device="cuda", generator=g)
        for cols in (False, True):
            got = []
            for tile in (None, "1x128x1"):
                force_tile(tile)
                got.append(sp.gemm_i8_dequant(vals, meta, x, scale, bias=bias, relu=True, out_scale=0.1, cd=cd, cd_col_major=cols))
            assert torch.equal(got[0], got[1]), (M, N, K, cols)


@pytest.mark.parametrize("kind", ["bf16", "i8"])
def test_convolution(sp, force_tile, kind):
    g = torch.Generator(device="cuda")
    g.manual_seed(13)
    for Nb, H, W, Cin, M in ((4, 14, 14, 256, 64), (16, 7, 7, 512, 256), (2, 9, 40, 256, 480)):
        w = _matrix(kind, M, 9 * Cin, g, 0)
        x = _matrix(kind, Nb * H * W // 32 * 32 if kind == "i8" else Nb * H * W, Cin, g, 0)
        if Nb * H * W % (32 if kind == "i8" else 16):
            continue
        vals, meta, _ = sp.compress(w)
        got = []
        for tile in (None, "1x128x1"):
            force_tile(tile)
            got.append(sp.conv3x3_nhwc(vals, meta, x.view(Nb, H, W, Cin), nhwc_out=True))
        assert torch.equal(got[0], got[1]), (Nb, H, W, Cin, M)
