"""Tall tiles (at most 128 columns, two or three m-blocks that share each B box): their results are, bit for bit, those
of 128 x 128 tiles (same K order, same instructions per row), which other tests compare with the oracle."""
import pytest
import torch

pytestmark = pytest.mark.gpu

OUT = {"bf16": "bf16", "f16": "f16", "i8": "i32", "tf32": "f32", "e4m3": "bf16", "e5m2": "f32"}
TORCH = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32, "i32": torch.int32}


@pytest.fixture(scope="module")
def sp():
    from paper_2104_08378_b200 import binding
    return binding


def _matrix(kind, rows, cols, g, pad=0):
    if kind == "i8":
        return torch.randint(-128, 128, (rows, cols + pad), dtype=torch.int8, device="cuda", generator=g)[:, :cols]
    dt = {"bf16": torch.bfloat16, "f16": torch.float16, "tf32": torch.float32, "f32": torch.float32,
          "e4m3": torch.float8_e4m3fn, "e5m2": torch.float8_e5m2}[kind]
    return torch.randn((rows, cols + pad), device="cuda", generator=g).to(dt)[:, :cols]


# rows: less than one m-block, tiles with one, two or three m-blocks left, a last m-block of 16 or 32 rows, the smallest
# and largest M with two and three m-blocks, two rounds of tiles (M > 148 * 384)
@pytest.mark.parametrize("kind", ["bf16", "f16", "i8", "tf32", "e4m3"])
@pytest.mark.parametrize("M", [16, 160, 400, 18944, 18976, 37888, 37920, 49152, 60000])
def test_same_bits_as_square_tiles(sp, force_tile, kind, M):
    if kind in ("i8", "e4m3"):
        M = max(32, M // 32 * 32)
    g = torch.Generator(device="cuda")
    g.manual_seed(M)
    cd = OUT[kind]
    for N, K, pad in ((32, 288, 0), (96, 1088, 32), (128, 512, 0)) + (((16, 272, 16),) if kind not in ("i8", "e4m3") else ()):
        vals, meta, _ = sp.compress(_matrix(kind, M, K, g, pad))
        x = _matrix(kind, N, K, g, pad)
        C = _matrix({"i8": "i8", "tf32": "tf32"}.get(kind, cd), M, N, g).to(TORCH[cd]).contiguous()
        for order in (False, True):
            beta = 1 if kind == "i8" else -1.5
            for c, b in ((None, 0), (C.t().contiguous() if order else C, beta)):
                got = []
                for tile in ("1x128x1", "1x128x2", "1x128x3"):
                    force_tile(tile)
                    out = torch.full((N, M + 32) if order else (M, N + 32), 7, device="cuda").to(TORCH[cd])
                    sp.gemm(vals, meta, x, beta=b, C=c, cd=cd, out=out[:, : M if order else N], cd_col_major=order)
                    got.append(out)
                assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])
        desc = sp.make_desc("f32" if kind == "tf32" else kind, cd, M, N, K, K // 2, K, N, N)
        force_tile(None)
        blocks = (M + 127) // 128          # on the 148 SMs of the device
        assert sp.gemm_plan(desc) == ("1x128x1" if blocks <= 148 else "1x128x2" if blocks <= 296 or blocks > 444 else "1x128x3")
    assert sp.gemm_status(device=x.device) == 0


@pytest.mark.parametrize("cd", ["i8", "bf16", "f32"])
def test_dequantising_form(sp, force_tile, cd):
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    for M, N, K in ((32, 32, 64), (416, 96, 512), (26048, 64, 320), (37920, 128, 288)):
        vals, meta, _ = sp.compress(_matrix("i8", M, K, g))
        x = _matrix("i8", N, K, g)
        scale, bias = torch.rand(M, device="cuda", generator=g) * 0.01, torch.randn(M, device="cuda", generator=g)
        for order in (False, True):
            got = []
            for tile in ("1x128x1", "1x128x2", "1x128x3"):
                force_tile(tile)
                got.append(sp.gemm_i8_dequant(vals, meta, x, scale, bias=bias, relu=True, out_scale=0.1, cd=cd,
                                              cd_col_major=order))
            assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])


def test_expired_wait_is_reported(sp, force_tile):
    """The bounded waits of the tall tiles' own roles: one slot is left out, every role gives up and returns, and the
    next launch is good again."""
    g = torch.Generator(device="cuda")
    g.manual_seed(6)
    vals, meta, _ = sp.compress(_matrix("bf16", 1184, 1024, g))
    x = _matrix("bf16", 96, 1024, g)
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    force_tile("1x128x3")
    good = sp.gemm(vals, meta, x, ws=ws)
    try:
        sp.set_fault_hooks(20000000, True)             # about 10 ms of SM clock per wait
        sp.gemm(vals, meta, x, ws=ws)
        torch.cuda.synchronize()
    finally:
        sp.set_fault_hooks(0, False)
    again = sp.gemm(vals, meta, x, ws=ws)
    assert torch.equal(again, good)
    assert sp.gemm_status(ws) == 9 and sp.gemm_status(ws) == 0


@pytest.mark.parametrize("kind,cd,order,M,N,K,plan", [
    # wide outputs: pairs of CTAs, whose epilogue overlaps (on the 148 SMs of the device)
    ("bf16", "f32", True, 49152, 128, 512, "2x224x1"), ("bf16", "f32", False, 98304, 128, 1024, "2x224x1"),
    ("i8", "i32", False, 98304, 128, 1024, "2x224x1"), ("f32", "f32", True, 60000, 96, 512, "2x224x1"),
    # a long K and a last round that leaves SMs idle
    ("bf16", "bf16", False, 60000, 128, 12288, "2x224x2"), ("e4m3", "bf16", True, 60000, 96, 12288, "2x224x2"),
    # narrow outputs: tall tiles
    ("bf16", "bf16", True, 49152, 32, 12288, "1x128x3"), ("bf16", "bf16", True, 49152, 128, 12288, "1x128x3"),
    ("e4m3", "bf16", True, 37888, 128, 4096, "1x128x2"), ("bf16", "f32", True, 49152, 64, 512, "1x128x3"),
    ("i8", "i32", False, 37888, 96, 1024, "1x128x2"), ("bf16", "bf16", True, 98304, 96, 4096, "1x128x3")])
def test_tall_tiles_only_where_the_output_is_narrow(sp, kind, cd, order, M, N, K, plan):
    out = M if order else N
    assert sp.gemm_plan(sp.make_desc(kind, cd, M, N, K, K // 2, K, out, out, False, False, order)) == plan


@pytest.mark.parametrize("kind,cd,acc_f16", [("f16", "f16", True), ("f16", "f32", True), ("e5m2", "f32", False),
                                             ("e5m2", "bf16", False), ("e4m3", "f16", False)])
def test_other_kinds_and_paddings(sp, force_tile, kind, cd, acc_f16):
    """FP16 accumulation and both 8-bit floats; the columns between the result and its leading dimension keep their fill."""
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    for M, N, K in ((32, 32, 288), (416, 96, 1088), (37920, 128, 320)):
        vals, meta, _ = sp.compress(_matrix(kind, M, K, g))
        x, C = _matrix(kind, N, K, g), _matrix(cd, M, N, g)
        for order in (False, True):
            for beta in (0.0, -1.5):
                got = []
                for tile in ("1x128x1", "1x128x2", "1x128x3"):
                    force_tile(tile)
                    out = torch.full((N, M + 32) if order else (M, N + 32), 7, device="cuda").to(TORCH[cd])
                    width = M if order else N
                    sp.gemm(vals, meta, x, beta=beta, C=(C.t().contiguous() if order else C) if beta else None, cd=cd,
                            out=out[:, :width], cd_col_major=order, acc_f16=acc_f16)
                    assert (out[:, width:] == 7).all() and (out[:, :width] != 7).any()
                    got.append(out)
                assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])
    assert sp.gemm_status(device=x.device) == 0


def test_convolutions_take_no_tall_tiles(sp, force_tile):
    """They have no im2col view of B: a forced one is refused, and the automatic choice, with more 128-row blocks than
    SMs and 128 output pixels, is the product with the unfolded activation."""
    g = torch.Generator(device="cuda")
    g.manual_seed(8)
    M, Cin = 19200, 512
    vals, meta, _ = sp.compress(_matrix("f16", M, 9 * Cin, g))
    x = _matrix("f16", 128, Cin, g).view(1, 8, 16, Cin)
    for tile in ("1x128x2", "1x128x3"):
        force_tile(tile)
        with pytest.raises(sp.Sp24Error) as refused:
            sp.conv3x3_nhwc(vals, meta, x)
        assert refused.value.status == 6           # not built
    force_tile(None)
    got = sp.conv3x3_nhwc(vals, meta, x)
    want = sp.gemm(vals, meta, sp.im2col_nhwc_3x3(x))
    assert torch.equal(got, want) and sp.gemm_status(device=x.device) == 0
