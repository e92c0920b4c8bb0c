"""The native form of the binding's calls against the Python form of the same call (the native one replaced by one that
declines everything): results, their types, shapes and strides, refused calls, and arguments the native form must decline."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    from paper_2104_08378_b200 import binding
    return binding


@pytest.fixture
def both(sp, monkeypatch):
    """both(call): what the call gives natively and in Python, each a tuple of tensors or an error."""
    class Declines:
        gemm = gemm_i8_dequant = conv3x3_nhwc = compress = apply_mask = staticmethod(lambda *args: None)

    def outcome(call):
        try:
            got = call()
            return tuple(got) if isinstance(got, (tuple, list)) else (got,)
        except Exception as e:  # noqa: BLE001
            return type(e), getattr(e, "status", None)

    def run(call):
        native = outcome(call)
        with monkeypatch.context() as m:
            m.setattr(sp, "_native", Declines)
            python = outcome(call)
        assert len(native) == len(python)
        for a, b in zip(native, python):
            if isinstance(a, torch.Tensor):
                assert a.dtype == b.dtype and a.shape == b.shape and a.stride() == b.stride() and a.device == b.device
                assert torch.equal(a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8))
            else:
                assert a == b
        return native
    return run


def test_products(sp, both):
    g = torch.Generator(device="cuda").manual_seed(1)
    for kind, dt in (("bf16", torch.bfloat16), ("f16", torch.float16), ("f32", torch.float32), ("e4m3", torch.float8_e4m3fn),
                     ("i8", torch.int8)):
        def rand(*shape):
            return (torch.randn(shape, device="cuda", generator=g) * 3).to(dt)
        M, N, K = 96, 64, 128
        w, x, xr = rand(M, K), rand(N, K + 32)[:, :K], rand(K, N)
        vals, meta, _ = both(lambda: sp.compress(w))
        both(lambda: sp.compress(w, layout=sp.META_CANONICAL))
        both(lambda: sp.compress(w[:, : K - 6]))                                      # refused
        both(lambda: sp.apply_mask(w, meta, out=w.clone())) if kind != "f32" else None
        for cols in (False, True):
            C = torch.ones((N, M) if cols else (M, N), device="cuda").to(sp.TORCH_DTYPE["i32" if kind == "i8" else "bf16" if kind == "e4m3" else kind])
            wide = torch.zeros((C.shape[0], C.shape[1] + 16), device="cuda").to(C.dtype)[:, :C.shape[1]]
            both(lambda: sp.gemm(vals, meta, x, cd_col_major=cols))
            both(lambda: sp.gemm(vals, meta, xr, b_row_major=True, beta=1.0, C=C, cd_col_major=cols))
            both(lambda: sp.gemm(vals, meta, x, beta=1, C=C, out=wide, cd_col_major=cols))
            both(lambda: sp.gemm(sp.prune(w), None, x, a_is_dense=True, alpha=1 if kind == "i8" else 0.5, cd_col_major=cols))
        both(lambda: sp.gemm(vals, meta, x[:, : K // 2]))                             # K does not match
        both(lambda: sp.gemm(vals, None, x))                                          # no metadata
        both(lambda: sp.gemm(vals, meta, x, beta=1.0))                                # no C
        both(lambda: sp.gemm(vals, meta, x, cd="none"))
        both(lambda: sp.gemm(vals[:0], meta, x))
        both(lambda: sp.gemm(vals, meta, x[:0]))
        both(lambda: sp.gemm(vals[:, ::2], meta, x))
        if kind == "i8":
            scale = torch.full((M,), 0.01, device="cuda")
            for cd in ("i8", "bf16", "f32"):
                both(lambda: sp.gemm_i8_dequant(vals, meta, x, scale, bias=scale, relu=True, out_scale=0.5, cd=cd))
                both(lambda: sp.gemm_i8_dequant(vals, meta, x, scale, cd=cd, cd_col_major=True, out_scale=1))
            both(lambda: sp.gemm_i8_dequant(vals, meta, x, scale, out_scale=0.0, cd="i8"))
            both(lambda: sp.gemm(vals, meta, x, alpha=2))
    w = torch.randn((64, 9 * 128), device="cuda", generator=g).half()
    vals, meta, _ = sp.compress(w)
    x = torch.randn((8, 8, 16, 128), device="cuda", generator=g).half()
    for nhwc in (False, True):
        both(lambda: sp.conv3x3_nhwc(vals, meta, x, nhwc_out=nhwc))
        both(lambda: sp.conv3x3_nhwc(vals, meta, x, nhwc_out=nhwc, cd="f32", alpha=0.5))
    both(lambda: sp.conv3x3_nhwc(vals, meta, x[..., :64]))                           # refused


def test_streams_modes_and_wrappers(sp, both):
    """The current stream and its workspace are used; a subclass, a functorch wrapper and a torch-function mode are declined."""
    w, x = torch.randn((64, 128), device="cuda").half(), torch.randn((32, 128), device="cuda").half()
    vals, meta, _ = sp.compress(w)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        stream.wait_stream(torch.cuda.default_stream())
        both(lambda: sp.gemm(vals, meta, x))
        stream.synchronize()
    assert (x.device.index, stream.cuda_stream) in sp._workspaces

    class Sub(torch.Tensor):
        pass

    class Mode(torch.overrides.TorchFunctionMode):
        def __torch_function__(self, func, types, args=(), kwargs=None):
            return func(*args, **(kwargs or {}))

    def args(a, b):
        return sp._GEMM, sp._workspaces, a, meta, b, 1.0, 0.0, None, None, None, False, None, False, False
    assert sp._native.gemm(*args(vals, x)) is not None
    assert sp._native.gemm(*args(vals.as_subclass(Sub), x)) is None
    assert sp._native.gemm(*args(vals.cpu(), x)) is None and sp._native.gemm(*args(vals, x.cpu())) is None
    with Mode():
        assert sp._native.gemm(*args(vals, x)) is None
    seen = []
    torch.vmap(lambda t: (seen.append(sp._native.gemm(*args(vals, t))), t)[1])(torch.stack([x, x]))
    assert seen == [None]
