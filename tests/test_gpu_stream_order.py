"""Launches that start before the kernel ahead of them has ended still see all that it wrote, and overwrite nothing
that it still reads: chains of dependent calls give the bits of the same calls with a wait after each."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    from paper_2104_08378_b200 import binding
    return binding


def _chain(sp, w, x, steps, wait):
    """Buffers are reused from step to step, so each call reads what the one before wrote and overwrites what the one
    before that read; torch's own kernels (scaling, casts) stand between some of them."""
    pruned, vals = torch.empty_like(w), torch.empty_like(w[:, : w.shape[1] // 2]).contiguous()
    meta = torch.empty(sp.meta_bytes("bf16", *w.shape), dtype=torch.uint8, device="cuda")
    w, x, out = w.clone(), x.clone(), torch.empty((x.shape[0], w.shape[0]), dtype=x.dtype, device="cuda")
    sync = torch.cuda.synchronize if wait else (lambda: None)
    for i in range(steps):
        sp.prune_compress(w, pruned=pruned, vals=vals, meta=meta)
        sync()
        sp.gemm(vals, meta, x, out=out, cd_col_major=True)
        sync()       # x' = W x, scaled back to about 1
        torch.div(out, 2.0, out=x)
        sync()
        sp.apply_mask(w, meta, out=w)
        sync()
        sp.prune(w, out=w)
        sync()
        sp.gemm(vals, meta, x, out=out, cd_col_major=True)
        sync()
        sp.gemm(vals, meta, out, out=x, cd_col_major=True)
        sync()
        x.clamp_(-2, 2)
        sync()
        w.add_(w.roll(1, 1), alpha=0.25)
        sync()
    return [w, pruned, vals, meta, x, out]


@pytest.mark.parametrize("size", [256, 512, 2048])
@pytest.mark.parametrize("graph", [False, True])
def test_chained_calls_keep_stream_order(sp, size, graph):
    g = torch.Generator(device="cuda")
    g.manual_seed(size)
    w = (torch.randn((size, size), device="cuda", generator=g) / (0.85 * size) ** 0.5).bfloat16()
    x = torch.randn((size, size), device="cuda", generator=g).bfloat16()
    want = _chain(sp, w, x, 6, True)
    if graph:
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            _chain(sp, w, x, 1, True)                                    # the stream's workspace
            gr = torch.cuda.CUDAGraph()
            torch.cuda.synchronize()
            with torch.cuda.graph(gr, stream=s, capture_error_mode="thread_local"):
                got = _chain(sp, w, x, 6, False)
            gr.replay()
            gr.replay()
        torch.cuda.synchronize()
    else:
        for _ in range(3):
            got = _chain(sp, w, x, 6, False)
        torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
    assert sp.gemm_status(device=w.device) == 0


def _mixed(sp, w, x, side, steps, wait):
    """Copies, fills and work of a second stream (joined by events) between calls that start early."""
    meta = torch.empty(sp.meta_bytes("bf16", *w.shape), dtype=torch.uint8, device="cuda")
    vals, masked = torch.empty_like(w[:, : w.shape[1] // 2]).contiguous(), torch.empty_like(w)
    w, x, out = w.clone(), x.clone(), torch.empty((x.shape[0], w.shape[0]), dtype=x.dtype, device="cuda")
    main = torch.cuda.current_stream()
    sync = torch.cuda.synchronize if wait else (lambda: None)
    for i in range(steps):
        sp.compress_into(w, vals, meta)
        sync()
        sp.apply_mask(w, meta, out=masked)
        sync()
        w.copy_(masked)                            # device-to-device copy behind a call, and a call behind it
        sync()
        sp.gemm(vals, meta, x, out=out, cd_col_major=True)
        sync()
        side.wait_stream(main)
        with torch.cuda.stream(side):              # the other stream rewrites what the last call read
            x.copy_(out)
            x.mul_(0.5)
            out.zero_()
        main.wait_stream(side)
        sync()
        sp.gemm(vals, meta, x, beta=1.0, C=out, out=out, cd_col_major=True)
        sync()
        vals.zero_()                               # a fill of what it read
        sync()
        sp.prune(w, out=w)
        sync()
        x.copy_(out)
        x.clamp_(-2, 2)
        w.add_(w.roll(1, 1), alpha=0.25)
        sync()
    return [w, vals, meta, x, out, masked]


@pytest.mark.parametrize("size", [256, 1024])
@pytest.mark.parametrize("graph", [False, True])
def test_copies_fills_and_other_streams_keep_order(sp, size, graph):
    g = torch.Generator(device="cuda")
    g.manual_seed(size)
    w = (torch.randn((size, size), device="cuda", generator=g) / (0.85 * size) ** 0.5).bfloat16()
    x = torch.randn((size, size), device="cuda", generator=g).bfloat16()
    s, side = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        want = _mixed(sp, w, x, side, 5, True)
        if graph:
            gr = torch.cuda.CUDAGraph()
            torch.cuda.synchronize()
            with torch.cuda.graph(gr, stream=s, capture_error_mode="thread_local"):
                got = _mixed(sp, w, x, side, 5, False)
            gr.replay()
            gr.replay()
        else:
            for _ in range(3):
                got = _mixed(sp, w, x, side, 5, False)
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
    assert sp.gemm_status(device=w.device) == 0
