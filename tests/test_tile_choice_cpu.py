"""The shapes of test_gpu_tile_widths.py run every width of tile, and both forms of a stage, that the choice can give: a change
of the rule that takes one away from them fails here."""
import pytest

import tile_choice
from test_gpu_tile_widths import KINDS, shapes

CODE = {"f16": 0, "bf16": 1, "i8": 2, "f32": 3, "tf32": 3, "i32": 4, "e4m3": 5, "e5m2": 6}
ATOM = {"f16": 64, "bf16": 64, "tf32": 32}      # elements of 128 bytes


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    return tile_choice.compile_harness(tmp_path_factory.mktemp("tile_choice"))


def _taken(exe, kind, cd, b_rows):
    """{(CTAs, columns, k-blocks of a stage, whether the k-blocks are odd)} over the shapes and forms the GPU test runs."""
    forms = [(M, N, K, cols, c) for M, N, K in shapes(kind) for cols in (0, 1) for c in (0, 1)]
    got = tile_choice.choices(exe, [(CODE[kind], CODE[cd], M, N, K, 0, b_rows, cols, c) for M, N, K, cols, c in forms])
    return {(int(tile[0]), columns, k, k == 2 and K // (2 * ATOM[kind]) % 2 == 1) for (tile, columns, k), (_, _, K, _, _) in
            zip(got, forms)}


@pytest.mark.parametrize("b_rows", [False, True])
@pytest.mark.parametrize("kind,cd", KINDS)
def test_every_width_is_run(exe, kind, cd, b_rows):
    taken = _taken(exe, kind, cd, b_rows)
    widths = {(ctas, columns) for ctas, columns, _, _ in taken}
    # (N-contiguous B comes in chunks of 128 bytes: narrower pairs are not chosen)
    pairs = range({"tf32": 64, "e4m3": 160, "e5m2": 160, "i8": 160}.get(kind, 96) if b_rows else 64, 225, 32)
    assert widths >= {(1, n) for n in (32, 64, 96, 128)} | {(2, n) for n in pairs}, sorted(widths)
    if not b_rows and kind in ATOM:
        assert taken >= {(ctas, columns, 2, odd) for ctas, columns in ((1, 32), (2, 64)) for odd in (False, True)}, sorted(taken)


def test_the_timeout_test_stalls_stages_of_two_k_blocks(exe):
    got = tile_choice.choices(exe, [(1, 1, M, N, 1024, 0, 0, 0, 0) for M, N in ((512, 448), (448, 1216))])
    assert got == [("1x128x1", 32, 2), ("2x224x1", 64, 2)]


def test_the_harness_agrees_with_the_plan(exe):
    """On the shapes whose plan does not depend on the number of SMs."""
    from paper_2104_08378_b200 import binding as sp
    got = tile_choice.choices(exe, [(1, 1, 49152, 8192, 12288, 0, 0, 0, 0), (0, 0, 256, 256, 512, 0, 0, 0, 0)])
    assert [tile for tile, _, _ in got] == ["2x224x2", "1x128x1"]
    assert sp.gemm_plan(sp.make_desc("bf16", "bf16", 49152, 8192, 12288, 6144, 12288, 8192, 8192)) == got[0][0]
