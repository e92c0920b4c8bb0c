"""The products of test_gpu_split_k_blocks.py share their k-blocks among the CTAs that it names, and floating-point ones never do."""
import pytest

import tile_choice
from test_gpu_split_k_blocks import SHAPES

I8, BF16, F16, F32, I32, E4M3 = 2, 1, 0, 3, 4, 5


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    return tile_choice.compile_harness(tmp_path_factory.mktemp("split_choice"))


@pytest.fixture(scope="module", autouse=True)
def parts_for_columns():
    """The harness's last figure: the logarithm of the CTAs of a tile instead of the k-blocks of a stage."""
    old = tile_choice.HARNESS
    tile_choice.HARNESS = old.replace("t.tile_n, k);", "t.tile_n, (void(k), t.split_log));")
    assert tile_choice.HARNESS != old
    yield
    tile_choice.HARNESS = old


def test_the_gpu_tests_run_every_number_of_parts(exe):
    forms = [(cd, cols, c) for cd, c in ((I32, 0), (I32, 1), (BF16, 0)) for cols in (0, 1)]
    for M, N, K, parts in SHAPES:
        got = tile_choice.choices(exe, [(I8, I32, M, N, K, 0, 0, cols, c) for cd, cols, c in forms if cd == I32])
        assert {1 << log for _, _, log in got} == {parts}, (M, N, K, got)
    assert {parts for *_, parts in SHAPES} == {2, 4, 8}


def test_floating_point_dense_and_row_major_operands_keep_one_part(exe):
    M, N, K, _ = SHAPES[0]
    got = tile_choice.choices(exe, [(ab, cd, M, N, K, 0, 0, 1, 0) for ab, cd in ((BF16, BF16), (F16, F32), (F32, F32), (E4M3, BF16))] +
                              [(I8, I32, M, N, K, 1, 0, 0, 0), (I8, I32, M, N, K, 0, 1, 0, 0)])
    assert {log for _, _, log in got} == {0}
