"""The products of test_gpu_split_k_blocks.py share their k-blocks among the CTAs that it names, in tiles of as many columns,
floating-point ones never do, and the device is asked for its clusters as it should be."""
import pytest

import tile_choice
from test_gpu_split_k_blocks import EXPIRED_WAIT, SHAPES

I8, BF16, F16, F32, I32, E4M3 = 2, 1, 0, 3, 4, 5


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    return tile_choice.compile_harness(tmp_path_factory.mktemp("split_choice"))


def test_the_gpu_tests_run_every_number_of_parts_and_columns(exe):
    """In every form of the result that they run."""
    forms = [(cd, cols, c) for cd, c in ((I32, 0), (I32, 1), (BF16, 0), (F16, 0), (F32, 0), (I8, 0)) for cols in (0, 1)]
    for M, N, K, parts, columns in SHAPES + [EXPIRED_WAIT]:
        got = tile_choice.details(exe, [(I8, cd, M, N, K, 0, 0, cols, c) for cd, cols, c in forms])
        assert {(c.parts, c.columns) for c in got} == {(parts, columns)}, (M, N, K, got)
    # (all that came out of 6000 random products)
    assert {(parts, columns) for *_, parts, columns in SHAPES} == {(8, 32), (4, 32), (4, 64), (4, 96), (2, 32), (2, 64), (2, 96), (2, 128)}


def test_the_gpu_test_of_twelve_warps_runs_them(exe):
    from test_gpu_twelve_warps import SHAPES as shapes
    for M, N, K in shapes:
        for cd in (I8, BF16):
            got = tile_choice.details(exe, [(I8, cd, M, N, K, 0, 0, cols, 0) for cols in (0, 1)])
            assert {c.warps for c in got} == {12 if cd == I8 and K <= 6 * 256 else 8}, (M, N, K, got)
    assert {K <= 6 * 256 for _, _, K in shapes} == {False, True}


def test_floating_point_dense_and_row_major_operands_keep_one_part(exe):
    M, N, K, *_ = SHAPES[0]
    got = tile_choice.details(exe, [(ab, cd, M, N, K, 0, 0, 1, 0) for ab, cd in ((BF16, BF16), (F16, F32), (F32, F32), (E4M3, BF16))] +
                              [(I8, I32, M, N, K, 1, 0, 0, 0), (I8, I32, M, N, K, 0, 1, 0, 0)])
    assert {c.parts for c in got} == {1}


def test_a_device_that_holds_no_cluster_is_given_none(exe):
    got = tile_choice.details(exe, [(I8, I32, M, N, K, 0, 0, 0, 0) for M, N, K, *_ in SHAPES], NO_CLUSTERS=1)
    assert {c.parts for c in got} == {1}


def test_a_question_that_fails_is_asked_again(exe):
    M, N, K, parts, _ = SHAPES[0]
    got = tile_choice.details(exe, [(I8, I32, M, N, K, 0, 0, 0, 0)] * 12, FAILING_QUERIES=9)
    assert got[0].parts == 1 and got[-1].parts == parts, got
    assert got[-1].queries == 0, got        # and an answer is kept


def test_the_first_int8_product_asks_whatever_it_splits(exe):
    """So that none of it is left to a stream capture that follows."""
    M, N, K, parts, _ = SHAPES[0]
    first = [(64, 64, 512), (3072, 4096, 768), (8192, 8192, 8192)]
    for shape in first:
        got = tile_choice.details(exe, [(I8, I32, *shape, 0, 0, 0, 0), (I8, I32, M, N, K, 0, 0, 0, 0)])
        assert [(c.parts, c.queries) for c in got] == [(1, 3), (parts, 0)], (shape, got)
