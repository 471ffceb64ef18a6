"""Decode tilings that deal out the rows left after whole rounds by row groups: every tiling against the oracle, bit for bit,
where the last tile of a block holds one to four row groups, fewer than the block has warps for, or none."""
import pytest

from paper_2609_25624_b200 import binding as B
from paper_2609_25624_b200 import inputs
from tests.gpu_util import KERNEL_DECODE, assert_bits_equal, decode_tilings, oracle_y, run_gpu


# rows beyond one and two rounds of 148 x 56 (16-row tilings), batches that fill one, part of one and several batch blocks
@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K", [(16, 8288, 264), (16, 8289, 264), (13, 10001, 128), (9, 16600, 8), (33, 12500, 136), (16, 17000, 520)])
def test_rest_of_the_rows(M, N, K):
    every_tiling(M, N, K, "bf16")


# the same in the other formats: FP32 weights in segments on both sides of the length from which the loop loads a chunk ahead, whose
# warps without rows keep the ring in step by themselves
@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,wfmt", [(16, 8289, 264, "fp32"), (16, 8289, 264, "fp16"), (13, 10001, 132, "fp32"), (33, 12500, 136, "fp16"),
                                        (33, 12500, 136, "fp32"), (16, 8289, 1284, "fp32"), (13, 17000, 900, "fp32"), (33, 12500, 1540, "fp32")])
def test_rest_of_the_rows_in_other_formats(M, N, K, wfmt):
    every_tiling(M, N, K, wfmt)


# tiles of 112 rows: rests of one to eight row groups after one and two whole rounds, one to three batch blocks
@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,wfmt", [(8, 16577, 520, "bf16"), (5, 18001, 264, "fp16"), (8, 33500, 264, "bf16"), (16, 8300, 264, "fp16"), (20, 11100, 136, "bf16")])
def test_rest_of_112_row_tiles(M, N, K, wfmt):
    every_tiling(M, N, K, wfmt)


def every_tiling(M, N, K, wfmt):
    x, W, b = inputs.make_case_w(M, N, K, wfmt)
    want = oracle_y(x, W, b)
    for variant in range(decode_tilings(M, N, K, wfmt) + 1):
        assert_bits_equal(run_gpu(x, W, b, kernel=KERNEL_DECODE, variant=variant), want, f"variant {variant}")
    assert_bits_equal(run_gpu(x, W, b, max_blocks=7), want, "seven blocks")


# one wave of at most a block an SM: small blocks
@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,wfmt", [(12, 99, 5832, "bf16"), (42, 89, 4416, "fp16"), (24, 246, 6112, "bf16"), (35, 205, 5744, "bf16"), (17, 59, 2704, "fp16")])
def test_tilings_of_few_units(M, N, K, wfmt):
    plan = B.det_linear_plan_w(M, N, K, wfmt)
    t = B.det_linear_plan_describe(plan)["decode_tiling"]
    plan.close()
    assert (t["mt"], t["wm"], t["wr"], t["sk"]) == (4, 2, 1, 2)
