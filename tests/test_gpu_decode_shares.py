"""Decode tilings that deal out the rows left after whole rounds by row groups: every tiling against the oracle, bit for bit,
where the last tile of a block holds one to four row groups, fewer than the block has warps for, or none."""
import pytest

from paper_2609_25624_b200 import binding as B
from paper_2609_25624_b200 import inputs
from tests.gpu_util import KERNEL_DECODE, assert_bits_equal, oracle_y, run_gpu


# rows beyond one and two rounds of 148 x 56 (16-row tilings), batches that fill one, part of one and several batch blocks
@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K", [(16, 8288, 264), (16, 8289, 264), (13, 10001, 128), (9, 16600, 8), (33, 12500, 136), (16, 17000, 520)])
def test_rest_of_the_rows(M, N, K):
    x, W, b = inputs.make_case(M, N, K)
    want = oracle_y(x, W, b)
    for variant in range(0, 24):
        try:
            got = run_gpu(x, W, b, kernel=KERNEL_DECODE, variant=variant)
        except B.DetLinearError:
            break
        assert_bits_equal(got, want, f"variant {variant}")
    assert variant > 2
    assert_bits_equal(run_gpu(x, W, b, max_blocks=7), want, "seven blocks")
