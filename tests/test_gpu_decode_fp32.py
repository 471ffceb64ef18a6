"""Decode with FP32 weights: every tiling, at the sizes where the multiply loop that loads a chunk ahead can go wrong -- a last chunk
that is partly outside, one chunk only, one more than a ring of stages holds, segments of unequal length, several batch blocks."""
import pytest

from paper_2609_25624_b200 import binding as B
from paper_2609_25624_b200 import inputs
from tests.gpu_util import KERNEL_DECODE, assert_bits_equal, oracle_y, run_gpu


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K", [(3, 61, 128), (4, 85, 132), (5, 30, 260), (8, 113, 1156), (13, 57, 1028), (16, 225, 900), (33, 90, 516), (64, 29, 2048)])
def test_every_tiling(M, N, K):
    x, W, b = inputs.make_case_w(M, N, K, "fp32")
    want = oracle_y(x, W, b)
    for variant in range(0, 24):
        try:
            got = run_gpu(x, W, b, kernel=KERNEL_DECODE, variant=variant)
        except B.DetLinearError:
            break
        assert_bits_equal(got, want, f"variant {variant}")
    assert variant > 2
