"""Decode with FP32 weights: every tiling, at the sizes where the multiply loop that loads a chunk ahead can go wrong -- a last chunk
that is partly outside, one more than a ring of stages holds, segments of unequal length, several batch blocks --, and where shorter
segments take the other loop."""
import pytest

from paper_2609_25624_b200 import binding as B
from paper_2609_25624_b200 import inputs
from tests.gpu_util import KERNEL_DECODE, assert_bits_equal, decode_tilings, oracle_y, run_gpu


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K", [(3, 61, 128), (4, 85, 132), (5, 30, 260), (8, 113, 1156), (13, 57, 1028), (16, 225, 900), (33, 90, 516), (64, 29, 2048),
                                   (3, 61, 4100), (8, 113, 1540), (13, 57, 1284), (16, 225, 2564), (33, 90, 1156), (12, 16400, 772), (20, 16400, 264)])
def test_every_tiling(M, N, K):
    x, W, b = inputs.make_case_w(M, N, K, "fp32")
    want = oracle_y(x, W, b)
    for variant in range(decode_tilings(M, N, K, "fp32") + 1):
        assert_bits_equal(run_gpu(x, W, b, kernel=KERNEL_DECODE, variant=variant), want, f"variant {variant}")


# short segments: tilings by the rates of the loop that does not load ahead; one wave of at most a block an SM: small blocks
@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,tiling", [(16, 75, 176, (4, 2, 2, 1)), (39, 81, 176, (4, 2, 2, 1)), (4, 97, 8552, (2, 2, 1, 2)), (3, 953, 8928, (2, 2, 1, 2))])
def test_tilings_of_short_segments_and_few_units(M, N, K, tiling):
    plan = B.det_linear_plan_w(M, N, K, "fp32")
    t = B.det_linear_plan_describe(plan)["decode_tiling"]
    plan.close()
    assert (t["mt"], t["wm"], t["wr"], t["sk"]) == tiling
