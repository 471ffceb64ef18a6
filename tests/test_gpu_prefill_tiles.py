"""The TMA-fed prefill kernel's schedules against the oracle, bit for bit: every tile height and width, units dealt out in
equal stretches (accumulators handed from block to block) and one block per unit, segments folded in place."""
import pytest
import torch

from paper_2609_25624_b200 import binding as B
from paper_2609_25624_b200 import inputs
from tests.gpu_util import KERNEL_PREFILL, assert_bits_equal, oracle_y, run_gpu

pytestmark = pytest.mark.gpu

WIDTHS = {2: 256, 3: 128, 4: 64, 5: 32}

# one row or column past a tile edge, a partial last slab, one segment and several
SHAPES = [(129, 257, 136, "bf16"), (81, 33, 520, "fp16"), (113, 65, 1292, "fp32"), (97, 129, 776, "bf16"), (65, 31, 40, "fp32")]


@pytest.mark.parametrize("M,N,K,wfmt", SHAPES)
def test_every_tile_height_and_width(M, N, K, wfmt):
    x, W, b = inputs.make_case_w(M, N, K, wfmt)
    want = oracle_y(x, W, b)
    for width in WIDTHS:
        for tm in (5, 6, 7, 8):
            assert_bits_equal(run_gpu(x, W, b, kernel=KERNEL_PREFILL, variant=10 * width + tm), want,
                              f"tile {16 * tm} x {WIDTHS[width]}")


# more units than SMs: each block takes a stretch that begins and ends inside units
@pytest.mark.parametrize("M,N,K,wfmt", [(400, 8200, 264, "bf16"), (300, 3000, 1000, "fp32"), (1000, 6000, 136, "fp16"), (520, 2570, 1032, "bf16")])
def test_units_cut_between_blocks(M, N, K, wfmt):
    x, W, b = inputs.make_case_w(M, N, K, wfmt)
    want = oracle_y(x, W, b)
    xd, Wd, bd = x.cuda(), W.cuda(), b.cuda()
    plan = B.det_linear_plan_w(M, N, K, wfmt)
    d = B.det_linear_plan_describe(plan)
    tile = d["prefill_tile"]
    assert -(-M // tile["bm"]) * -(-N // tile["bn"]) * d["S"] > 148
    for rep in range(3):                         # ticket, flags and tile counters are back at zero after every run
        y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
        B.det_linear_run(plan, xd, Wd, bd, y)
        B.det_linear_plan_check(plan)
        assert_bits_equal(y.cpu().numpy(), want, f"run {rep}")
    for variant in (28, 37, 46, 55):             # other tiles of the same plan
        B.det_test_plan_set_variant(plan, variant)
        y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
        B.det_linear_run(plan, xd, Wd, bd, y)
        B.det_linear_plan_check(plan)
        assert_bits_equal(y.cpu().numpy(), want, f"variant {variant}")
    plan.close()
