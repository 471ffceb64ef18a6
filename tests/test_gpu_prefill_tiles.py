"""The TMA-fed prefill kernel's schedules against the oracle, bit for bit: every tile height and width, units dealt out in
equal stretches (accumulators handed from block to block) and one block per unit, segments folded in place."""
import numpy as np
import pytest
import torch

from paper_2609_25624_b200 import binding as B
from paper_2609_25624_b200 import inputs
from tests.gpu_util import KERNEL_GENERIC, KERNEL_PREFILL, assert_bits_equal, oracle_y, run_gpu

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
    for variant in (28, 37, 46, 55, 58):             # other tiles of the same plan
        B.det_test_plan_set_variant(plan, variant)
        y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
        B.det_linear_run(plan, xd, Wd, bd, y)
        B.det_linear_plan_check(plan)
        assert_bits_equal(y.cpu().numpy(), want, f"variant {variant}")
    plan.close()


def run_plain(x, W, b, offset=0):
    """The kernel's plain-load feed, with W and x `offset` elements behind an allocation's start."""
    M, K = x.shape
    N = W.shape[0]
    wbuf = torch.full((N * K + offset,), float("nan"), dtype=W.dtype, device="cuda")
    xbuf = torch.full((M * K + offset,), float("nan"), dtype=torch.float32, device="cuda")
    wbuf[offset:] = W.cuda().flatten()
    xbuf[offset:] = x.cuda().flatten()
    plan = B.det_linear_plan_w(M, N, K, {torch.bfloat16: "bf16", torch.float16: "fp16", torch.float32: "fp32"}[W.dtype])
    B.det_test_plan_force_kernel(plan, KERNEL_GENERIC)
    out = []
    for _ in range(2):
        y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
        B.det_linear_run(plan, xbuf[offset:].view(M, K), wbuf[offset:].view(N, K), b.cuda(), y)
        B.det_linear_plan_check(plan)
        out.append(y.cpu().numpy())
    assert out[0].tobytes() == out[1].tobytes()
    plan.close()
    return out[0]


# every remainder of K by 8, one column or row past a tile edge, one and several segments, every width and height, units cut
@pytest.mark.parametrize("wfmt", ["bf16", "fp16", "fp32"])
@pytest.mark.parametrize("M,N,K", [(65, 1, 1), (66, 33, 7), (81, 65, 33), (97, 129, 250), (113, 257, 515), (129, 33, 1020),
                                   (70, 2050, 1277), (300, 3001, 262), (520, 2570, 1030), (400, 8200, 67)])
def test_any_k_by_plain_loads(M, N, K, wfmt):
    x, W, b = inputs.make_case_w(M, N, K, wfmt)
    assert_bits_equal(run_plain(x, W, b), oracle_y(x, W, b), f"{M} x {N} x {K}")


@pytest.mark.parametrize("wfmt", ["bf16", "fp16", "fp32"])
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_plain_loads_from_any_alignment(offset, wfmt):
    for M, N, K in ((80, 40, 264), (130, 300, 35)):
        x, W, b = inputs.make_case_w(M, N, K, wfmt)
        assert_bits_equal(run_plain(x, W, b, offset), oracle_y(x, W, b), f"offset {offset}: {M} x {N} x {K}")


def test_plain_loads_special_values_at_a_ragged_end():
    """Operands beyond K change no accumulator: not one that ends on -0.0 (an underflowing negative product), no infinity, no NaN."""
    x, W, b = inputs.make_case_w(70, 40, 13, "bf16")
    x[::2], W[:20] = -1e-30, 1e-30
    x[1, 12], x[3, 12] = float("inf"), float("nan")
    b[:] = -0.0
    want, got = oracle_y(x, W, b), run_plain(x, W, b)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.signbit(want[::2, :20]).all() and not want[::2, :20].any()
    assert_bits_equal(np.nan_to_num(got, nan=0.0, posinf=1.0, neginf=2.0), np.nan_to_num(want, nan=0.0, posinf=1.0, neginf=2.0), "special values")


# a few columns, split in K: the plan's memory stays near that of the segment sums (a second pass folds them), and the sums of whole
# tiles are kept where they take little more
@pytest.mark.parametrize("M,N,K,most_mb", [(64000, 1, 2000, 16), (20000, 3, 2001, 16), (30000, 33, 1500, 32), (3000, 130, 2048, 24)])
def test_partials_of_narrow_layers(M, N, K, most_mb):
    x, W, b = inputs.make_case(M, N, K)
    want = oracle_y(x, W, b)
    xd, Wd, bd, y = x.cuda(), W.cuda(), b.cuda(), torch.full((M, N), float("nan"), device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    plan = B.det_linear_plan(M, N, K)
    took = free - torch.cuda.mem_get_info()[0]
    params = B.det_linear_plan_get_params(plan)
    assert params.S > 1 and params.workspace_bytes <= took + (2 << 20)
    assert took <= (most_mb + 24) << 20              # (19 MB are accumulators that blocks hand over)
    for rep in range(2):
        y.fill_(float("nan"))
        B.det_linear_run(plan, xd, Wd, bd, y)
        B.det_linear_plan_check(plan)
        assert_bits_equal(y.cpu().numpy(), want, f"run {rep}")
    plan.close()
