"""The decode kernel for any K and alignment against the oracle, bit for bit: chunk, group and segment edges, activations
that need several windows of shared memory, weight rows on every 2- or 4-byte offset, special values at a ragged end."""
import numpy as np
import pytest
import torch

from paper_2609_25624_b200 import binding as B
from paper_2609_25624_b200 import inputs
from tests.gpu_util import KERNEL_GENERIC, assert_bits_equal, oracle_y, run_gpu

pytestmark = pytest.mark.gpu


# one, two and four rows a warp; batches on both sides of 1, 2, 4, 8; K around 128, 256 (segment), 1024 and beyond one window
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (1, 9, 129), (2, 1300, 255), (3, 700, 257), (5, 5000, 127), (9, 2400, 385), (64, 700, 131),
                                   (1, 4800, 1025), (8, 33, 7169), (4, 70, 14211), (1, 17, 57001), (17, 40, 2049)])
@pytest.mark.parametrize("wfmt", ["bf16", "fp32"])
def test_ragged_sizes(M, N, K, wfmt):
    x, W, b = inputs.make_case_w(M, N, K, wfmt)
    assert_bits_equal(run_gpu(x, W, b, kernel=KERNEL_GENERIC), oracle_y(x, W, b), f"{M},{N},{K} {wfmt}")


@pytest.mark.parametrize("offset", [1, 2, 3, 5])
@pytest.mark.parametrize("wfmt", ["bf16", "fp16", "fp32"])
def test_misaligned_weights_and_activations(offset, wfmt):
    M, N, K = 6, 1300, 640                           # whole chunks: the rows differ in alignment by the offset only
    x, W, b = inputs.make_case_w(M, N, K, wfmt)
    Wd = torch.empty(N * K + offset, dtype=W.dtype, device="cuda")[offset:].view(N, K)
    xd = torch.empty(M * K + offset, dtype=x.dtype, device="cuda")[offset:].view(M, K)
    Wd.copy_(W)
    xd.copy_(x)
    y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
    plan = B.det_linear_plan_w(M, N, K, wfmt)
    B.det_linear_run(plan, xd, Wd, b.cuda(), y)
    B.det_linear_plan_check(plan)
    plan.close()
    assert_bits_equal(y.cpu().numpy(), oracle_y(x, W, b), f"offset {offset} {wfmt}")


def test_padding_changes_no_accumulator():
    """A chain that ends on -0.0 (an underflowing negative product) keeps its sign, infinities and NaN stay what they are:
    the elements beyond K are skipped, not added."""
    M, N, K = 3, 20, 133
    x = torch.zeros(M, K)
    x[0, :] = -1e-30
    x[1, 5] = float("inf")
    x[2, :] = torch.randn(K, generator=torch.Generator().manual_seed(1))
    W = torch.full((N, K), 1e-30).to(torch.bfloat16)
    W[1::2] = 1.0
    want, got = oracle_y(x, W, None), run_gpu(x, W, None, kernel=KERNEL_GENERIC)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert_bits_equal(np.nan_to_num(got, nan=0.0, posinf=1.0), np.nan_to_num(want, nan=0.0, posinf=1.0), "special values")


# small layers: batch blocks of fewer rows than there are, a warp for each of a row's two segments, a second segment of one chunk, a
# last block of one row, the largest K that one block holds
@pytest.mark.parametrize("M,N,K", [(6, 1333, 1001), (7, 250, 3001), (2, 3, 257), (1, 65, 385), (5, 129, 511), (13, 30, 4095), (30, 64, 1501),
                                   (3, 17, 13999), (1, 9, 55001), (64, 60, 4001)])
@pytest.mark.parametrize("wfmt", ["bf16", "fp16", "fp32"])
def test_small_layers(M, N, K, wfmt):
    x, W, b = inputs.make_case_w(M, N, K, wfmt)
    want = oracle_y(x, W, b)
    assert_bits_equal(run_gpu(x, W, b, kernel=KERNEL_GENERIC), want, f"{M},{N},{K} {wfmt}")
    assert_bits_equal(run_gpu(x, W, b, kernel=KERNEL_GENERIC, max_blocks=2), want, "two blocks")


@pytest.mark.parametrize("M,N,K,offset", [(6, 1333, 1001, 0), (3, 200, 640, 1)])
def test_runs_of_a_plan_search_for_nothing(M, N, K, offset):
    """Runs take a const plan: what is chosen for any K and alignment is chosen with the plan."""
    x, W, b = inputs.make_case(M, N, K)
    xd, bd, y = x.cuda(), b.cuda(), torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
    Wd = torch.empty(N * K + offset, dtype=W.dtype, device="cuda")[offset:].view(N, K)
    Wd.copy_(W)
    plan = B.det_linear_plan(M, N, K)
    before = B.det_test_schedule_searches()
    for _ in range(3):
        B.det_linear_run(plan, xd, Wd, bd, y)
    B.det_linear_plan_check(plan)
    plan.close()
    assert B.det_test_schedule_searches() == before
    assert_bits_equal(y.cpu().numpy(), oracle_y(x, W, b), f"{M},{N},{K} + {offset}")


def layouts(K, S):
    """Every layout that serves K elements in S segments: batch rows, weight rows, a warp a segment (in blocks that hold all of K)."""
    padded = -(-K // 128) * 128
    return [(mt, rt, split) for mt in (1, 2, 4, 8) for rt in (1, 2, 4) for split in (0, 1)
            if not split or (S == 2 and mt < 8 and (rt < 4 or mt == 4) and padded * 4 * mt + 1024 <= 220 * 1024)]


# every layout with an odd number of rows and a last batch block of one row: one segment, two, a second one of one chunk, two warps'
# blocks that just hold 4, 2 and 1 batch rows, activations of 8, 4, 2 and 1 batch rows in several windows
@pytest.mark.parametrize("M,N,K", [(9, 37, 129), (9, 133, 257), (17, 45, 1001), (9, 21, 7169), (9, 13, 13999), (5, 9, 14211), (3, 7, 28289), (2, 5, 57001)])
@pytest.mark.parametrize("wfmt", ["bf16", "fp16", "fp32"])
def test_every_layout(M, N, K, wfmt):
    x, W, b = inputs.make_case_w(M, N, K, wfmt)
    want = oracle_y(x, W, b)
    S = B.det_linear_plan_params(M, N, K).S
    for mt, rt, split in layouts(K, S):
        variant = 100 * mt + 10 * rt + split
        assert_bits_equal(run_gpu(x, W, b, kernel=KERNEL_GENERIC, variant=variant), want, f"layout {variant}")
        assert_bits_equal(run_gpu(x, W, b, kernel=KERNEL_GENERIC, variant=variant, max_blocks=1), want, f"layout {variant}, one block a batch block")


@pytest.mark.parametrize("K,variant", [(1001, 811), (1001, 330), (1001, 131), (1001, 141), (1001, 112), (14211, 411), (57001, 111), (100, 111)])
def test_layouts_that_do_not_fit_are_refused(K, variant):
    plan = B.det_linear_plan(8, 16, K)
    with pytest.raises(B.DetLinearError) as ei:
        B.det_test_plan_set_variant(plan, variant)
    assert ei.value.status == 1
    plan.close()


# several windows of activations in the layouts that calls of this size take: 8 and 4 batch rows
@pytest.mark.parametrize("M,N,K", [(32, 4096, 14335), (3, 8192, 14335)])
def test_several_windows_of_many_rows(M, N, K):
    x, W, b = inputs.make_case(M, N, K)
    assert_bits_equal(run_gpu(x, W, b), oracle_y(x, W, b), f"{M},{N},{K}")
