"""Decode runs of several streams on the same SMs, short ones whose predecessor in the stream has long finished: every warp of a block then
starts its work at once, in any order, and none may use a barrier before the warp that initialises it has done so."""
import pytest
import torch

from paper_2609_25624_b200 import binding as B
from paper_2609_25624_b200 import inputs
from tests.gpu_util import assert_bits_equal, oracle_y

pytestmark = pytest.mark.gpu


# tilings with a producer warp of their own for the activations: one and two segment groups, one and two blocks to an SM
@pytest.mark.parametrize("M,N,K,wfmt", [(4, 20000, 512, "bf16"), (8, 32768, 264, "bf16"), (1, 4096, 512, "fp16"), (4, 6144, 776, "bf16"), (16, 5000, 512, "fp32")])
def test_streams_share_the_sms(M, N, K, wfmt):
    x, W, b = inputs.make_case_w(M, N, K, wfmt)
    want = oracle_y(x, W, b)
    xd, Wd, bd = x.cuda(), W.cuda(), b.cuda()
    streams = [torch.cuda.Stream() for _ in range(4)]
    plans = [B.det_linear_plan_w(M, N, K, wfmt) for _ in streams]
    ys = [torch.full((M, N), float("nan"), device="cuda") for _ in streams]
    copies = [torch.empty_like(xd) for _ in streams]
    torch.cuda.synchronize()
    for rep in range(40):
        for stream, plan, y, xc in zip(streams, plans, ys, copies):
            with torch.cuda.stream(stream):
                xc.copy_(xd)                         # a copy, after which the run starts without a kernel to wait for
                B.det_linear_run(plan, xc, Wd, bd, y)
    torch.cuda.synchronize()
    for stream, plan, y in zip(streams, plans, ys):
        B.det_linear_plan_check(plan, stream=stream)
        assert_bits_equal(y.cpu().numpy(), want, f"{M},{N},{K}")
        plan.close()
