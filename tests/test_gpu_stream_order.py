"""W and b written in the stream shortly before a run.  The decode kernel requests its weights and reads the bias ahead of its wait
for the kernel before it; here that kernel is one of the library's own, and the kernel before that one, a long decode run that
lets its successors start as soon as it has started itself, writes b, or W of an FP32 layer.  The kernel in between must not let
the run begin before the writer is complete."""
import pytest
import torch

from paper_2609_25624_b200 import binding as B
from tests.gpu_util import KERNEL_GENERIC, assert_bits_equal

pytestmark = pytest.mark.gpu


def _normal(seed, *shape):
    return torch.randn(*shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))


def _rmsnorm(M, H):
    x, g, y = _normal(1, M, H), _normal(2, H), torch.empty(M, H, device="cuda")
    return lambda: B.det_rmsnorm(x, g, 1e-5, y)


def _attention(batch, T):
    q, k, v = _normal(1, batch, 8, 64), _normal(2, batch, 4, T, 64), _normal(3, batch, 4, T, 64)
    o = torch.empty_like(q)
    return lambda: B.det_attention_decode(q, k, v, 0.125, o)


def _linear(M, N, K, kernel=None, noalloc=False):
    x, W, y = _normal(1, M, K), _normal(2, N, K).to(torch.bfloat16), torch.empty(M, N, device="cuda")
    if noalloc:
        return lambda: B.det_linear_run_noalloc(x, W, None, y)
    plan = B.det_linear_plan(M, N, K)
    if kernel is not None:
        B.det_test_plan_force_kernel(plan, kernel)
    return lambda: B.det_linear_run(plan, x, W, None, y)


BETWEEN = {
    "rmsnorm, a block per row": lambda: _rmsnorm(4, 4096),
    "rmsnorm, a warp per row": lambda: _rmsnorm(600, 1024),
    "attention": lambda: _attention(1, 300),
    "prefill": lambda: _linear(65, 32, 64),
    "prefill with a second pass": lambda: _linear(65, 32, 2048, noalloc=True),
    "prefill by plain loads": lambda: _linear(65, 32, 63),
    "decode for any K": lambda: _linear(2, 64, 63),
    "decode without a plan": lambda: _linear(2, 64, 64, noalloc=True),
    "decode without a plan, a producer for both operands": lambda: _linear(16, 300, 512, noalloc=True),
}


def _writer(M, N, K):
    """A run that writes [M, N] floats: some ten microseconds and more, on a few SMs only, so that what comes after it has room to
    start."""
    x, W = _normal(11, M, K), (0.02 * _normal(12, N, K)).to(torch.bfloat16)
    plan = B.det_linear_plan(M, N, K)
    assert B.det_linear_plan_describe(plan)["kernel"] == "decode"
    return lambda out: B.det_linear_run(plan, x, W, None, out)


def _check(write, out, between, run, y):
    """The calls as a program issues them, against the same calls with a synchronisation after each."""
    torch.cuda.synchronize()
    write(out)
    torch.cuda.synchronize()
    run()
    torch.cuda.synchronize()
    want = y.cpu().numpy()
    for rep in range(5):
        out.fill_(float(rep))
        y.fill_(float("nan"))
        torch.cuda.synchronize()
        write(out)
        between()
        run()
        torch.cuda.synchronize()
        assert_bits_equal(y.cpu().numpy(), want, f"repetition {rep}")


@pytest.mark.parametrize("between", BETWEEN)
def test_bias_written_before_the_kernel_in_between(between):
    N = 256
    b, x, W, y = torch.empty(1, N, device="cuda"), _normal(21, 3, 512), _normal(22, N, 512).to(torch.bfloat16), torch.empty(3, N, device="cuda")
    plan = B.det_linear_plan(3, N, 512)
    _check(_writer(1, N, 65536), b, BETWEEN[between](), lambda: B.det_linear_run(plan, x, W, b[0], y), y)
    plan.close()


@pytest.mark.parametrize("between", BETWEEN)
def test_weights_written_before_the_kernel_in_between(between):
    W, x, y = torch.empty(64, 256, device="cuda"), _normal(21, 2, 256), torch.empty(2, 64, device="cuda")
    plan = B.det_linear_plan_w(2, 64, 256, "fp32")
    _check(_writer(64, 256, 16384), W, BETWEEN[between](), lambda: B.det_linear_run(plan, x, W, None, y), y)
    plan.close()


# activations that come over by a kernel (pinned and small) and by a copy
@pytest.mark.parametrize("M,N,pinned", [(3, 256, True), (30, 256, True), (3, 256, False), (70, 256, True)])
def test_bias_written_before_a_run_on_host_activations(M, N, pinned):
    W, b = _normal(22, N, 512).to(torch.bfloat16), torch.empty(1, N, device="cuda")
    x, y = _normal(21, M, 512).cpu(), torch.empty(M, N)
    if pinned:
        x, y = x.pin_memory(), y.pin_memory()
    plan = B.det_linear_plan(M, N, 512)
    _check(_writer(1, N, 65536), b, lambda: None, lambda: B.det_linear_run_host(plan, x, W, b[0], y), y)
    plan.close()


def test_weights_written_before_a_run_on_host_activations():
    W, x, y = torch.empty(64, 256, device="cuda"), _normal(21, 2, 256).cpu().pin_memory(), torch.empty(2, 64).pin_memory()
    plan = B.det_linear_plan_w(2, 64, 256, "fp32")
    _check(_writer(64, 256, 16384), W, lambda: None, lambda: B.det_linear_run_host(plan, x, W, None, y), y)
    plan.close()


# the bias by a long run that lets its successors start early, straight before: decode kernels with one and two segment groups and one
# producer for both operands, decode for any K, prefill by TMA and by plain loads
@pytest.mark.parametrize("M,N,K", [(3, 256, 512), (16, 300, 512), (1, 20000, 264), (3, 256, 511), (65, 256, 512), (65, 256, 63)])
def test_bias_written_before_a_run_without_a_plan(M, N, K):
    x, W, y = _normal(21, M, K), _normal(22, N, K).to(torch.bfloat16), torch.empty(M, N, device="cuda")
    b = torch.empty(1, N, device="cuda")
    _check(_writer(1, N, 65536 if N < 1000 else 4096), b, lambda: None, lambda: B.det_linear_run_noalloc(x, W, b[0], y), y)
