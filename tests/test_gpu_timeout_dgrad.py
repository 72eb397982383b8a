"""The bounded-wait failure path of the input gradient's tap product, as
tests/test_gpu_timeout.py has it for the other pipelined kernels: with the wait
limit lowered far below the time of its first stages the call gives up, the
status reads HC_ERR_TIMEOUT, and with the limit back the same call is correct.
No kernel is made to hang. The unwind waits for the weight copies alone, so
giving up takes far less than one full wait limit."""
import time

import pytest

import oracle
from paper_2608_09388_gb300 import hc, inputs

from _util import to_torch

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHORT_LIMIT_NS = 500


@pytest.mark.parametrize("C_in", [64, 128])
def test_input_gradient_wait_timeout_reported_then_correct(C_in):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_09388_gb300 import build
    build.build()
    hc.load_library()
    assert hc.hc_get_device_status() == hc.HC_OK
    C_out = 128
    sp, m, x, W, b = inputs.random_case(7003, 8, 4000, 9, C_in, C_out, "bf16", 1.0)
    c, r, _, n = oracle.mask_compact(m)
    rb = to_torch(oracle.conv_rulebook(c, r, sp, oracle.LAYOUT_COMPACT))
    L, Wt = sp.shape[1], to_torch(W)
    gen = torch.Generator("cuda").manual_seed(4)
    y, dy = (torch.randn((n, C_out), generator=gen, device="cuda").to(torch.bfloat16) for _ in "ab")
    xt = torch.empty((n, C_in), dtype=torch.bfloat16, device="cuda")
    count = torch.tensor([n], dtype=torch.int32, device="cuda")
    ptr = torch.empty((n + 1,), dtype=torch.int32, device="cuda")
    taps = torch.empty((L * n,), dtype=torch.int32, device="cuda")
    hc.hc_conv_rulebook_transpose(rb, count, n, ptr, taps)
    dx = torch.empty_like(xt)

    def bwd():
        hc.hc_sparse_conv_rulebook_bwd(xt, rb, count, Wt, y, dy, hc.HC_ACT_ELU, ptr, taps, dx,
                                       None, None)

    bwd()
    assert hc.hc_get_device_status() == hc.HC_OK
    want = dx.clone()
    try:
        hc.hc_test_set_option(hc.HC_TEST_WAIT_LIMIT_NS, SHORT_LIMIT_NS)
        t = time.monotonic()
        bwd()
        assert hc.hc_get_device_status() == hc.HC_ERR_TIMEOUT
        assert time.monotonic() - t < 1.5  # the full limit is 2 s
    finally:
        hc.hc_test_set_option(hc.HC_TEST_WAIT_LIMIT_NS, 0)
    dx.fill_(float("nan"))
    bwd()
    assert hc.hc_get_device_status() == hc.HC_OK
    assert torch.equal(dx, want)
