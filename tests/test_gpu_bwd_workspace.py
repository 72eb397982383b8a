"""The backward's workspace is what include/hc.h states: the first call on a new
stream takes a copy of dy, the per-tap products and 8 bytes per rulebook entry,
not more than partial sums beside them."""
import pytest

from paper_2608_09388_gb300 import hc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("C_in", [8, 40])
def test_backward_workspace(C_in):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_09388_gb300 import build
    build.build()
    hc.load_library()
    cap, n, L, C_out = 3 << 20, 300, 9, 8
    g = torch.Generator("cuda").manual_seed(1)
    rb = torch.randint(0, n, (L, cap), generator=g, dtype=torch.int32, device="cuda")
    count = torch.tensor([n], dtype=torch.int32, device="cuda")
    ptr = torch.empty((n + 1,), dtype=torch.int32, device="cuda")
    taps = torch.empty((L * cap,), dtype=torch.int32, device="cuda")
    hc.hc_conv_rulebook_transpose(rb, count, n, ptr, taps)
    bf = dict(dtype=torch.bfloat16, device="cuda")
    x, W = torch.randn((n, C_in), **bf), torch.randn((L * C_in, C_out), **bf)
    y, dy = torch.zeros((cap, C_out), **bf), torch.zeros((cap, C_out), **bf)
    dx, dW = torch.empty_like(x), torch.empty((L * C_in, C_out), device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    hc.hc_sparse_conv_rulebook_bwd(x, rb, count, W, y, dy, hc.HC_ACT_ELU, ptr, taps, dx, dW, None,
                                   stream=side)
    assert hc.hc_get_device_status(side) == hc.HC_OK
    taken = free - torch.cuda.mem_get_info()[0]
    stated = cap * C_out * 2 + cap * L * (C_in * 2 + 8)
    assert taken <= stated + (64 << 20), (taken, stated)
