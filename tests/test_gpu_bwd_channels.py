"""The input gradient's two products (over the present taps, and with few input
channels over all pairs) and the weight gradient's two tiles on CUDA cores (16
and 64 input channels) at the channel counts where they change and where rows of
dz, W and P are padded, alone and with the other gradients, against the CPU
oracle; a key outside the mapping is reported by both. Cases, tolerances: those
of tests/test_gpu_bwd.py."""
import pytest

import oracle
from paper_2608_09388_gb300 import hc

torch = pytest.importorskip("torch")
from test_gpu_bwd import _case, _lib, check_against_oracle, run_bwd  # noqa: E402,F401
from _util import to_torch  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,C_in,C_out", [
    ("bf16", 1, 64), ("bf16", 7, 42), ("bf16", 32, 10), ("bf16", 32, 64), ("bf16", 33, 42),
    ("bf16", 64, 1), ("bf16", 40, 66), ("bf16", 130, 42), ("f32", 1, 6), ("f32", 5, 64),
    ("f32", 8, 20), ("f32", 9, 20), ("f32", 16, 3), ("f32", 3, 130), ("bf16", 15, 70),
    ("f32", 17, 130)])
@pytest.mark.parametrize("layout", [oracle.LAYOUT_DENSE, oracle.LAYOUT_COMPACT])
def test_bwd_channels(dtype, C_in, C_out, layout):
    c = _case(C_in * 100 + C_out, 3, 260, 7, C_in, C_out, dtype, layout, oracle.ACT_ELU)
    for want in (("dx", "dW", "db"), ("dx",)):
        check_against_oracle(c, run_bwd(c, want), want)


@pytest.mark.parametrize("C_in", [16, 64])
def test_bwd_bad_keys(C_in):
    c = _case(5, 2, 200, 5, C_in, 32, "bf16", oracle.LAYOUT_COMPACT, oracle.ACT_NONE)
    L, cap = c["rb"].shape
    x = to_torch(c["x"])
    ptr, taps = (torch.from_numpy(t).cuda() for t in run_bwd(c, ("dx",))[3:])
    count = torch.tensor([c["n"]], dtype=torch.int32, device="cuda")
    y = torch.zeros((cap, 32), dtype=torch.bfloat16, device="cuda")
    for bad in (-3, L * cap, 2**31 - 1):
        wrong = taps.clone()
        wrong[4] = bad
        hc.hc_sparse_conv_rulebook_bwd(x, to_torch(c["rb"]), count, to_torch(c["W"]), y, y,
                                       hc.HC_ACT_NONE, ptr, wrong, torch.empty_like(x))
        assert hc.hc_get_device_status() == hc.HC_ERR_INVALID_INDEX, bad
    hc.hc_sparse_conv_rulebook_bwd(x, to_torch(c["rb"]), count, to_torch(c["W"]), y, y,
                                   hc.HC_ACT_NONE, ptr, taps, torch.empty_like(x))
    assert hc.hc_get_device_status() == hc.HC_OK
