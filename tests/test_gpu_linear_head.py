"""The narrow linear heads (at most 64 output channels that the tensor-core
kernel does not take) through the C-ABI against the CPU oracle: row counts
around the staged block, ragged channel counts, wide and element loads, every
activation. Tolerances are the ones of every conv test (tests/_util.py)."""
import numpy as np
import pytest

import oracle
from paper_2608_09388_gb300 import hc, inputs

from _util import check_close, to_numpy, to_torch

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_09388_gb300 import build
    build.build()
    hc.load_library()


# C_in, C_out, dtype: one channel; ragged rows (45 channels: element loads);
# group remainders; the widest rows and weights the kernel stages
@pytest.mark.parametrize("C_in,C_out,dtype", [
    (1, 1, "bf16"), (3, 2, "f32"), (45, 1, "bf16"), (45, 42, "bf16"), (64, 63, "bf16"),
    (256, 5, "bf16"), (8, 7, "f32"), (64, 64, "f32"), (128, 30, "f32"), (61, 13, "f32")])
@pytest.mark.parametrize("n,cap", [(0, 5), (1, 1), (127, 300), (129, 129), (1000, 4000)])
@pytest.mark.parametrize("shift", [0, 1])
def test_linear_head(C_in, C_out, dtype, n, cap, shift):
    rng = np.random.default_rng(C_in * 131 + C_out * 7 + n + shift)
    act = (oracle.ACT_NONE, oracle.ACT_ELU, oracle.ACT_RELU)[(C_in + C_out + n) % 3]
    x = inputs.features(rng, (cap, C_in), dtype)
    W = inputs.weights(rng, C_in, C_out, dtype)
    b = inputs.features(rng, (C_out,), "f32")
    buf = torch.zeros(cap * C_in + shift, dtype=to_torch(x[:1]).dtype, device="cuda")
    xt = buf[shift:].view(cap, C_in)  # shift 1: rows off the 16-byte boundary
    xt.copy_(to_torch(x))
    y = torch.full((cap, C_out), float("nan"), dtype=xt.dtype, device="cuda")
    count = torch.tensor([n], dtype=torch.int32, device="cuda")
    hc.hc_sparse_linear_fwd(xt, count, to_torch(W), to_torch(b), act, y)
    assert hc.hc_get_device_status() == hc.HC_OK
    y_pre, _ = oracle.sparse_linear(x[:n], W, b, act)
    check_close(to_numpy(y)[:n], y_pre, f"head {C_in}->{C_out} {dtype}")
    assert torch.isnan(y[n:].float()).all()
