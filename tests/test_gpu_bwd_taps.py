"""The backward over the present taps, at the sizes where its pieces change:
tiles of 64 / 128 channels on either side, C_in padded to whole 16-byte
chunks in the per-tap products, row units longer than 64 rows, slots without
any tap, runs that end inside a slot, one tap in all. Against the CPU oracle,
tolerance as in test_gpu_bwd."""
import numpy as np
import pytest

import oracle
from paper_2608_09388_gb300 import hc, inputs

from test_gpu_bwd import check_against_oracle, run_bwd

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_09388_gb300 import build
    build.build()
    hc.load_library()


# L, rows, x_rows, C_in, C_out, share of absent taps
SHAPES = [(1, 1, 1, 8, 8, 0.0), (9, 63, 40, 64, 128, 0.7), (9, 65, 70, 45, 64, 0.5),
          (5, 200, 90, 72, 136, 0.3), (3, 400, 333, 200, 40, 0.6), (32, 130, 129, 16, 24, 0.9),
          (4, 9000, 500, 24, 16, 0.97), (2, 300, 128, 8, 264, 0.2), (7, 129, 257, 136, 20, 0.4),
          (6, 64, 64, 3, 5, 0.5), (2, 50, 10, 64, 64, 1.0)]


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("shape", SHAPES)
def test_backward_present_taps(shape, dtype):
    L, n, x_rows, C_in, C_out, absent = shape
    rng = np.random.default_rng(n * 31 + C_in)
    rb = rng.integers(0, x_rows, size=(L, n)).astype(np.int32)
    rb[rng.random((L, n)) < absent] = -1
    if L > 3:
        rb[2] = -1  # a slot without taps
    W = inputs.weights(rng, L * C_in, C_out, dtype)
    x = inputs.features(rng, (x_rows, C_in), dtype)
    y = inputs.features(rng, (n, C_out), dtype)
    dy = inputs.features(rng, (n, C_out), dtype)
    c = dict(x=x, W=W, y=y, dy=dy, rb=rb, n=n, cap=n, dtype=dtype,
             act=(oracle.ACT_NONE, oracle.ACT_RELU)[C_in % 2])
    check_against_oracle(c, run_bwd(c))
