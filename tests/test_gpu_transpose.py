"""The transposed Eq. 4 mapping through the C-ABI, bit-exact against a sort in
numpy: input-row counts around the sort's block (256 rows) and the scan's
tile (4096), more entries in a block than it stages (5120), empty slots, no
rows, rows with one entry and with hundreds."""
import numpy as np
import pytest

from paper_2608_09388_gb300 import hc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_09388_gb300 import build
    build.build()
    hc.load_library()


@pytest.mark.parametrize("L,cap,n,x_rows,absent", [
    (1, 1, 1, 1, 0.0), (3, 300, 257, 255, 0.5), (9, 1500, 1024, 256, 0.3),
    (5, 5000, 4999, 257, 0.0), (9, 700, 613, 4097, 0.8), (12, 9000, 8193, 12289, 0.2),
    (32, 400, 0, 100, 0.0), (7, 3000, 2500, 3, 0.1), (16, 2000, 1999, 8192, 1.0)])
def test_rulebook_transpose(L, cap, n, x_rows, absent):
    rng = np.random.default_rng(L * 1009 + n)
    rb = rng.integers(0, x_rows, size=(L, cap)).astype(np.int32)
    rb[rng.random((L, cap)) < absent] = -1
    if L > 2:
        rb[1] = -1  # a slot without entries
    count = torch.tensor([n], dtype=torch.int32, device="cuda")
    row_ptr = torch.full((x_rows + 1,), -7, dtype=torch.int32, device="cuda")
    taps = torch.full((L * cap,), -7, dtype=torch.int32, device="cuda")
    hc.hc_conv_rulebook_transpose(torch.from_numpy(rb).cuda(), count, x_rows, row_ptr, taps)
    assert hc.hc_get_device_status() == hc.HC_OK
    j = rb[:, :n].T.reshape(-1)  # entry n * L + l
    key = np.flatnonzero(j >= 0)
    order = np.lexsort((key, j[key]))
    np.testing.assert_array_equal(
        row_ptr.cpu().numpy(), np.concatenate([[0], np.cumsum(np.bincount(j[key], minlength=x_rows))]))
    got = taps.cpu().numpy()
    np.testing.assert_array_equal(got[:key.size], key[order])
    assert (got[key.size:] == -7).all()
