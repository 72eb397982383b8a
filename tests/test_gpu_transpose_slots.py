"""The transposed mapping at every spiral length: the sort's blocks hold their
entries (256 input rows up to 16 slots, 128 above), and where a few rows have so
many that they do not, the rows beside them are right too. Bit-exact against a
sort in numpy. And no step in time between 16 and 24 slots."""
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


def transpose(rb, n, x_rows):
    L, cap = rb.shape
    count = torch.tensor([n], dtype=torch.int32, device="cuda")
    row_ptr = torch.full((x_rows + 1,), -7, dtype=torch.int32, device="cuda")
    taps = torch.full((L * cap,), -7, dtype=torch.int32, device="cuda")
    rbt = torch.from_numpy(rb).cuda()
    return rbt, count, row_ptr, taps, lambda: hc.hc_conv_rulebook_transpose(
        rbt, count, x_rows, row_ptr, taps)


def neighbours(rng, L, n):
    """Every tap present; each row read about L times."""
    return np.stack([rng.permutation(n) for _ in range(L)]).astype(np.int32)


@pytest.mark.parametrize("L,n,hubs", [
    (16, 1500, 0), (17, 1023, 0), (20, 700, 0), (21, 513, 0), (24, 900, 0), (32, 1100, 0),
    (9, 900, 1), (20, 640, 3), (32, 600, 2)])
def test_rulebook_transpose_slots(L, n, hubs):
    rng = np.random.default_rng(L * 31 + hubs)
    rb = neighbours(rng, L, n)
    if hubs:  # these rows are read by two thirds of every other slot
        to_hub = rng.random((L, n)) < 0.67
        to_hub[::2] = False
        rb[to_hub] = rng.integers(100, 100 + hubs, size=to_hub.sum())
    *_, row_ptr, taps, call = transpose(rb, n, n)
    call()
    assert hc.hc_get_device_status() == hc.HC_OK
    j = rb.T.reshape(-1)
    order = np.lexsort((np.arange(j.size), j))
    np.testing.assert_array_equal(
        row_ptr.cpu().numpy(), np.concatenate([[0], np.cumsum(np.bincount(j, minlength=n))]))
    np.testing.assert_array_equal(taps.cpu().numpy(), order)


def test_rulebook_transpose_time():
    """1.5 times the entries take no more than 3 times as long (13 times with
    256 rows to a block at every L: its slices did not fit)."""
    from _timing import device_us
    t = {L: device_us(transpose(neighbours(np.random.default_rng(L), L, 41920), 41920, 41920)[-1])
         for L in (16, 24)}
    assert t[24] < 3 * t[16], t
