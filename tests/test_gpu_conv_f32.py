"""The fp32 sparse conv over its tile shapes, against the CPU oracle: both tile
heights (the batch's vertices decide), tiles shared out unevenly, every unit
height (few, some and all taps present), channel counts around a step (16 and
32 channels) and around an output tile, element loads, spirals of 1 to 32.
The output must equal an fp32 chain, so the bound is the one of every fp32
test (tests/_util.py). Non-finite inputs reach only the rows that read them."""
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


def _run(x, layout, m, sp, W, b, act, fused):
    B, V = m.shape
    L = sp.shape[1]
    coords = torch.empty((B * V, 2), dtype=torch.int32, device="cuda")
    row_of = torch.empty((B, V), dtype=torch.int32, device="cuda")
    offs = torch.empty((B + 1,), dtype=torch.int32, device="cuda")
    count = torch.empty((1,), dtype=torch.int32, device="cuda")
    rb = torch.empty((L, B * V), dtype=torch.int32, device="cuda")
    hc.hc_mask_compact_rulebook(to_torch(m), to_torch(sp), layout, coords, row_of, offs, count, rb)
    y = torch.full((B * V, W.shape[1]), float("nan"), device="cuda")
    out = torch.zeros((B, V, W.shape[1]), device="cuda") if fused else None
    hc.hc_sparse_conv_rulebook_fwd(to_torch(x), rb, count, to_torch(W), to_torch(b), act, y,
                                   coords=coords if fused else None, out=out)
    assert hc.hc_get_device_status() == hc.HC_OK
    n = int(count.item())
    if fused:
        c = coords[:n].long()
        assert torch.equal(out[c[:, 0], c[:, 1]], y[:n])
    assert torch.isnan(y[n:]).all()
    return to_numpy(y)[:n], coords[:n].cpu().numpy(), row_of.cpu().numpy()


# B, V, L, C_in, C_out, density
CASES = [(1, 655, 9, 16, 64, 0.1), (1, 70, 1, 5, 3, 0.5), (2, 500, 32, 17, 65, 0.05),
         (3, 333, 12, 33, 130, 1.0), (1, 17, 4, 64, 128, 0.9), (4, 655, 9, 32, 40, 0.3),
         (20, 655, 9, 64, 128, 0.02), (20, 655, 9, 48, 64, 0.6), (17, 655, 7, 16, 72, 0.15),
         (30, 655, 5, 7, 129, 1.0), (16, 655, 32, 36, 32, 0.08)]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("layout", [oracle.LAYOUT_DENSE, oracle.LAYOUT_COMPACT])
def test_conv_f32(case, layout):
    B, V, L, C_in, C_out, density = case
    sp, m, x, W, b = inputs.random_case(B * 7 + C_out, B, V, L, C_in, C_out, "f32", density,
                                        neg_frac=0.1)
    act = (oracle.ACT_ELU, oracle.ACT_NONE, oracle.ACT_RELU)[(B + C_in) % 3]
    c, r, _, n = oracle.mask_compact(m)
    xin = x if layout == oracle.LAYOUT_DENSE else oracle.gather_rows(x, c)
    got, coords, _ = _run(xin, layout, m, sp, W, b, act, fused=C_out % 2 == 0)
    assert np.array_equal(coords, c)
    y_pre, _ = oracle.sparse_spiral_conv(xin, layout, c, r, sp, W, b, act)
    check_close(got, y_pre, f"fp32 conv {case}")


def test_conv_f32_non_finite_rows_stay_apart():
    """A NaN and an infinity in two input rows: only the output rows whose
    present taps read them are non-finite."""
    B, V, L, C_in, C_out = 2, 300, 9, 24, 64
    sp, m, x, W, b = inputs.random_case(3, B, V, L, C_in, C_out, "f32", 0.3)
    c, r, _, n = oracle.mask_compact(m)
    (b0, v0), (b1, v1) = c[5], c[n - 3]
    x[b0, v0, 3] = np.nan
    x[b1, v1, 7] = np.inf
    got, _, _ = _run(x, oracle.LAYOUT_DENSE, m, sp, W, b, oracle.ACT_NONE, fused=False)
    reads = np.array([any((bb, u) in ((b0, v0), (b1, v1)) and r[bb, u] >= 0 for u in sp[v])
                      for bb, v in c])
    assert (~np.isfinite(got)).any(axis=1).tolist() == reads.tolist()
