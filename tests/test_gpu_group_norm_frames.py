"""The group norm that keeps frames in the shared memory of a cluster, over the
frame tables it takes: many small frames (one CTA each, several rounds, eight at
a time in a cluster), a few CTAs a frame with empty frames beside full ones,
frames above 6144 rows (64-byte parts, several rounds), frames far above the
average (taken first, by whole clusters), 512-channel rows, both types, in place
and not; against the CPU oracle with the tolerances of every group-norm test
(tests/_util.py). A table out of order is reported. And uneven frames take no
longer than on the row-range kernels, which cut the rows evenly."""
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


def rows(seed, n, most):
    return list(np.random.default_rng(seed).integers(0, most + 1, size=n))


def large_among(n, every, full, rest):
    return [full if i % every == every // 2 else rest for i in range(n)]


CASES = {  # dtype, C, G, rows per frame
    "small frames": ("bf16", 128, 8, rows(1, 300, 700)),
    "small frames f32": ("f32", 64, 4, rows(2, 700, 300)),
    "tiny frames": ("bf16", 64, 8, rows(3, 3000, 9)),
    "two CTAs a frame": ("bf16", 128, 8, [0, 1400, 3, 1537, 0, 1100] * 12),
    "four CTAs a frame": ("bf16", 128, 8, [0, 2900, 2500, 0, 3070, 1] * 9),
    "64-byte parts": ("bf16", 128, 8, [6145 + 37 * (i % 7) for i in range(40)]),
    "64-byte parts f32": ("f32", 64, 8, [6200, 6400, 0, 9100] * 5),
    "512 channels": ("bf16", 512, 2, [90, 600, 17, 400] * 2),
    "one large": ("bf16", 128, 8, large_among(64, 64, 10475, 0)),
    "one large, small ones": ("bf16", 128, 8, large_among(64, 64, 7000, 200)),
    "several rounds of large": ("bf16", 128, 4, large_among(240, 6, 1900, 11)),
    "large in wide groups": ("bf16", 256, 2, large_among(40, 20, 5000, 30)),
    "large f32": ("f32", 128, 8, large_among(96, 12, 2500, 1)),
    "large among many": ("bf16", 64, 2, large_among(2000, 500, 6000, 20)),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("in_place", [False, True])
def test_group_norm_frames(name, in_place):
    dtype, C, G, frames = CASES[name]
    case = list(CASES).index(name)
    rng = np.random.default_rng(100 + case)
    offs = np.concatenate([[0], np.cumsum(frames)]).astype(np.int32)
    n, spare = int(offs[-1]), 100
    x = inputs.features(rng, (n + spare, C), dtype)
    gamma = rng.standard_normal(C).astype(np.float32)
    beta = rng.standard_normal(C).astype(np.float32)
    act = (oracle.ACT_ELU, oracle.ACT_RELU, oracle.ACT_NONE)[case % 3]
    xt = to_torch(x)
    y = xt if in_place else torch.full_like(xt, float("nan"))
    keep = xt[n:].clone()
    hc.hc_sparse_group_norm_fwd(xt, to_torch(offs), G, 1e-5, to_torch(gamma), to_torch(beta), act, y)
    assert hc.hc_get_device_status() == hc.HC_OK
    ref, _ = oracle.sparse_group_norm(x[:n], offs, G, 1e-5, gamma, beta, act)
    check_close(to_numpy(y)[:n], ref, f"group norm, {name}")
    if in_place:
        assert torch.equal(y[n:], keep)
    else:
        assert torch.isnan(y[n:].float()).all()


def test_group_norm_table_out_of_order():
    frames = large_among(64, 16, 3000, 100)
    offs = np.concatenate([[0], np.cumsum(frames)]).astype(np.int32)
    n = int(offs[-1])
    offs[20], offs[21] = offs[21], offs[20]
    x = torch.randn((n, 64), generator=torch.Generator("cuda").manual_seed(1), device="cuda")
    y = torch.empty_like(x)
    hc.hc_sparse_group_norm_fwd(x, to_torch(offs), 2, 1e-5, None, None, hc.HC_ACT_NONE, y)
    assert hc.hc_get_device_status() == hc.HC_ERR_INVALID_INDEX


@pytest.mark.parametrize("C", [128, 512])
@pytest.mark.parametrize("frames", [large_among(64, 64, 10475, 0), large_among(64, 64, 10475, 524),
                                    large_among(64, 8, 10475, 100)])
def test_group_norm_uneven_time(frames, C):
    """(One full frame among empty ones took 2.4 times as long, 3.5 at 512
    channels, with the CTAs per frame chosen for the average.)"""
    from _timing import device_us
    offs = torch.tensor(np.concatenate([[0], np.cumsum(frames)]), dtype=torch.int32, device="cuda")
    x = torch.randn((max(64 * 1310, sum(frames)), C), device="cuda").to(torch.bfloat16)
    y = torch.empty_like(x)
    t = {}
    try:
        for path in (0, 2):  # 2: the row ranges
            hc.hc_test_set_option(hc.HC_TEST_GROUP_NORM_PATH, path)
            t[path] = device_us(lambda: hc.hc_sparse_group_norm_fwd(x, offs, 8, 1e-5, None, None,
                                                                    hc.HC_ACT_ELU, y))
    finally:
        hc.hc_test_set_option(hc.HC_TEST_GROUP_NORM_PATH, 0)
    assert t[0] < 1.25 * t[2], t
