"""The group norm that keeps each frame's rows in shared memory across a
cluster (many large frames), against the CPU oracle: empty and single-row
frames beside large ones, rows beyond the shared memory (read twice), every
group width it takes, few and many frames, in place, fp32 and bf16. Tolerances
are the ones of every group-norm test (tests/_util.py)."""
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


# dtype, C, G, rows per frame; spare rows make the average frame (by capacity)
# too large for the per-(frame, group) kernel
CASES = [
    ("bf16", 64, 1, [700, 0, 1, 33, 650] * 4, 0),
    ("bf16", 128, 8, [1, 0, 3, 2, 0, 5, 1, 7] * 2, 40000),
    ("bf16", 128, 4, [2049, 100, 0, 1500] * 3, 9000),
    ("bf16", 256, 1, [300, 31, 32, 257] * 4, 3000),
    ("bf16", 512, 2, [90, 600, 17, 400], 4000),
    ("f32", 64, 8, [900, 901, 0, 2500] * 4, 20000),
    ("f32", 128, 1, [64, 1, 300, 299] * 4, 8000),
    ("bf16", 1024, 8, [7000, 6145], 0),  # past 8 x 384 rows a part: read twice
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("in_place", [False, True])
def test_group_norm_cluster(case, in_place):
    dtype, C, G, frames, spare = CASES[case]
    rng = np.random.default_rng(case)
    offs = np.concatenate([[0], np.cumsum(frames)]).astype(np.int32)
    n = int(offs[-1])
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
    check_close(to_numpy(y)[:n], ref, f"group norm {CASES[case][:3]}")
    if in_place:
        assert torch.equal(y[n:], keep)
    else:
        assert torch.isnan(y[n:].float()).all()


def test_group_norm_cluster_constant_groups_and_bad_table():
    """Equal values normalise to exactly beta; a table outside the rows is
    reported."""
    frames = [1100, 1000, 7, 1300] * 4
    offs = np.concatenate([[0], np.cumsum(frames)]).astype(np.int32)
    n = int(offs[-1])
    x = torch.full((n, 64), 3.7, device="cuda")
    y = torch.empty_like(x)
    beta = torch.arange(64, dtype=torch.float32, device="cuda")
    hc.hc_sparse_group_norm_fwd(x, to_torch(offs), 2, 1e-5, None, beta, hc.HC_ACT_NONE, y)
    assert hc.hc_get_device_status() == hc.HC_OK
    assert torch.equal(y, beta.expand_as(y))
    bad = offs.copy()
    bad[-1] = n + 5
    hc.hc_sparse_group_norm_fwd(x, to_torch(bad), 2, 1e-5, None, beta, hc.HC_ACT_NONE, y)
    assert hc.hc_get_device_status() == hc.HC_ERR_INVALID_INDEX
