"""Calls small enough for a path of their own, bit-exact against the oracle:
compaction + mapping without a count pass (masks up to 16 KB) around its limit
and on unaligned masks, and the one-pass selection of few masks (ties, NaN, every
kappa)."""
import numpy as np
import pytest

import oracle
from paper_2608_09388_gb300 import hc, inputs

from _util import to_numpy, to_torch
from test_gpu_compact_map import check, run_fused

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_09388_gb300 import build
    build.build()
    hc.load_library()


@pytest.mark.parametrize("B,V,density", [(25, 655, 0.2), (26, 655, 0.2), (1, 16384, 0.05),
                                         (1, 16385, 0.05), (5, 3277, 1.0), (16383, 1, 0.5),
                                         (4, 4096, 0.0), (7, 1025, 0.6)])
@pytest.mark.parametrize("offset", [0, 3])
def test_compact_map_small_masks(B, V, density, offset):
    rng = np.random.default_rng(B + V)
    m = inputs.uniform_mask(rng, B, V, density)
    L = min(5, V)
    sp = rng.integers(-1, V, size=(V, L)).astype(np.int32)
    for layout in (hc.HC_LAYOUT_DENSE, hc.HC_LAYOUT_COMPACT):
        check(m, sp, layout, run_fused(m, sp, layout, offset))
        assert hc.hc_get_device_status() == hc.HC_OK


@pytest.mark.parametrize("K", [1, 2, 31, 33, 255, 256, 257])
def test_topk_few_masks(K):
    rng = np.random.default_rng(K)
    alpha = rng.integers(-3, 4, size=K).astype(np.float32)  # many ties
    alpha[rng.random(K) < 0.1] = np.nan
    alpha[rng.random(K) < 0.05] = np.inf
    alpha[rng.random(K) < 0.05] = -np.inf
    for kappa in sorted({1, (K + 1) // 2, K}):
        sel = torch.full((kappa,), -7, dtype=torch.int32, device="cuda")
        hc.hc_mask_select_topk(to_torch(alpha), kappa, sel)
        assert hc.hc_get_device_status() == hc.HC_OK
        np.testing.assert_array_equal(to_numpy(sel), oracle.select_topk(alpha, kappa))
