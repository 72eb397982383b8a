"""Every call of the Python binding goes to the library that load_library()
opened, also one at another path than the built one: its kernels' errors are
in that library's device status and error string."""
import os
import shutil
import subprocess
import sys

import pytest

pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run(code, tmp_path):
    from paper_2608_09388_gb300 import build, hc
    build.build()
    copy = str(tmp_path / "libhc_elsewhere.so")
    shutil.copy(hc.LIB_PATH, copy)
    r = subprocess.run([sys.executable, "-c", code, copy], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr
    assert r.stdout.strip().endswith("done")


def test_one_library_is_mapped(tmp_path):
    run("""
import sys
from paper_2608_09388_gb300 import hc
hc.load_library(sys.argv[1])
hc._load_native()
maps = {l.split()[-1] for l in open("/proc/self/maps") if "libhc" in l}
assert maps == {sys.argv[1]}, maps
print("done")
""", tmp_path)


@pytest.mark.gpu
def test_errors_reach_the_library_that_was_opened(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    run("""
import sys
import torch
from paper_2608_09388_gb300 import hc
hc.load_library(sys.argv[1])
i32 = dict(dtype=torch.int32, device="cuda")
mask = torch.ones((1, 4), dtype=torch.uint8, device="cuda")
spiral = torch.tensor([[0, 1], [1, 9], [2, 3], [3, 0]], **i32)  # 9: no such vertex
out = [torch.empty((4, 2), **i32), torch.empty((1, 4), **i32), torch.empty((2,), **i32),
       torch.empty((1,), **i32), torch.empty((2, 4), **i32)]
hc.hc_mask_compact_rulebook(mask, spiral, hc.HC_LAYOUT_DENSE, *out)
assert hc.hc_get_device_status() == hc.HC_ERR_INVALID_INDEX
try:
    hc.hc_mask_select_topk(torch.zeros(4, device="cuda"), 9, torch.empty((9,), **i32))
    raise SystemExit("kappa above K was taken")
except hc.HcError as e:
    assert "kappa=9" in str(e), e
print("done")
""", tmp_path)
