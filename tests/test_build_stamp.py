"""The binding is built for one torch and one Python: build() makes it again
for others, and builds the library alone where there is no torch."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run(code, *args):
    r = subprocess.run([sys.executable, "-c", code, *map(str, args)], cwd=ROOT,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    assert r.stdout.strip().endswith("done")


@pytest.fixture(scope="module", autouse=True)
def _built():
    pytest.importorskip("torch")
    from paper_2608_09388_gb300 import build
    build.build()
    assert build.up_to_date()


def test_binding_of_another_torch_is_out_of_date(tmp_path):
    other = tmp_path / "torch"
    other.mkdir()
    (other / "__init__.py").write_text("__version__ = '9.9.9'\n")
    (other / "version.py").write_text("__version__ = '9.9.9'\n")
    run("""
import sys
sys.path.insert(0, sys.argv[1])
from paper_2608_09388_gb300 import build, hc
assert not build.up_to_date()
try:
    hc._load_native()
    raise SystemExit("the binding of another torch was loaded")
except RuntimeError as e:
    assert "another torch" in str(e), e
print("done")
""", tmp_path)


def test_library_builds_without_torch(tmp_path):
    (tmp_path / "one.cu").write_text('extern "C" int one() { return 1; }\n')
    run("""
import ctypes, os, sys
sys.modules["torch"] = None
from paper_2608_09388_gb300 import build
build.CSRC = build.BUILD = sys.argv[1]
build.LIB = os.path.join(sys.argv[1], "libone.so")
build.NATIVE = os.path.join(sys.argv[1], "native.so")
assert ctypes.CDLL(build.build()).one() == 1
assert build.up_to_date() and not os.path.exists(build.NATIVE)
print("done")
""", tmp_path)
