"""The package without its built parts: it can be imported (a read-only place, no compiler), says what is missing at the first
use, and works in the same process once it has been built.  No GPU."""
import os
import shutil
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import glob, os, sys
import paper_2502_20853_b200 as mx
assert not [f for f in glob.glob("paper_2502_20853_b200/*.so") if os.path.getsize(f) > 100], "the import has built something"
for use in (lambda: mx.QMat(64, 64, "cpu"), mx.lib, lambda: mx.scale_bytes(64, 64)):
    try:
        use()
    except RuntimeError as e:
        assert "paper_2502_20853_b200.build" in str(e), e
    else:
        raise AssertionError("nothing was said")
os.environ["CXX"] = "g++"
from paper_2502_20853_b200 import build
path = build.build_host()
assert path.endswith(__import__("sysconfig").get_config_var("EXT_SUFFIX")), path
q = mx.QMat(64, 64, "cpu")
assert q.data_addr % 16 == 0 and isinstance(q, mx.binding._host.Mat)
print("done")
"""


def test_import_without_the_built_parts(tmp_path):
    src = os.path.join(ROOT, "paper_2502_20853_b200")
    shutil.copytree(src, tmp_path / "paper_2502_20853_b200", ignore=shutil.ignore_patterns("*.so", "_build", "__pycache__", "*.tmp.*"))
    shutil.copytree(os.path.join(ROOT, "include"), tmp_path / "include")
    (tmp_path / "paper_2502_20853_b200" / "_host.so").write_text("not of this interpreter")
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=tmp_path, env=dict(os.environ, CXX="/bin/false", PYTHONPATH=str(tmp_path)), capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("done"), r.stdout + r.stderr
