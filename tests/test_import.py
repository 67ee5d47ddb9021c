"""The binding without a usable torch: a program that works on numpy arrays imports it and calls it
where torch is not installed, and where it is installed but cannot be loaded."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import numpy as np
import paper_1001_1774_gb300 as tv
opt = tv.tvcs_default_options()
assert opt.max_iter == 500
a = np.zeros(4, np.float32)
assert tv._ptr(a, 4).value == a.ctypes.data
tv._ready(a, None, [a])
try:
    tv._ptr([1.0])
except TypeError:
    print("ok")
"""


@pytest.mark.parametrize("error", ["OSError('libtorch_cpu.so: cannot open shared object file')", "ImportError('no torch')"])
def test_the_binding_works_where_torch_does_not_load(tmp_path, error):
    (tmp_path / "torch.py").write_text("raise %s\n" % error)
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([str(tmp_path), ROOT]))
    p = subprocess.run([sys.executable, "-c", PROGRAM], env=env, cwd=str(tmp_path), capture_output=True, text=True)
    assert p.returncode == 0 and p.stdout.strip() == "ok", p.stderr


def test_torch_imported_after_the_binding_is_found():
    pytest.importorskip("torch")
    program = PROGRAM + """
import torch
t = torch.zeros(4)
for _ in range(2):
    assert tv._ptr(t, 4).value == t.data_ptr()
    assert tv._ptr(a, 4).value == a.ctypes.data
    try:
        tv._ptr(t.double())
    except TypeError:
        print("tensor")
"""
    p = subprocess.run([sys.executable, "-c", program], env=dict(os.environ, PYTHONPATH=ROOT), cwd=ROOT,
                       capture_output=True, text=True)
    assert p.returncode == 0 and p.stdout.split() == ["ok", "tensor", "tensor"], p.stderr
