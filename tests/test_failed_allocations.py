"""Failed allocations in set-up and factorisation, on the CPU with a runtime that computes nothing.

Whichever allocation fails, the call reports it, leaves no error behind in the runtime (the next
launch check, the library's or the caller's, would take it for its own) and no memory, and the
handle can be factored again.
"""
import os
import shutil
import subprocess
import sys

import pytest

from paper_1602_07652_gb300 import binding, build_lib

HERE = os.path.dirname(os.path.abspath(__file__))
CHILD = r"""
import ctypes, sys
fake, precision = ctypes.CDLL(sys.argv[1]), int(sys.argv[2])
from paper_1602_07652_gb300 import binding
lib = binding.load_library()
n = 16
m = (ctypes.c_double * (n * n))()
grid = binding.Grid(n, n, 2, 2, precision)
failures = {"set-up": 0, "factor": 0}
for k in range(1000):
    h = ctypes.c_void_p()
    fake.fake_fail_at(k)
    where = "set-up"
    rc = lib.ls_setup(ctypes.byref(grid), 1.0 / n, 3.0, ctypes.cast(m, ctypes.c_void_p), None, None, ctypes.byref(h))
    if rc == 0:
        where = "factor"
        rc = lib.ls_factor(h)
    assert fake.cudaPeekAtLastError() == 0, (k, where, rc, "an error is left")
    if rc == 0:
        break
    failures[where] += 1
    assert rc in (-2, -3) and b"memory" in lib.ls_strerror(rc), (k, where, rc)
    if where == "factor":
        fake.fake_fail_at(-1)
        assert lib.ls_factor(h) == 0, (k, "not factored again")
    lib.ls_destroy(h)
    assert fake.fake_live() == 0, (k, where, fake.fake_live(), "allocations left")
assert rc == 0 and min(failures.values()) > 10, (rc, failures)
lib.ls_destroy(h)
assert fake.fake_live() == 0
"""


@pytest.mark.skipif(shutil.which("gcc") is None, reason="needs a C compiler")
@pytest.mark.parametrize("precision", [binding.LS_FP64, binding.LS_MIXED])
def test_a_failed_allocation_leaves_nothing_behind(tmp_path, precision):
    if not os.path.exists(binding.LIB_PATH):
        build_lib.build()
    fake = str(tmp_path / "fake.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-w", "-o", fake, os.path.join(HERE, "_fake_runtime.c")], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD, fake, str(precision)], cwd=os.path.dirname(HERE),
                       env=dict(os.environ, LD_PRELOAD=fake), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
