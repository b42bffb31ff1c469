"""Engine admission when a CUDA call fails, on the CPU: the library's objects
linked against a runtime in host memory (tests/fake_cuda) that fails the call
asked for.  A slot whose admission fails must not take part in the reductions."""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import ctypes, sys
import numpy as np
from paper_1510_08886_gb300 import _lib
_lib.LIB_PATH = sys.argv[1]
L = _lib.lib()
import paper_1510_08886_gb300 as lbm
e, w, c = lbm.dvm("D2V16")
d = lbm._DVM(e, w, c)
rho = np.ones(64)
arenas = []                            # (the runtime remembers the flags in them)
for prec in (0, 1, 2):
    size = 8 << 20
    raw = ctypes.create_string_buffer(size + 256)
    arenas.append(raw)
    base = (ctypes.addressof(raw) + 255) & ~255
    eng, slot = ctypes.c_void_p(), ctypes.c_int(-1)
    assert L.lbm_engine_create(prec, 4, ctypes.c_void_p(base), size, None, ctypes.byref(eng)) == 0
    add = lambda: L.lbm_engine_add(eng, d.ref(), 3, 1, 64, 0.1, 1e-3,
                                   rho.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), ctypes.byref(slot))
    active = L.fake_active()
    for name, nth in ((b"k_generic", 1), (b"memcpy", 1), (b"memcpy", 2), (b"k_admit", 1)):
        L.fake_fail(name, nth)
        assert add() == _lib.LBM_ECUDA, (prec, name)
        assert L.fake_active() == active, (prec, name, "a failed admission left its flag set")
        L.cudaGetLastError()               # as a program that goes on after an error does
    assert add() == 0 and L.fake_active() == active + 1 and slot.value == 0
    L.fake_fail(b"k_generic", 1)
    assert add() == _lib.LBM_ECUDA and L.fake_active() == active + 1
    assert L.lbm_engine_remove(eng, 0) == 0 and L.fake_active() == active
    assert add() == 0 and L.fake_active() == active + 1 and slot.value == 0
    assert L.lbm_engine_remove(eng, 0) == 0
    L.lbm_engine_destroy(eng)
"""


@pytest.mark.skipif(shutil.which("gcc") is None, reason="no host compiler")
def test_failed_admission_leaves_no_flag(tmp_path):
    import __graft_entry__
    __graft_entry__.build_library()
    from paper_1510_08886_gb300 import build
    objects = [build.object_path(u) for u in build.UNITS]
    if not all(map(os.path.exists, objects)):
        build.build(force=True)
    so = str(tmp_path / "liblbm_fake.so")
    subprocess.run(["gcc", "-O1", "-fPIC", "-c", "-o", str(tmp_path / "fake.o"),
                    os.path.join(ROOT, "tests", "fake_cuda", "fake_cudart.c")], check=True)
    subprocess.run(["g++", "-shared", "-o", so, str(tmp_path / "fake.o")]
                   + objects, check=True)
    r = subprocess.run([sys.executable, "-c", SCRIPT, so], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
