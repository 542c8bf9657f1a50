"""The library's host code linked against a stand-in for the CUDA runtime (fake_runtime.c), without a GPU.

Handles on two devices of one process: limits and numbers that CUDA keeps per device have to be set and found per
device.  Launches of a round: where they are the time of a small problem, there are no more of them than needed."""
import glob
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TESTS = os.path.join(ROOT, "tests")

PROGRAM = r"""
import ctypes, sys
sys.path.insert(0, sys.argv[2])
import numpy as np
from paper_1507_02087_gb300 import sp2
sp2.LIB_PATH = sys.argv[1]
L = sp2.lib()
ok = lambda rc, what: rc == 0 or sys.exit(f"{what} on device {device}: status {rc}")
F, D = np.zeros(4 << 20), np.zeros(4 << 20)
info = np.zeros(4, dtype=np.int32)
rp, ci = np.arange(65, dtype=np.int32), np.arange(64, dtype=np.int32)
grids = []
for device in (0, 1):
    L.cudaSetDevice(device)
    for N, precision, norm, tile in [(300, 0, 0, 0), (300, 0, 2, 0), (2000, 0, 2, 0), (300, 3, 0, 0), (700, 3, 0, 0),
                                     (300, 1, 0, 1), (300, 1, 0, 2), (300, 4, 0, 1), (300, 4, 2, 2)]:
        for launch_mode in (0, 1):
            o = sp2.sp2_opts()
            L.sp2_default_opts(ctypes.byref(o))
            o.max_iter, o.norm, o.tile, o.launch_mode = 4, norm, tile, launch_mode
            h = ctypes.c_void_p()
            ok(L.sp2_create(N, N // 2, precision, ctypes.byref(o), ctypes.byref(h)), f"create {N, precision, norm, tile}")
            ok(L.sp2_run(h, F.ctypes.data, D.ctypes.data, None), f"run {N, precision, norm, tile}")
            L.sp2_destroy(h)
    for cuda_cores in (0, 1):
        for launch_mode in (0, 1):
            o = sp2.sp2_opts()
            L.sp2_default_opts(ctypes.byref(o))
            o.max_iter, o.norm, o.bsr_cuda_cores, o.launch_mode = 4, 1, cuda_cores, launch_mode
            h = ctypes.c_void_p()
            ok(L.sp2_create_bsr_ex(2048, 1024, 1e-4, 2, ctypes.byref(o), ctypes.byref(h)), f"create bsr {cuda_cores}")
            ok(L.sp2_run_bsr(h, rp.ctypes.data, ci.ctypes.data, F.ctypes.data, 64, D.ctypes.data, None), "run bsr")
            L.sp2_destroy_bsr(h)
    ok(L.sp2_run_fp64_noalloc(F.ctypes.data, D.ctypes.data, 300, 150, info.ctypes.data, None), "noalloc")
    assert L.fake_launched(device) > 0
    grids.append((L._ZN3sp211tc_grid_forEii(10000, 0), L._ZN3sp211tc_grid_forEii(10000, 1)))
assert L.fake_refused() == 0, L.fake_refused()
assert grids == [(152, 2 * (152 // 16)), (100, 2 * (100 // 16))], grids
"""


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    objects = sorted(glob.glob(os.path.join(ROOT, "paper_1507_02087_gb300", "_build", "*.o")))
    if not objects:
        from paper_1507_02087_gb300 import build
        build.build()
        objects = sorted(glob.glob(os.path.join(ROOT, "paper_1507_02087_gb300", "_build", "*.o")))
    d = tmp_path_factory.mktemp("fake")
    from paper_1507_02087_gb300 import build
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    fake, lib = str(d / "fake.o"), str(d / "libsp2.so")
    subprocess.run(["gcc", "-c", "-fPIC", "-I", include, os.path.join(TESTS, "fake_runtime.c"), "-o", fake], check=True)

    def symbols(kind, paths):
        out = subprocess.run(["nm", kind, *paths], capture_output=True, text=True, check=True).stdout
        return {line.split()[-1] for line in out.splitlines() if len(line.split()) >= 2}
    rest = {s for s in symbols("-u", objects) if s.startswith(("cuda", "__cuda"))} - symbols("--defined-only", [fake])
    stubs = d / "stubs.c"                                    # calls whose success is all that matters
    stubs.write_text("".join(f"int {s}(void) {{ return 0; }}\n" for s in sorted(rest)))
    subprocess.run(["g++", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-x", "c", str(stubs), "-x", "none", fake, *objects,
                    "-o", lib, "-ldl"], check=True)
    return lib


def test_handles_on_a_second_device(library):
    r = subprocess.run([sys.executable, "-c", PROGRAM, library, ROOT], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]


SELECTION = r"""
import ctypes, sys
sys.path.insert(0, sys.argv[2])
import numpy as np
from paper_1507_02087_gb300 import sp2
sp2.LIB_PATH = sys.argv[1]
L = sp2.lib()
F, D = np.zeros(4 << 20), np.zeros(4 << 20)
rp, ci = np.arange(65, dtype=np.int32), np.arange(64, dtype=np.int32)

def launches(nb, rule):
    o = sp2.sp2_opts()
    L.sp2_default_opts(ctypes.byref(o))
    o.max_iter, o.launch_mode = 7, 1                          # every round is launched, in pairs: ten of them
    h = ctypes.c_void_p()
    assert L.sp2_create_bsr_ex(32 * nb, 16 * nb, 1e-4, rule, ctypes.byref(o), ctypes.byref(h)) == 0
    before = L.fake_launched(0)
    assert L.sp2_run_bsr(h, rp.ctypes.data, ci.ctypes.data, F.ctypes.data, nb, D.ctypes.data, None) == 0
    n = L.fake_launched(0) - before
    L.sp2_destroy_bsr(h)
    return n

for nb in (1, 4, 44):
    print(nb, launches(nb, 1) - launches(nb, 0))
"""


def test_the_selection_of_a_small_lattice_is_one_launch(library):
    # the error-controlled rule against the rule per block, which needs no selection: one launch more for X_0 and for
    # each of ten rounds
    r = subprocess.run([sys.executable, "-c", SELECTION, library, ROOT], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    extra = dict(tuple(map(int, line.split())) for line in r.stdout.splitlines())
    assert extra == {1: 11, 4: 11, 44: 11}, extra


UNITS = r"""
import ctypes, sys
sys.path.insert(0, sys.argv[2])
import numpy as np
from paper_1507_02087_gb300 import sp2
sp2.LIB_PATH = sys.argv[1]
L = sp2.lib()
L.fake_no_limits(1)
F, D, info = np.zeros(300 * 300), np.zeros(300 * 300), np.zeros(4, dtype=np.int32)
h = ctypes.c_void_p()
print(L.sp2_create(300, 150, 0, None, ctypes.byref(h)), L.sp2_run(h, F.ctypes.data, D.ctypes.data, None))
print(L.sp2_run_fp64_noalloc(F.ctypes.data, D.ctypes.data, 300, 150, info.ctypes.data, None), L.fake_refused())
"""


def test_fp64_runs_where_the_tensor_core_kernels_cannot(library):
    # kernels that need a raised limit are left out; the FP64 units need none, in a handle and without one
    r = subprocess.run([sys.executable, "-c", UNITS, library, ROOT], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split() == ["0"] * 4, r.stdout
