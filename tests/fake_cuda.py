"""Runs a Python script against libxs with the CUDA calls of fake_cuda.c in place of the runtime's."""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import ctypes, numpy as np, molgen
from paper_2505_24807_gb300 import xs
fake = ctypes.CDLL(None)
fake.fake_used.restype = fake.fake_peak.restype = ctypes.c_size_t
fake.fake_set_capacity.argtypes = [ctypes.c_int, ctypes.c_size_t]
fake.fake_pending.restype = ctypes.c_longlong
fake.fake_fill.argtypes = [ctypes.c_size_t, ctypes.c_int]
fake.fake_fail.argtypes = [ctypes.c_longlong, ctypes.c_longlong]
fake.fake_launched.restype = ctypes.c_longlong
class device_array:                            # float64, zero
    def __init__(self, *shape):
        self.shape, p = shape, ctypes.c_void_p()
        assert fake.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(8 * int(np.prod(shape)))) == 0
        self.p = p.value
    def data_ptr(self):
        return self.p
PARAMS = molgen.params_table(molgen.make_params(0))
def context(device=0):
    h = xs.xs_create(device)
    xs.xs_set_params(h, PARAMS)
    return h
"""


def run(tmp_path, script):
    """The script's standard output; the script sees `fake` (fake_cuda.c), xs, np, molgen and context()."""
    from paper_2505_24807_gb300 import build
    cc = shutil.which("gcc")
    try:
        build.build()
        include = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    except RuntimeError as e:
        pytest.skip(f"cannot build libxs.so here: {e}")
    if not cc or not os.path.exists(os.path.join(include, "cuda_runtime_api.h")):
        pytest.skip("no C compiler or CUDA headers")
    lib = os.path.join(tmp_path, "fake_cuda.so")
    subprocess.run([cc, "-O1", "-shared", "-fPIC", "-pthread", "-I", include, os.path.join(ROOT, "tests", "fake_cuda.c"),
                    "-o", lib], check=True)
    # past the exit handlers of the real libraries, which have no device here
    script = PRELUDE + script + "\nimport os, sys\nsys.stdout.flush()\nos._exit(0)\n"
    r = subprocess.run([sys.executable, "-c", script], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, LD_PRELOAD=lib))
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout
