"""liblnr's host code on a pretended CUDA runtime (fake_cudart.cpp): the library's own objects
linked with it, so that call order, failed calls and second devices can be tested without a
GPU.  run(script) runs a Python script in a process of its own with the library loaded: `lnr`
(the binding), `r` (a Renderer on device 0), `fk` (the runtime's controls), small inputs."""
import os
import subprocess
import sys
import sysconfig

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_PRELUDE = r"""
import ctypes, sys
sys.path.insert(0, {root!r})
import numpy as np
import synth
import paper_2502_11618_gb300 as lnr
from paper_2502_11618_gb300 import _lib
_lib.LIB_PATH = {lib!r}
fk = lnr.lib()
fk.fk_get.restype = ctypes.c_long
fk.fk_fail_alloc.argtypes = [ctypes.c_long]
get = lambda name: fk.fk_get(name.encode())

CH = (32, 64)
W, H = 64, 48
INTR = synth.intrinsics_for(W, H)
class V: pass
VIEW = V(); VIEW.R = np.eye(3); VIEW.C = np.zeros(3)

class Dev:
    "a device buffer, as far as the binding looks at one"
    is_cuda = True
    def __init__(self, n):
        self.p = ctypes.c_void_p()
        assert fk.cudaMalloc(ctypes.byref(self.p), ctypes.c_size_t(n)) == 0
    def data_ptr(self):
        return self.p.value

def cloud(n, seed=0):
    g = np.random.default_rng(seed)
    return g.uniform(0, 4, (n, 3)), g.integers(0, 256, (n, 3), dtype=np.uint8), g.integers(0, 4, n, dtype=np.uint8)

def renderer(device=0, prec="fp32", ch=CH, n=1000, **kw):
    r = lnr.Renderer(device)
    r.load_cloud(*cloud(n))
    r.build_grid(0.5)
    r.set_unet(ch, synth.unet_weights(ch, seed=1, **kw), prec, **kw)
    return r

def status(f, *a, **k):
    try:
        f(*a, **k)
    except lnr.LnrError as e:
        return e.status
    return 0
"""


def build_library(folder):
    from paper_2502_11618_gb300 import build

    build.build()
    objs = [os.path.join(build.OUT, s[:-3] + ".o") for s in build.sources()]
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    out = os.path.join(str(folder), "liblnr_host" + (sysconfig.get_config_var("SHLIB_SUFFIX") or ".so"))
    cmd = ["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", cuda,
           os.path.join(ROOT, "tests", "fake_cudart.cpp"), *objs, "-lpthread", "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


@pytest.fixture(scope="session")
def run(tmp_path_factory):
    lib = build_library(tmp_path_factory.mktemp("host"))

    def go(script, timeout=120):
        code = _PRELUDE.format(root=ROOT, lib=lib) + script
        r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=timeout)
        assert r.returncode == 0, r.stdout + r.stderr

    return go
