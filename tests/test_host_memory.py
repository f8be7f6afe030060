"""The host code's memory handling, without a GPU: the library's own objects
linked to a stand-in for the CUDA runtime (host_runtime.cu) in which kernels
do nothing. Host buffers outlive the asynchronous copies made from them."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.join(ROOT, "tests")

CHILD = """
import ctypes as C
import sys
import numpy as np
from paper_2112_07115_gb300 import dcem, scenes
dcem.LIB_PATH = sys.argv[1]
L = dcem.lib()
L.fake_bad_text.restype = C.c_char_p
"""


@pytest.fixture(scope="module")
def stand_in(tmp_path_factory):
    from paper_2112_07115_gb300 import build
    build.build()
    out = tmp_path_factory.mktemp("host_runtime")
    src, nvcc = os.path.join(HERE, "host_runtime.cu"), build._nvcc()
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    objs = [os.path.join(build.BUILD, f.replace(".cu", ".o")) for f in build.SOURCES]
    run = lambda *cmd: subprocess.run(cmd, check=True, capture_output=True, text=True)
    run(nvcc, *build.ARCH, *build.NVCC_FLAGS, "-c", src, "-o", str(out / "a.o"))
    run("g++", "-x", "c++", "-std=c++17", "-O1", "-fPIC", "-I" + inc, "-c", src, "-o", str(out / "b.o"))
    lib = str(out / "libdcem_host.so")
    run(nvcc, *build.ARCH, "-shared", "-cudart", "none", "-Xlinker", "-Bsymbolic", "-o", lib, *objs,
        str(out / "a.o"), str(out / "b.o"))
    return lib


def _child(lib, code):
    r = subprocess.run([sys.executable, "-c", CHILD + code, lib], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]


def test_sources_of_copies_outlive_them_scene(stand_in):
    _child(stand_in, """
for sc in (scenes.city_blocks(n=2), scenes.toy_street()):
    s = dcem.Scene.from_scene(sc)
    s.set_rays(scenes.fibonacci_sphere(100))
    s.close()
assert L.fake_stale() == 0, L.fake_stale()
""")


def test_sources_of_copies_outlive_them_derivatives(stand_in):
    _child(stand_in, """
sc = scenes.toy_street()
s = dcem.Scene.from_scene(sc)
before = L.fake_stale()
prm = dcem.default_params(max_refl=3)
none = np.zeros(0, dcem.PATH_DTYPE)
for n in (1, 40):
    rx = np.ones((n, 3), np.float32)
    s.gradients(sc.tx, rx, none, prm)
    s.adjoint(sc.tx, rx, none, prm, theta=s.theta(sc.xf[0]), pcoh_bar=np.ones(n))
assert L.fake_stale() == before, L.fake_stale() - before
s.close()
""")
