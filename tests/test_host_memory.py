"""The host code's memory handling, without a GPU: the library's own objects
linked to a stand-in for the CUDA runtime (host_runtime.cu) in which kernels
do nothing. Host buffers outlive the asynchronous copies made from them, and
after an allocation that failed, whichever it was, a repeated call finds every
buffer that its kernels take."""
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


@pytest.mark.parametrize("order,refl", [(1, 2), (3, 1), (3, 3)])
def test_every_allocation_may_fail(stand_in, order, refl):
    _child(stand_in, f"""
order, refl = {order}, {refl}
sc = scenes.city_blocks(n=2, n_rx=30)
prm = dcem.default_params(max_refl=3)
rx = np.asarray(sc.rx[0], np.float32)

def attempt(step):
    # the call, and once more when an allocation failed
    try:
        return step()
    except dcem.DcemError as e:
        assert e.status == dcem.ERR_NOMEM, e
        L.fake_fail_alloc(0)
        return step()

def steps(s):
    yield lambda: s.set_rays(scenes.fibonacci_sphere(200))
    yield lambda: s.set_diffraction(True)
    yield lambda: s.set_diffraction_reflections(refl)
    yield lambda: s.set_diffraction_order(order)
    yield lambda: s.trace(sc.tx, rx[:10], prm)
    def more():
        L.fake_overflow(1, 5000, 40000, 9000, 9000)
        s.trace(sc.tx, np.repeat(rx, 20, 0), prm)
    yield more
    yield lambda: s.trace(sc.tx, rx[:10], prm)
    yield lambda: s.gradients(sc.tx, rx[:9], np.zeros(3, dcem.PATH_DTYPE), prm)

n, seen = 1, 0
while True:
    s = dcem.Scene.from_scene(sc)
    first = L.fake_allocs()
    for step in steps(s):
        # the n-th allocation from here on fails, wherever that is
        L.fake_fail_alloc(max(0, n - (L.fake_allocs() - first)))
        attempt(step)
    done = L.fake_allocs() - first
    s.close()
    assert L.fake_bad() == 0, (n, L.fake_bad_text())
    if done < n:
        break
    n, seen = n + 1, done
assert seen > 60, seen
""")
