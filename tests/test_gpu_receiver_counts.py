"""Receiver counts around the sizes at which the capture kernel's shared memory
(the stacks, the staged receivers and their tree, and its own arrays) passes
the 48 KB a launch gets without asking for more, and the largest staged count.
Each in a process of its own: a kernel keeps the limit that an earlier call
raised."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import sys
import numpy as np
from paper_2112_07115_gb300 import dcem, scenes
sc = scenes.toy_street()
n = int(sys.argv[1])
s = dcem.Scene.from_scene(sc)
s.set_rays(scenes.fibonacci_sphere(2_000))
s.update_transforms(sc.xf[0])
rx = np.stack([np.linspace(-40, 40, n), np.linspace(-9, 9, n), np.full(n, 1.5)], 1).astype(np.float32)
f = s.trace(sc.tx, rx, dcem.default_params(max_refl=sc.max_refl, freq_hz=sc.freq_hz))
assert f.paths.shape[0] > 0 and np.isfinite(f.p_coh_dbm).any()
s.close()
"""


@pytest.mark.parametrize("nrx", [1, 316, 317, 390, 391, 1024, 1025])
def test_first_frame_of_a_process(nrx):
    r = subprocess.run([sys.executable, "-c", CHILD, str(nrx)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
