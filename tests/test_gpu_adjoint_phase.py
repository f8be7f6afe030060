"""The adjoint kernel's path lengths are those of a plain FP64 evaluation, as
the forward-mode kernel's: at 28 GHz the phase is 587 radians a metre, so one
unit in the last place of a length of 250 m or more (5.7e-14 m) moves the field
by 3.3e-11 of itself."""
import numpy as np
import pytest

from paper_2112_07115_gb300 import dcem, scenes
from tests import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("freq", [28e9, 5.9e9])
def test_field_of_single_paths_equals_forward_mode(freq):
    """Every path at a receiver of its own. With equal lengths the two fields
    differ by the rounding of some hundred operations on unit vectors and
    coefficients: 100 x 2^-53 = 1.1e-14 of the field, taken ten times."""
    import torch
    sc = scenes.urban_gradient(n_frames=1, blocks=3, parcels=4, n_rx=60, n_vehicles=40, n_rays=100_000)
    s = dcem.Scene.from_scene(sc, stream=torch.cuda.current_stream().cuda_stream)
    s.set_rays(scenes.fibonacci_sphere(100_000))
    s.update_transforms(sc.xf[0])
    prm = P.gpu_params(sc, max_refl=4, freq_hz=freq)
    rec = s.trace(sc.tx, sc.rx[0], prm).paths
    assert rec.shape[0] >= 50
    rx = np.asarray(sc.rx[0], np.float32)[rec["rx"]]
    rec = rec.copy()
    rec["rx"] = np.arange(rec.shape[0])
    e = s.adjoint(sc.tx, rx, rec, prm)[0]
    f = s.gradients(sc.tx, rx, rec, prm)[0]
    assert np.all(np.abs(f) > 0)
    assert np.max(np.abs(e - f) / np.abs(f)) <= 1.1e-13
    s.close()
