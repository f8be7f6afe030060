"""How many diffraction candidates reach the FP64 stage, on the GPU."""
import pytest

from paper_2112_07115_gb300 import dcem, scenes
from tests import parity as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stream():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2112_07115_gb300 import build
    build.build()
    return torch.cuda.current_stream().cuda_stream


def _scene(stream, sc, order, refl, n_rays=5_000):
    s = dcem.Scene.from_scene(sc, stream=stream)
    s.set_rays(scenes.fibonacci_sphere(n_rays))
    s.set_diffraction(True)
    if refl:
        s.set_diffraction_reflections(refl)
    s.set_diffraction_order(order)
    if sc.nobj:
        s.update_transforms(sc.xf[0])
    return s


@pytest.mark.parametrize("vehicles,length,order,refl,count", [(40, 1000.0, 3, 0, 131), (60, 2000.0, 2, 1, 3378)])
def test_chains_off_their_edges_are_dropped_in_fp32(stream, vehicles, length, order, refl, count):
    """Along a road the Keller points of most chains lie far off their edges,
    where the length is nearly flat: the FP32 estimate follows them there and
    rejects the chain. `count` chains are left when it does (a tenth more is
    allowed for changes of rounding)."""
    sc = scenes.highway(n_frames=1, n_vehicles=vehicles, n_rays=5_000, length=length)
    s = _scene(stream, sc, order, refl)
    f = s.trace(sc.tx, sc.rx[0], P.gpu_params(sc))
    assert 0 < f.stats["diff_candidates"] <= 1.1 * count
    s.close()
