"""How many diffraction candidates reach the FP64 stage, and the forms that
stage takes with their number, on the GPU."""
import numpy as np
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


def _ids(p):
    p = p[p["ray"] < 0]
    return sorted((int(q["depth"]), *q["tri"].tolist(), q["len_m"], q["amp_re"], q["amp_im"]) for q in p)


@pytest.mark.parametrize("where,nrx,order,refl", [("city", 64, 1, 2), ("city", 64, 2, 2), ("city", 600, 1, 2),
                                                  ("road", 200, 1, 2)])
def test_forms_of_the_exact_stage_agree(stream, where, nrx, order, refl):
    """A receiver alone has few candidates: none is tested for occlusion and
    each takes four lanes. The 64 receivers' go through the occlusion test; the
    600 receivers', and without that test the road's, take one lane each. The
    paths are the same, bit for bit."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sc = scenes.city_blocks(n_rx=nrx) if where == "city" else scenes.highway(n_frames=1)
    s = _scene(stream, sc, order, refl)
    prm = P.gpu_params(sc, max_refl=3)
    rx = np.asarray(sc.rx[0])
    assert rx.shape[0] == nrx
    whole = s.trace(sc.tx, rx, prm)
    n = whole.stats["diff_candidates"]
    one_lane = where == "road" or nrx > 64
    assert (n > 128 * sms) == one_lane
    alone = 0
    for r in range(nrx):
        one = s.trace(sc.tx, rx[r:r + 1], prm)
        assert where == "road" or one.stats["diff_candidates"] <= 16 * sms
        alone += one.stats["diff_candidates"]
        assert _ids(one.paths) == _ids(whole.paths[whole.paths["rx"] == r]), r
    # the candidates are the receivers' own: untested there are as many together as alone, tested fewer
    assert alone > 16 * sms and (alone > n if where == "city" else alone == n)
    s.close()


def _road(pieces):
    """The highway with its barriers in `pieces` stretches, each a little further out: more planes, no more walls."""
    sc = scenes.highway(n_frames=1, n_vehicles=100, n_rays=5_000)
    t = np.array(sc.tris, np.float32).reshape(-1, 3, 3)
    wall = (np.asarray(sc.tri_obj) < 0) & (t[:, :, 2].max(1) > 0.1)
    k = np.minimum((t[:, :, 0].mean(1) / 2000.0 * pieces).astype(int), pieces - 1)
    t[wall, :, 1] += 0.1 * k[wall, None]
    sc.tris = t.reshape(np.asarray(sc.tris).shape)
    return sc


@pytest.mark.parametrize("where", ["road", "road in pieces", "city"])
def test_open_scenes_are_told_by_what_their_walls_hide(stream, where):
    """Whether the tests of what is hidden are made depends on how much is, not
    on the number of planes: not along a road, however many pieces its barriers
    have, but among buildings. (Untested, the receivers have as many candidates
    together as alone.)"""
    sc = scenes.city_blocks(n=4, n_rx=100) if where == "city" else _road(8 if "pieces" in where else 1)
    s = _scene(stream, sc, 1, 2)
    prm = P.gpu_params(sc, max_refl=3)
    rx = np.asarray(sc.rx[0])
    whole = s.trace(sc.tx, rx, prm)
    alone = 0
    for r in range(rx.shape[0]):
        one = s.trace(sc.tx, rx[r:r + 1], prm)
        alone += one.stats["diff_candidates"]
        assert _ids(one.paths) == _ids(whole.paths[whole.paths["rx"] == r]), r
    n = whole.stats["diff_candidates"]
    assert n < alone if where == "city" else n == alone
    s.close()
