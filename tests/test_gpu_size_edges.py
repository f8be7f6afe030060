"""Sizes at which the kernels change their way of working, on the GPU: records
per receiver of the allocation-free reduction, the frame reduction's links and
records (a warp or a block per link, mapped or copied host results), the two
forms of the validation, few rays spread over all SMs, diffraction candidates
with and without the occlusion test, and the adjoint's paths per warp and
parameters. Each side of an edge must give the bits of the other (or of the
same sum formed on the host in the same order)."""
import ctypes as C

import numpy as np
import pytest

from paper_2112_07115_gb300 import dcem, scenes
from tests import parity as P
from tests.test_gpu_links import _compare_links_vs_single, _tx_set

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cuda():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2112_07115_gb300 import build
    build.build()
    torch.cuda.set_device(0)
    return torch


# ---- the allocation-free reduction ----
def _ordered_sums(key, amp, rx, nrx):
    """Sums as the kernels order them: sorted position i to partial sum i mod
    256, in order, then a binary tree over the 256."""
    out = np.zeros((nrx, 3))
    order = np.lexsort((np.arange(key.size), key, rx))
    start = np.searchsorted(rx[order], np.arange(nrx + 1))
    for r in range(nrx):
        i = order[start[r]:start[r + 1]]
        v = np.stack([amp[i].real, amp[i].imag, amp[i].real * amp[i].real + amp[i].imag * amp[i].imag], 1)
        part = np.zeros((256, 3))
        for j in range(0, len(i), 256):
            part[:len(v[j:j + 256])] += v[j:j + 256]
        h = 128
        while h:
            part[:h] += part[h:2 * h]
            h //= 2
        out[r] = part[0]
    return out


@pytest.mark.parametrize("nrx,counts", [
    (1, [0]), (1, [1]), (1, [4096]),
    (13, [0, 1, 2, 31, 32, 33, 63, 64, 65, 255, 256, 257, 300]),
    (511, [3]), (512, [17]), (513, [32, 0, 33]),
    (1025, [64, 63]), (4096, [16]), (4095, [8, 0, 40, 1])])
def test_noalloc_records_per_receiver(cuda, nrx, counts):
    torch = cuda
    rng = np.random.default_rng(nrx)
    cnt = np.resize(counts, nrx)
    rx = np.repeat(np.arange(nrx), cnt)
    n = rx.size
    rec = np.zeros(max(n, 1), dcem.PATH_DTYPE)[:n]
    rec["rx"] = rx[rng.permutation(n)]
    rec["key"] = rng.integers(0, 1 << 63, n, dtype=np.uint64) if n < 200 else rng.integers(0, 50, n, dtype=np.uint64)
    rec["amp_re"], rec["amp_im"] = rng.normal(size=n), rng.normal(size=n)
    dev = torch.device("cuda", 0)
    buf = torch.from_numpy(np.frombuffer(rec.tobytes() or b"\0", np.uint8).copy()).to(dev)
    f, pc, pi = (torch.full((nrx, k), float("nan"), dtype=torch.float64, device=dev) for k in (2, 1, 1))
    st = torch.cuda.current_stream().cuda_stream
    rc = dcem.dcem_reduce_paths_noalloc(buf.data_ptr(), n, nrx, 2.0, f.data_ptr(), pc.data_ptr(), pi.data_ptr(), st)
    assert rc == dcem.OK, dcem.status_string(rc)
    s = _ordered_sums(rec["key"], rec["amp_re"] + 1j * rec["amp_im"], rec["rx"], nrx)
    assert np.array_equal(f.cpu().numpy(), s[:, :2])
    with np.errstate(divide="ignore"):
        wc = 10 * np.log10(2.0 * (s[:, 0] ** 2 + s[:, 1] ** 2)) + 30
        wi = 10 * np.log10(2.0 * s[:, 2]) + 30
    # two FP64 logarithms of equal arguments: a few units in the last place of up to 400 dB
    for got, want in ((pc, wc), (pi, wi)):
        g = got.cpu().numpy()[:, 0]
        fin = np.isfinite(want)
        assert np.array_equal(np.isfinite(g), fin) and np.all(np.abs(g[fin] - want[fin]) <= 1e-12)


# ---- frames: links, records and the two validation forms ----
def _rx_grid(n):
    k = int(np.ceil(np.sqrt(n)))
    g = np.stack(np.meshgrid(np.linspace(-40, 40, k), np.linspace(-9, 9, k), indexing="ij"), -1).reshape(-1, 2)[:n]
    return np.concatenate([g, np.full((n, 1), 1.5)], 1).astype(np.float32)


@pytest.mark.parametrize("ntx,nrx", [(1, 1), (4, 33), (4, 256), (4, 257), (4, 512), (4, 513), (8, 640)])
def test_host_results_equal_device_results(cuda, ntx, nrx):
    """Host results (the first records and the links of smaller frames through
    mapped memory, the rest copied) equal the device results, records past
    n_paths stay as they were, and a short buffer gets its part."""
    torch = cuda
    sc = scenes.toy_street()
    txs, rx = _tx_set(sc, ntx, seed=3), _rx_grid(nrx)
    s = dcem.Scene.from_scene(sc, stream=torch.cuda.current_stream().cuda_stream)
    s.set_ray_sets([scenes.fibonacci_sphere(4_000)] * ntx)
    s.update_transforms(sc.xf[0])
    prm = P.gpu_params(sc)
    room, nl = 40_000, ntx * nrx
    size = C.sizeof(dcem.Path)
    dev = torch.device("cuda", 0)
    out = []
    for kind in (dcem.PTR_DEVICE, dcem.PTR_HOST):
        where = dev if kind == dcem.PTR_DEVICE else torch.device("cpu")
        f = torch.full((4, nl), -7.0, dtype=torch.float64, device=where)
        paths = torch.full((room * size,), 0x5a, dtype=torch.uint8, device=where)
        r = dcem.Result()
        r.ptr_kind, r.max_paths, r.paths = kind, room, paths.data_ptr()
        r.field, r.p_coh_dbm, r.p_inc_dbm = f[0].data_ptr(), f[2].data_ptr(), f[3].data_ptr()
        assert dcem.dcem_trace_links(s.h, txs, rx, prm, r) == dcem.OK
        out.append((r.n_paths, f.cpu().numpy(), paths.cpu().numpy()))
    (nd, fd, pd), (nh, fh, ph) = out
    assert nd == nh > 0 and np.array_equal(fd, fh) and np.array_equal(pd, ph)
    assert np.all(ph[nh * size:] == 0x5a)
    for short in (1, max(1, nh // 2)):
        fr = s.trace_links(txs, rx, prm, max_paths=short, raise_on_error=False)
        assert fr.status == (dcem.OK if short >= nh else dcem.ERR_CAPACITY)
        assert fr.paths.tobytes() == ph[:min(short, nh) * size].tobytes()
    s.close()


@pytest.mark.parametrize("nrx", [256, 257])
@pytest.mark.parametrize("mode", [dcem.MODE_FULL, dcem.MODE_COHERENT])
def test_validation_forms_agree(cuda, nrx, mode):
    """4 x 256 links take one validation kernel, 4 x 257 three; a single
    transmitter's frames take the one either way."""
    sc = scenes.toy_street()
    _compare_links_vs_single(cuda, sc, _tx_set(sc, 4, seed=9), [3_000, 2_001, 4_000, 999], range(0, 3), mode=mode,
                             rx=_rx_grid(nrx))


def test_more_links_than_one_level_of_sums(cuda):
    """33 x 2048 links: the groups' path counts are scanned before the
    reduction."""
    sc = scenes.toy_street()
    _compare_links_vs_single(cuda, sc, _tx_set(sc, 33, seed=5), [400 + t for t in range(33)], [0], rx=_rx_grid(2048))


# ---- few rays ----
@pytest.mark.parametrize("n", [1, 31, 33, 64, 65, 4864, 4865, 9729])
def test_few_rays_over_all_sms(cuda, n):
    """The shared-memory kernel's CTAs shrink with the number of rays; the last
    chunk of 32 rays may be short. The binary-node kernel gives the same."""
    torch = cuda
    sc = scenes.toy_street()
    rays = scenes.fibonacci_sphere(10_000)[:n]
    frames = []
    for kernel in (1, 0):
        s = dcem.Scene.from_scene(sc, stream=torch.cuda.current_stream().cuda_stream)
        s.set_rays(rays)
        s.set_trace_config(kernel)
        s.update_transforms(sc.xf[0])
        fr = s.trace(sc.tx, sc.rx[0], P.gpu_params(sc))
        assert fr.stats["trace_kernel"] == kernel
        frames.append((fr, s.ray_log()))
        s.close()
    (a, la), (b, lb) = frames
    assert a.paths.tobytes() == b.paths.tobytes() and np.array_equal(a.p_coh_dbm, b.p_coh_dbm)
    for x, y in zip(la, lb):
        assert np.asarray(x).tobytes() == np.asarray(y).tobytes()


# ---- diffraction candidates ----
@pytest.mark.parametrize("order,refl", [(1, 0), (1, 1), (1, 2), (2, 1), (3, 0)])
def test_diffraction_of_many_receivers_equals_one_by_one(cuda, order, refl):
    """A frame of 40 receivers (enough candidates for the occlusion test) has
    the paths of 40 frames of one receiver (few enough to go without it)."""
    torch = cuda
    sc = scenes.city_blocks(n=4, n_rx=40)
    s = dcem.Scene.from_scene(sc, stream=torch.cuda.current_stream().cuda_stream)
    s.set_rays(scenes.fibonacci_sphere(5_000))
    s.set_diffraction(True)
    if refl:
        s.set_diffraction_reflections(refl)
    if order > 1:
        s.set_diffraction_order(order)
    prm = P.gpu_params(sc, max_refl=max(4, order))
    whole = s.trace(sc.tx, sc.rx[0], prm)
    for r in range(40):
        one = s.trace(sc.tx, sc.rx[0][r:r + 1], prm)
        ids = lambda p: sorted((int(q["depth"]), *q["tri"].tolist(), q["len_m"], q["amp_re"], q["amp_im"]) for q in p)
        want = whole.paths[(whole.paths["rx"] == r) & (whole.paths["ray"] < 0)]
        assert ids(one.paths[one.paths["ray"] < 0]) == ids(want), r
    assert (whole.paths["ray"] < 0).sum() > 0
    s.close()


# ---- the adjoint ----
@pytest.mark.parametrize("copies", [1, 120, 400])
def test_adjoint_of_repeated_paths(cuda, copies):
    """Several paths per warp: every path `copies` times gives `copies` times
    the field and its derivatives (sums of equal terms in other orders, each
    addition within 2^-53 of the sum of magnitudes)."""
    torch = cuda
    sc = scenes.toy_street()
    s = dcem.Scene.from_scene(sc, stream=torch.cuda.current_stream().cuda_stream)
    s.set_rays(scenes.fibonacci_sphere(8_000))
    s.update_transforms(sc.xf[0])
    prm = P.gpu_params(sc)
    paths = s.trace(sc.tx, sc.rx[0], prm).paths
    assert paths.shape[0] >= 8
    e1, _, d1, _, _ = s.adjoint(sc.tx, sc.rx[0], paths, prm)
    e, _, d, _, _ = s.adjoint(sc.tx, sc.rx[0], np.repeat(paths, copies), prm)
    single = np.zeros(sc.nrx)
    np.add.at(single, paths["rx"], np.hypot(paths["amp_re"], paths["amp_im"]))
    bound = paths.shape[0] * copies * 2.0 ** -52
    assert np.all(np.abs(e - copies * e1) <= bound * copies * single)
    for r in range(sc.nrx):
        one = np.zeros(d.shape[1])
        for p in paths[paths["rx"] == r]:
            one += np.abs(s.adjoint(sc.tx, sc.rx[0], p.reshape(1), prm)[2][r])
        assert np.all(np.abs(d[r] - copies * d1[r]) <= bound * copies * one + 1e-300), r
    s.close()


def test_adjoint_of_many_objects(cuda):
    """More parameters than a receiver's sums have shared memory for: the
    derivatives equal the forward-mode ones (two FP64 evaluations in different
    orders, 1e-8 of the receiver's largest)."""
    torch = cuda
    sc = scenes.toy_street()
    extra = 1300
    k = np.arange(extra, dtype=np.float32)
    far = np.stack([np.stack([500 + k, 500 + 0 * k, 5 + 0 * k], 1), np.stack([500.5 + k, 500 + 0 * k, 5 + 0 * k], 1),
                    np.stack([500 + k, 500.5 + 0 * k, 5 + 0 * k], 1)], 1).astype(np.float32)
    tris = np.concatenate([np.asarray(sc.tris, np.float32).reshape(-1, 3, 3), far])
    obj = np.concatenate([sc.tri_obj, sc.nobj + np.arange(extra)]).astype(np.int32)
    mat = np.concatenate([sc.tri_mat, np.zeros(extra)]).astype(np.int32)
    eye = np.tile(np.array([1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0], np.float32), (extra, 1))
    xf = np.concatenate([np.asarray(sc.xf[0], np.float32).reshape(-1, 12), eye])
    s = dcem.Scene(tris, mat, sc.materials, obj, sc.nobj + extra, torch.cuda.current_stream().cuda_stream)
    s.set_rays(scenes.fibonacci_sphere(8_000))
    s.update_transforms(xf)
    prm = P.gpu_params(sc)
    paths = s.trace(sc.tx, sc.rx[0], prm).paths
    assert paths.shape[0] >= 8
    e, _, d, dp, _ = s.adjoint(sc.tx, sc.rx[0], paths, prm)
    ef, df, _ = s.gradients(sc.tx, sc.rx[0], paths, prm)
    assert d.shape[1] > 2560
    for r in range(sc.nrx):
        assert abs(e[r] - ef[r]) <= 1e-9 * abs(ef[r]) + 1e-300
        assert np.abs(d[r] - df[r]).max() <= 1e-8 * np.abs(df[r]).max() + 1e-300, r
    s.close()
