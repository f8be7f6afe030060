"""What a user of the tracer has it do, as measurable cases.

Every case goes through the documented entry points of the binding
(`dcem.Scene`, `dcem.dcem_trace_links`, `dcem.Batch`, `dcem.path_power`,
`dcem.dcem_reduce_paths_noalloc`) with host transforms and receivers and
page-locked outputs that the caller owns, the end-to-end form of the
benchmark. The scenes are the seeded generators of `scenes.py` at the sizes
the benchmark and the tests use.

Kinds
  street     one small vehicular scene per call (latency: 58 triangles)
  highway    the 2 km road, roof or roadside receivers, optionally with
             edge diffraction
  links      the urban grid with several transmitters in one call
  batch      independent scenes traced together
  office     indoor, transmission through walls (full frames by definition)
  city       box buildings, diffraction with reflections or wedge chains
  gradient   differentiable received power over a frame's paths
  reduce     the allocation-free sum of given path records

A pass of the kinds that trace is `frames` consecutive frames, each an update
of the moving objects and a trace; with two frames the passes alternate
between two neighbouring time steps, the steady state of a coherent sequence.
"""
import functools
import math

import numpy as np
import torch

from paper_2112_07115_gb300 import dcem, scenes

MODES = {"full": dcem.MODE_FULL, "coherent": dcem.MODE_COHERENT, "sticky": dcem.MODE_STICKY}
# path records a caller makes room for, per scene
PATHS = {"street": 512, "highway": 4096, "office": 8192, "city": 4096, "links": 131_072, "batch": 16_384}


def listed():
    return [
        # a small street corner polled frame by frame: launches and latency
        {"name": "street_full", "kind": "street", "rays": 10_000, "refl": 3, "mode": "full", "frames": 1,
         "freq": 28e9, "prec": 0},
        # the same as a drive, with reuse between frames
        {"name": "street_coherent", "kind": "street", "rays": 10_000, "refl": 3, "mode": "coherent", "frames": 2,
         "freq": 28e9, "prec": 0},
        # the headline: one highway frame retraced in full
        {"name": "highway_full", "kind": "highway", "rays": 1_000_000, "refl": 4, "mode": "full", "frames": 1,
         "freq": 28e9, "prec": 0, "vehicles": 200, "roadside": 0, "order": 0, "refl_diff": 0},
        # the headline in coherent mode
        {"name": "highway_coherent", "kind": "highway", "rays": 1_000_000, "refl": 4, "mode": "coherent", "frames": 2,
         "freq": 28e9, "prec": 0, "vehicles": 200, "roadside": 0, "order": 0, "refl_diff": 0},
        # a city's roadside units against all vehicles in one call: the largest traversal
        {"name": "urban_links", "kind": "links", "blocks": 10, "parcels": 4, "vehicles": 1000, "tx": 16,
         "rays_lo": 65_536, "rays_hi": 1_048_576, "static_rx": 96, "refl": 5, "mode": "full", "frames": 1},
        # several independent deployments of uneven size stepped together
        {"name": "scene_batch", "kind": "batch", "scenes": 7, "tris_hi": 40_000, "vehicles_hi": 300, "tx_hi": 4,
         "rays_hi": 262_144, "refl": 4, "mode": "coherent", "frames": 2},
        # indoor coverage with wall losses
        {"name": "office", "kind": "office", "rays": 1_000_000, "refl": 2, "trans": 2, "rooms_x": 4, "rooms_y": 3,
         "carts": 4, "mode": "full", "frames": 1},
        # the highway with every vehicle and barrier edge diffracting
        {"name": "highway_diffraction", "kind": "highway", "rays": 1_000_000, "refl": 4, "mode": "coherent",
         "frames": 2, "freq": 28e9, "prec": 0, "vehicles": 200, "roadside": 0, "order": 1, "refl_diff": 0},
        # two reflections and one diffraction per path, the paper's evaluation limits
        {"name": "city_diffraction", "kind": "city", "n": 8, "rx": 64, "rays": 200_000, "refl": 3, "order": 1,
         "refl_diff": 2},
        # rooftop and corner chains of up to three wedges
        {"name": "city_chains", "kind": "city", "n": 8, "rx": 64, "rays": 200_000, "refl": 3, "order": 3,
         "refl_diff": 0},
        # received power and its gradient by materials and vehicle positions
        {"name": "gradient", "kind": "gradient", "blocks": 6, "vehicles": 300, "rx": 256, "rays": 500_000, "refl": 4,
         "way": "power"},
        # a real-time loop's sums over path records it holds
        {"name": "reduce_noalloc", "kind": "reduce", "paths": 16_384, "rx": 1024},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["street", "highway", "links", "batch", "office", "city", "gradient", "reduce", "highway",
                       "links"])
    mode = rng.choice(["full", "coherent", "coherent", "sticky"])
    frames = 1 if mode == "full" else 2
    freq, prec = rng.choice([28e9, 5.9e9, 30e9]), rng.choice([0, 0, 1])
    if kind == "street":
        return {"kind": kind, "rays": _log(rng, 1_000, 200_000), "refl": rng.randint(1, 5), "mode": mode,
                "frames": frames, "freq": freq, "prec": prec}
    if kind == "highway":
        order = rng.choice([0, 0, 0, 1])
        return {"kind": kind, "rays": _log(rng, 50_000, 1_000_000), "refl": rng.randint(2, 6), "mode": mode,
                "frames": frames, "freq": freq, "prec": prec, "vehicles": rng.randint(20, 200),
                "roadside": rng.choice([0, 0, rng.randint(7, 200)]), "order": order,
                "refl_diff": rng.randint(0, 2) if order else 0}
    if kind == "links":
        blocks = rng.randint(3, 10)
        return {"kind": kind, "blocks": blocks, "parcels": rng.randint(2, 4), "vehicles": rng.randint(5, 10 * blocks),
                "tx": rng.randint(2, 16), "rays_lo": 32_768, "rays_hi": _log(rng, 65_536, 1_048_576),
                "static_rx": rng.randint(4, 96), "refl": rng.randint(2, 5), "mode": mode, "frames": frames}
    if kind == "batch":
        mode = rng.choice(["full", "coherent"])
        return {"kind": kind, "scenes": rng.randint(2, 7), "tris_hi": _log(rng, 5_000, 40_000),
                "vehicles_hi": rng.randint(30, 300), "tx_hi": rng.randint(1, 4), "rays_hi": _log(rng, 32_768, 262_144),
                "refl": rng.randint(2, 4), "mode": mode, "frames": 1 if mode == "full" else 2}
    if kind == "office":
        return {"kind": kind, "rays": _log(rng, 30_000, 1_000_000), "refl": rng.randint(1, 2),
                "trans": rng.randint(1, 2), "rooms_x": rng.randint(2, 6), "rooms_y": rng.randint(1, 4),
                "carts": rng.randint(1, 8), "mode": "full", "frames": 1}
    if kind == "city":
        order = rng.randint(1, 3)
        return {"kind": kind, "n": rng.randint(3, 8), "rx": rng.randint(5, 64), "rays": _log(rng, 20_000, 200_000),
                "refl": max(order, rng.randint(2, 4)), "order": order, "refl_diff": {1: rng.randint(0, 2), 2: rng.randint(0, 1), 3: 0}[order]}
    if kind == "gradient":
        blocks = rng.randint(3, 6)
        return {"kind": kind, "blocks": blocks, "vehicles": rng.randint(5, 30 * blocks), "rx": rng.randint(17, 256),
                "rays": _log(rng, 100_000, 500_000), "refl": rng.randint(2, 4), "way": rng.choice(["power", "forward"])}
    return {"kind": kind, "paths": _log(rng, 50, 65_536), "rx": _log(rng, 33, 4096)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=48)
def _rays(n):
    return scenes.fibonacci_sphere(n)


def _scene(case, seed):
    """The generated scene of a case (of the kinds that have one)."""
    kind = case["kind"]
    if kind == "street":
        sc = scenes.toy_street(seed=1 + seed % 100_003, n_frames=3, n_rays=case["rays"], max_refl=case["refl"],
                               freq_hz=case["freq"])
        # the pedestrians stand where they stand; the layout's own points are one choice
        g = np.random.default_rng([seed, 12])
        sc.rx[...] += g.uniform([-3.0, -1.0, -0.2], [3.0, 1.0, 0.2], (sc.nrx, 3)).astype(np.float32)
        return sc
    if kind == "highway":
        return scenes.highway(seed=seed % 100_003, n_frames=3, n_vehicles=case["vehicles"], n_rays=case["rays"],
                              max_refl=case["refl"], freq_hz=case["freq"], roadside_rx=case["roadside"])
    if kind == "links":
        return scenes.urban_grid(seed=seed % 100_003, blocks=case["blocks"], parcels=case["parcels"],
                                 n_vehicles=case["vehicles"], n_tx=case["tx"],
                                 budgets=(case["rays_lo"], case["rays_hi"]), n_static_rx=case["static_rx"],
                                 n_frames=3, max_refl=case["refl"])
    if kind == "office":
        return scenes.office(seed=seed % 100_003, rooms_x=case["rooms_x"], rooms_y=case["rooms_y"],
                             n_carts=case["carts"], n_frames=3, n_rays=case["rays"], max_refl=case["refl"],
                             max_trans=case["trans"])
    if kind == "city":
        return scenes.city_blocks(n=case["n"], seed=seed % 100_003, n_rx=case["rx"], n_rays=case["rays"],
                                  max_refl=case["refl"])
    if kind == "gradient":
        sc = scenes.urban_gradient(seed=seed % 100_003, blocks=case["blocks"], parcels=4, n_rx=case["rx"],
                                   n_vehicles=case["vehicles"], n_rays=case["rays"], max_refl=case["refl"],
                                   n_frames=2)
        # off the corner points that transmitter and receivers share (a vertical path has no polarisation)
        g = np.random.default_rng([seed, 13])
        sc.rx[...] += g.uniform(-0.5, 0.5, (sc.nrx, 3)).astype(np.float32)
        return sc
    raise ValueError(kind)


def _batch_scenes(case, seed):
    """Urban grids of sizes spread evenly over the logarithm from 1,000
    triangles, 10 vehicles and one transmitter to the case's largest, the
    three mixed among the scenes."""
    n, out = case["scenes"], []
    for i in range(n):
        a, b, c = i / max(n - 1, 1), (3 * i % n) / max(n - 1, 1), (2 * i % n) / max(n - 1, 1)
        target = 1_000 * (case["tris_hi"] / 1_000) ** a
        blocks = max(2, round(math.sqrt(target / 1_000)))
        parcels = max(1, round(math.sqrt(target / 30.0) / blocks))
        vehicles = int(min(0.01 * 8 * (blocks + 1) * (100 * blocks + 20), 10 * (case["vehicles_hi"] / 10) ** b))
        out.append(scenes.urban_grid(seed=1000 * (seed % 100_003) + i, blocks=blocks, parcels=parcels,
                                     n_vehicles=vehicles, n_tx=1 + round(c * (case["tx_hi"] - 1)),
                                     budgets=(16_384, case["rays_hi"]), n_static_rx=8, n_frames=3,
                                     max_refl=case["refl"]))
    return out


def _params(case, sc):
    return dcem.default_params(max_refl=sc.max_refl, freq_hz=sc.freq_hz, mode=MODES[case.get("mode", "full")],
                               prec=case.get("prec", 0), tx_power_w=sc.meta.get("tx_power_w", 5.0))


def _outputs(case, links):
    """Per frame the page-locked arrays of scenes with these link counts, and
    their result structs. Records past a frame's path count stay zero."""
    def pinned(n, t):
        return torch.zeros(n, dtype=t, pin_memory=True).numpy()
    out, room = [], PATHS[case["kind"]]
    for _ in range(case.get("frames", 1)):
        o = {"field": pinned(2 * sum(links), torch.float64), "p_coh": pinned(sum(links), torch.float64),
             "p_inc": pinned(sum(links), torch.float64), "paths": [], "results": []}
        at = 0
        for n in links:
            raw = pinned(room * dcem.PATH_DTYPE.itemsize, torch.uint8).reshape(room, -1)
            # rx .. key as 32-bit words, length and delay, amplitude, interaction points
            o["paths"].append([raw.view(np.int32)[:, :18], raw.view(np.float64)[:, 9:11],
                               raw.view(np.float64)[:, 11:13], raw.view(np.float32)[:, 26:56]])
            r = dcem.Result()
            r.ptr_kind, r.max_paths, r.paths = dcem.PTR_HOST, room, raw.ctypes.data
            r.field = o["field"][2 * at:].ctypes.data
            r.p_coh_dbm, r.p_inc_dbm = o["p_coh"][at:].ctypes.data, o["p_inc"][at:].ctypes.data
            o["results"].append(r)
            at += n
        out.append(o)
    return out


def prepare(case, seed):
    kind = case["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    st = {"case": dict(case)}
    if kind == "reduce":
        n, nrx = case["paths"], case["rx"]
        g = np.random.default_rng([seed, 11])
        rec = np.zeros(n, dcem.PATH_DTYPE)
        rec["rx"] = g.integers(0, nrx, n)
        rec["depth"] = g.integers(0, 5, n)
        rec["key"] = g.integers(1, 1 << 63, n).astype(np.uint64)
        rec["len_m"] = g.uniform(5.0, 1500.0, n)
        amp = 0.0107 / (4 * np.pi) / rec["len_m"] * g.uniform(0.05, 1.0, n)
        ph = g.uniform(0.0, 2 * np.pi, n)
        rec["amp_re"], rec["amp_im"] = amp * np.cos(ph), amp * np.sin(ph)
        dev = torch.device("cuda")
        st["paths"] = torch.from_numpy(rec.view(np.uint8).reshape(n, -1)).to(dev)
        st["field"] = torch.empty(nrx, 2, dtype=torch.float64, device=dev)
        st["pc"] = torch.empty(nrx, dtype=torch.float64, device=dev)
        st["pi"] = torch.empty(nrx, dtype=torch.float64, device=dev)
        st["records"] = rec
        dcem.dcem_reduce_paths_noalloc(None, 0, 0, 5.0, None, None, None, stream)  # the documented set-up call
        return st
    if kind == "batch":
        scs = _batch_scenes(case, seed)
        st["handles"] = []
        for sc in scs:
            s = dcem.Scene.from_scene(sc, stream=stream)
            s.set_ray_sets([_rays(int(b)) for b in sc.meta["budgets"]])
            st["handles"].append(s)
        st["batch"] = dcem.Batch(st["handles"], stream=stream)
        st["scenes"] = scs
        st["prm"] = _params(case, scs[0])
        st["txs"] = [sc.meta["tx"] for sc in scs]
        st["out"] = _outputs(case, [len(t) * sc.nrx for t, sc in zip(st["txs"], scs)])
        return st
    sc = _scene(case, seed)
    s = dcem.Scene.from_scene(sc, stream=stream)
    st["sc"], st["s"], st["prm"] = sc, s, _params(case, sc)
    if kind == "links":
        s.set_ray_sets([_rays(int(b)) for b in sc.meta["budgets"]])
    else:
        s.set_rays(_rays(sc.n_rays))
    if kind == "office":
        s.set_transmission(sc.meta["trans_db"], sc.meta["max_trans"])
    if case.get("order", 0):
        s.set_diffraction(True)
        if case["refl_diff"]:
            s.set_diffraction_reflections(case["refl_diff"])
        s.set_diffraction_order(case["order"])
    st["tx"] = sc.meta["tx"] if kind == "links" else sc.tx
    if kind != "gradient":
        st["out"] = _outputs(case, [len(st["tx"].reshape(-1, 3)) * sc.nrx])
    else:
        s.update_transforms(sc.xf[1])
        st["rx"] = sc.rx[1]
        st["paths"] = s.trace(sc.tx, st["rx"], st["prm"]).paths
        st["theta"] = torch.tensor(s.theta(sc.xf[1]), dtype=torch.float64, device="cuda")
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "reduce":
        rc = dcem.dcem_reduce_paths_noalloc(st["paths"].data_ptr(), case["paths"], case["rx"], 5.0,
                                            st["field"].data_ptr(), st["pc"].data_ptr(), st["pi"].data_ptr(),
                                            torch.cuda.current_stream().cuda_stream)
        if rc != dcem.OK:
            raise dcem.DcemError(rc, "dcem_reduce_paths_noalloc")
        return {"field": st["field"], "p_coh": st["pc"], "p_inc": st["pi"]}
    if kind == "batch":
        b, scs, out = st["batch"], st["scenes"], []
        for f, o in enumerate(st["out"], 1):
            b.update_transforms([sc.xf[f] for sc in scs])
            rc, failed = b.trace_raw(st["txs"], [sc.rx[f] for sc in scs], st["prm"], o["results"])
            if rc != dcem.OK:
                raise dcem.DcemError(rc, f"dcem_batch_trace (scene {failed})")
            out.append({k: o[k] for k in ("field", "p_coh", "p_inc", "paths")})
        return out
    s, sc, prm = st["s"], st["sc"], st["prm"]
    if kind == "gradient":
        if case["way"] == "forward":
            e, de, dp = s.gradients(sc.tx, st["rx"], st["paths"], prm)
            return {"field": e, "dfield": de, "dp": dp}
        theta = st["theta"].clone().requires_grad_(True)
        p = dcem.path_power(s, theta, sc.tx, st["rx"], st["paths"], prm)
        p[torch.isfinite(p)].sum().backward()
        return {"p_coh": p.detach(), "grad": theta.grad}
    out = []
    for f, o in enumerate(st["out"], 1):
        if sc.nobj:
            s.update_transforms(sc.xf[f])
        rc = dcem.dcem_trace_links(s.h, st["tx"], sc.rx[f if sc.nframes > 1 else 0], prm, o["results"][0])
        if rc != dcem.OK:
            raise dcem.DcemError(rc, "dcem_trace_links")
        out.append({k: o[k] for k in ("field", "p_coh", "p_inc", "paths")})
    return out


def work(case):
    """Inputs read once and outputs written once, and the arithmetic of one
    hierarchy descent (20 flops a level, 50 for the triangle) per ray; the
    path counts are not known before the trace and left out."""
    kind = case["kind"]
    if kind == "reduce":
        return {"bytes": 32 * case["paths"] + 32 * case["rx"], "flops": 6 * case["paths"]}
    if kind == "street":
        tris, obj, rx, rays, links = 58, 4, 8, case["rays"], 8
    elif kind == "highway":
        obj = case["vehicles"]
        tris, rx, rays = 2000 + 10 * obj, case["roadside"] or obj, case["rays"]
        links = rx
    elif kind == "links":
        obj = case["vehicles"]
        lo, hi = case["rays_lo"], case["rays_hi"]
        tris = 30 * (case["blocks"] * case["parcels"]) ** 2 + 10 * obj
        rays = int(case["tx"] * ((hi - lo) / math.log(hi / lo) if hi > lo else lo))
        rx = 4 * obj + case["static_rx"]
        links = rx * case["tx"]
    elif kind == "batch":
        def mean(lo, hi):
            return (hi - lo) / math.log(hi / lo)
        n = case["scenes"]
        ntx = n * (1 + case["tx_hi"]) / 2
        tris, obj = n * mean(1_000, case["tris_hi"]), n * mean(10, case["vehicles_hi"])
        rays, rx = ntx * mean(16_384, case["rays_hi"]), 4 * obj + 8 * n
        links = rx * ntx / n
    elif kind == "office":
        tris = 4 * case["rooms_x"] * case["rooms_y"] * 5 + 10 * case["carts"]
        rx = links = 4 * case["rooms_x"] * case["rooms_y"]
        obj, rays = case["carts"], case["rays"]
    elif kind == "city":
        tris, obj, rx, rays, links = 2 + 10 * case["n"] ** 2, 0, case["rx"], case["rays"], case["rx"]
    else:  # gradient: theta and the records in, power and the gradient out; a few paths per receiver
        npar = 18 + 2 * case["vehicles"]
        return {"bytes": 16 * npar + 224 * case["rx"] + 20 * case["rx"], "flops": 2000 * case["rx"]}
    frames = case.get("frames", 1)
    wedges = (12 * case["n"] ** 2 if kind == "city" else 800 + 8 * obj) if case.get("order", 0) else 0
    return {"bytes": frames * (36 * tris + 48 * obj + 12 * rx + 12 * rays + 32 * links),
            "flops": frames * (rays * (20 * math.log2(tris + 2) + 50) + 60.0 * links * wedges)}


# ---------------------------------------------------------------------------
# the same in 64 bits, by brute force in torch
# ---------------------------------------------------------------------------
C0, EPS0, TBIT = 299792458.0, 8.8541878128e-12, 0x40000000


def _world(sc, xf):
    """World vertices (T, 3, 3): the single-precision vertices the geometry is
    defined by, each row fmaf(R0, x, fmaf(R1, y, fmaf(R2, z, t)))."""
    v = sc.tris.astype(np.float32).copy()
    m = sc.tri_obj >= 0
    if m.any():
        M = xf.reshape(-1, 3, 4).astype(np.float64)[sc.tri_obj[m]]
        p = v[m].astype(np.float64)
        for r in range(3):
            acc = np.broadcast_to(M[:, r, 3, None], p.shape[:2])
            for k in (2, 1, 0):
                acc = (M[:, r, k, None] * p[:, :, k] + acc).astype(np.float32).astype(np.float64)
            v[m, :, r] = acc
    return torch.tensor(v, dtype=torch.float64, device="cuda")


class _Tris:
    """Triangles as affine maps to (u, v, w) with w = 0 on the plane."""

    def __init__(self, V):
        self.V = V
        e1, e2 = V[:, 1] - V[:, 0], V[:, 2] - V[:, 0]
        self.n = torch.linalg.cross(e1, e2)
        A = torch.linalg.inv(torch.stack([e1, e2, self.n], dim=2))
        c = -(A @ V[:, 0, :, None])[..., 0]
        self.A, self.c = A, c

    def hits(self, o, d):
        """t of every (ray, triangle) pair, inf where the ray misses."""
        q = [(o @ self.A[:, k].T + self.c[:, k], d @ self.A[:, k].T) for k in range(3)]
        t = -q[2][0] / q[2][1]
        u, v = q[0][0] + t * q[0][1], q[1][0] + t * q[1][1]
        ok = (u >= 0) & (v >= 0) & (u + v <= 1) & (q[2][1] != 0)
        return torch.where(ok, t, torch.full_like(t, math.inf))


def _captures(sc, tri, loss, dirs, tx, rx, prm, n_trans):
    """Distinct (receiver, interactions) of the rays' reception-sphere captures."""
    N, W = prm.max_refl, prm.max_refl + n_trans
    n = dirs.shape[0]
    alpha = float(np.float32(prm.rx_radius_scale)) * math.sqrt(4 * math.pi / n) / math.sqrt(3.0)
    T, found = tri.V.shape[0], []
    step = max(256, int(3e7) // max(T, 1))
    cap = max(256, int(3e7) // max(rx.shape[0], 1))
    o = tx.expand(n, 3).contiguous()
    work = [(o, dirs, torch.zeros(n, device="cuda", dtype=torch.float64),
             torch.full((n, W), -1, device="cuda", dtype=torch.int64), 0, 0)]
    while work:
        o, d, D, seq, nr, nt = work.pop()
        b = nr + nt
        tb, ib = [], []
        for i in range(0, o.shape[0], step):
            t = tri.hits(o[i:i + step], d[i:i + step])
            t[~(t > prm.t_min)] = math.inf
            if b:
                t.scatter_(1, (seq[i:i + step, b - 1] & ~TBIT)[:, None], math.inf)
            m = t.min(dim=1)
            tb.append(m.values)
            ib.append(m.indices)
        t, hit = torch.cat(tb), torch.cat(ib)
        miss = torch.isinf(t)
        tend = torch.where(miss, torch.full_like(t, prm.escape_len), t)
        for i in range(0, o.shape[0], cap):
            w = rx[None] - o[i:i + cap, None]
            s = torch.minimum((w * d[i:i + cap, None]).sum(-1).clamp(min=0), tend[i:i + cap, None])
            far = (w - s[..., None] * d[i:i + cap, None]).square().sum(-1)
            at = torch.nonzero(far <= (alpha * (D[i:i + cap, None] + s)).square())
            found.append(torch.cat([at[:, 1:2], torch.full_like(at[:, :1], b), seq[i:i + cap][at[:, 0]]], 1))
        k = torch.nonzero(~miss)[:, 0]
        o, d, t, hit, D, seq = o[k], d[k], t[k], hit[k], D[k], seq[k]
        p, D = o + t[:, None] * d, D + t
        if nt < n_trans:
            c = torch.nonzero(loss[hit] >= 0)[:, 0]
            if len(c):
                child = seq[c].clone()
                child[:, b] = hit[c] | TBIT
                work.append((p[c], d[c], D[c], child, nr, nt + 1))
        if nr < N and len(k):
            nrm = tri.n[hit]
            r = d - 2 * ((d * nrm).sum(-1) / nrm.square().sum(-1))[:, None] * nrm
            seq = seq.clone()
            seq[:, b] = hit
            work.append((p, r / r.norm(dim=-1, keepdim=True), D, seq, nr + 1, nt))
    return torch.unique(torch.cat(found), dim=0)


def _images(V, n, tx, rx, ids, refl):
    """Path points (K, k + 2, 3) of sequences with one reflect/transmit
    pattern, and which of them cross their triangles in order."""
    k, K = len(refl), ids.shape[0]
    rj = [j for j in range(k) if refl[j]]
    v0 = [V[ids[:, j], 0] for j in range(k)]
    nn = [n[ids[:, j]] for j in range(k)]
    dot = lambda a, b: (a * b).sum(-1, keepdim=True)  # noqa: E731
    img = [tx.expand(K, 3)]
    for j in rj:
        img.append(img[-1] - 2 * dot(img[-1] - v0[j], nn[j]) / dot(nn[j], nn[j]) * nn[j])
    ok = torch.ones(K, dtype=torch.bool, device=V.device)
    XR = [None] * (len(rj) + 2)
    XR[0], XR[-1] = tx.expand(K, 3), rx
    for q in range(len(rj), 0, -1):
        j = rj[q - 1]
        dr = img[q] - XR[q + 1]
        s = dot(v0[j] - XR[q + 1], nn[j]) / dot(dr, nn[j])
        ok = ok & ((s > 0) & (s < 1))[:, 0]
        XR[q] = XR[q + 1] + s * dr
    X, q, prev = [XR[0]], 0, torch.zeros(K, 1, dtype=V.dtype, device=V.device)
    for j in range(k):
        if refl[j]:
            q += 1
            X.append(XR[q])
            prev = torch.zeros_like(prev)
        else:
            dr = XR[q + 1] - XR[q]
            s = dot(v0[j] - XR[q], nn[j]) / dot(dr, nn[j])
            ok = ok & ((s > prev) & (s < 1))[:, 0]
            X.append(XR[q] + s * dr)
            prev = s
        T = V[ids[:, j]]
        for a in range(3):
            side = dot(torch.linalg.cross(T[:, (a + 1) % 3] - T[:, a], X[-1] - T[:, a]), nn[j])[:, 0]
            ok = ok & ~(side < 0)
    X.append(rx)
    return torch.stack(X, 1), ok


def _unit(a):
    return a / a.norm(dim=-1, keepdim=True)


def _pol(u, d):
    p = u - (d * u).sum(-1, keepdim=True) * d
    return p / p.norm(dim=-1, keepdim=True)


def _amplitude(X, nrm, er, sg, pec, db, refl, u, freq):
    """Complex amplitudes of paths through X (Fresnel TE/TM with vector
    polarisation, free-space spreading, phase k L)."""
    leg = X[:, 1:] - X[:, :-1]
    L = leg.norm(dim=-1).sum(-1)
    d = _unit(leg)
    E = _pol(u, d[:, 0]).to(torch.complex128)
    for j in range(len(refl)):
        if not refl[j]:
            E = E * (10.0 ** (-db[:, j] / 20.0))[:, None]
            continue
        # the direction in, and the next one out, along the real path
        di, do, nh = d[:, j], d[:, j + 1], _unit(nrm[:, j])
        ct = (di * nh).sum(-1).abs()
        s = _unit(torch.linalg.cross(di, nh))
        pi, po = torch.linalg.cross(s, di), torch.linalg.cross(s, do)
        ec = torch.complex(er[:, j], -sg[:, j] / (2 * math.pi * freq * EPS0))
        rt = torch.sqrt(ec - (1 - ct * ct))
        te, tm = (ct - rt) / (ct + rt), (ec * ct - rt) / (ec * ct + rt)
        one = torch.ones_like(te)
        te, tm = torch.where(pec[:, j], -one, te), torch.where(pec[:, j], one, tm)
        E = (te * (E * s).sum(-1))[:, None] * s + (tm * (E * pi).sum(-1))[:, None] * po
    proj = (E * _pol(u, -d[:, -1])).sum(-1)
    ph = 2 * math.pi * freq / C0 * L
    return proj * torch.complex(torch.cos(ph), -torch.sin(ph)) * (C0 / freq / (4 * math.pi) / L)


def _powers(E, inc, pt):
    return 10 * torch.log10(pt * (E.real ** 2 + E.imag ** 2)) + 30, 10 * torch.log10(pt * inc) + 30


def _exact_frame(sc, prm, f, dirs, n_trans):
    V = _world(sc, sc.xf[f] if sc.nobj else None)
    tri = _Tris(V)
    tx = torch.tensor(sc.tx, dtype=torch.float64, device="cuda")
    rx = torch.tensor(sc.rx[f], dtype=torch.float64, device="cuda")
    mat = torch.tensor(sc.materials, dtype=torch.float64, device="cuda")[torch.tensor(sc.tri_mat, device="cuda").long()]
    db = torch.tensor(sc.meta.get("trans_db", [-1.0] * len(sc.materials)), dtype=torch.float64, device="cuda")
    loss = db[torch.tensor(sc.tri_mat, device="cuda").long()]
    keys = _captures(sc, tri, loss, dirs, tx, rx, prm, n_trans)
    u = torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device="cuda")
    nrx = rx.shape[0]
    E = torch.zeros(nrx, dtype=torch.complex128, device="cuda")
    inc = torch.zeros(nrx, dtype=torch.float64, device="cuda")
    for k in range(prm.max_refl + n_trans + 1):
        at = keys[keys[:, 1] == k]
        pattern = (((at[:, 2:2 + k] & TBIT) != 0).long() * (2 ** torch.arange(k, device="cuda"))).sum(-1)
        for pat in torch.unique(pattern).tolist():
            sel = at[pattern == pat]
            refl = [not (pat >> j) & 1 for j in range(k)]
            ids = sel[:, 2:2 + k] & ~TBIT
            X, ok = _images(V, tri.n, tx, rx[sel[:, 0]], ids, refl)
            sel, ids, X = sel[ok], ids[ok], X[ok]
            free = torch.ones(len(sel), dtype=torch.bool, device="cuda")
            step = max(64, int(3e7) // V.shape[0])
            for j in range(k + 1):
                for i in range(0, len(sel), step):
                    t = tri.hits(X[i:i + step, j], X[i:i + step, j + 1] - X[i:i + step, j])
                    for e in ([j - 1] if j else []) + ([j] if j < k else []):
                        t.scatter_(1, ids[i:i + step, e:e + 1], math.inf)
                    free[i:i + step] &= ~((t > prm.eps_occ) & (t < 1 - prm.eps_occ)).any(1)
            sel, ids, X = sel[free], ids[free], X[free]
            m = mat[ids]
            a = _amplitude(X, tri.n[ids], m[..., 0], m[..., 1], m[..., 2] != 0, loss[ids], refl, u, prm.freq_hz)
            E.index_add_(0, sel[:, 0], a)
            inc.index_add_(0, sel[:, 0], a.abs() ** 2)
    pc, pi = _powers(E, inc, prm.tx_power_w)
    return {"field": torch.view_as_real(E).reshape(-1), "p_coh": pc, "p_inc": pi, "paths": [[None] * 4]}


def _exact_gradient(case, seed):
    """Powers and derivatives over the given records by automatic differentiation."""
    st = prepare(case, seed)
    sc, prm, rec = st["sc"], st["prm"], st["paths"]
    V0 = _world(sc, sc.xf[1])
    dev = V0.device
    theta = st["theta"].clone().requires_grad_(True)
    nm, nrx = len(sc.materials), case["rx"]
    move = theta[2 * nm:].reshape(-1, 2) - st["theta"][2 * nm:].reshape(-1, 2)
    obj = torch.tensor(sc.tri_obj, device=dev).long()
    shift = torch.zeros(V0.shape[0], 3, dtype=torch.float64, device=dev)
    m = torch.nonzero(obj >= 0)[:, 0]
    shift = shift.index_put((m,), torch.cat([move[obj[m]], torch.zeros(len(m), 1, dtype=torch.float64, device=dev)], 1))
    V = V0 + shift[:, None]
    n = torch.linalg.cross(V[:, 1] - V[:, 0], V[:, 2] - V[:, 0])
    tm = torch.tensor(sc.tri_mat, device=dev).long()
    pec = torch.tensor(sc.materials[:, 2] != 0, device=dev)
    tx = torch.tensor(sc.tx, dtype=torch.float64, device=dev)
    rx = torch.tensor(st["rx"], dtype=torch.float64, device=dev)
    u = torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device=dev)
    E = torch.zeros(nrx, dtype=torch.complex128, device=dev)
    for k in np.unique(rec["depth"]).tolist():
        p = rec[rec["depth"] == k]
        r = torch.tensor(p["rx"], device=dev).long()
        ids = torch.tensor(p["tri"][:, :k].astype(np.int64), device=dev)
        X, _ = _images(V, n, tx, rx[r], ids, [True] * k)
        a = _amplitude(X, n[ids], theta[0:2 * nm:2][tm[ids]], theta[1:2 * nm:2][tm[ids]], pec[tm[ids]],
                       torch.zeros(ids.shape, dtype=torch.float64, device=dev), [True] * k, u, prm.freq_hz)
        E = E.index_add(0, r, a)
    have = torch.tensor(np.unique(rec["rx"]), device=dev).long()
    if case["way"] == "power":
        pc = 10 * torch.log10(prm.tx_power_w * (E.real ** 2 + E.imag ** 2)) + 30
        g, = torch.autograd.grad(pc[have].sum(), theta)
        return {"p_coh": pc.detach(), "grad": g}
    dE = torch.zeros(nrx, theta.numel(), dtype=torch.complex128, device=dev)
    for r in have.tolist():
        re, = torch.autograd.grad(E[r].real, theta, retain_graph=True)
        im, = torch.autograd.grad(E[r].imag, theta, retain_graph=True)
        dE[r] = torch.complex(re, im)
    E = E.detach()
    dp = torch.zeros(nrx, theta.numel(), dtype=torch.float64, device=dev)
    dp[have] = (20 / math.log(10)) * (E[have].conj()[:, None] * dE[have]).real / (E[have].abs() ** 2)[:, None]
    return {"field": E, "dfield": dE, "dp": dp}


def exact(case, seed):
    """Field and powers in 64 bits; the path records (their order is by an
    internal key) have none. None for the larger searches, which brute force
    does not finish in time: the urban kinds and diffraction."""
    kind = case["kind"]
    if kind == "reduce":
        rec = prepare(case, seed)["records"]
        E = np.zeros(case["rx"], np.complex128)
        inc = np.zeros(case["rx"])
        a = rec["amp_re"] + 1j * rec["amp_im"]
        np.add.at(E, rec["rx"], a)
        np.add.at(inc, rec["rx"], np.abs(a) ** 2)
        with np.errstate(divide="ignore"):
            return {"field": np.stack([E.real, E.imag], 1), "p_coh": 10 * np.log10(5.0 * np.abs(E) ** 2) + 30,
                    "p_inc": 10 * np.log10(5.0 * inc) + 30}
    if kind == "gradient":
        return _exact_gradient(case, seed)
    if kind in ("street", "highway", "office") and not case.get("order", 0) and case["mode"] != "sticky":
        sc = _scene(case, seed)
        dirs = torch.tensor(_rays(sc.n_rays), dtype=torch.float64, device="cuda")
        return [_exact_frame(sc, _params(case, sc), f, dirs, case.get("trans", 0))
                for f in range(1, 1 + case["frames"])]
    return None
