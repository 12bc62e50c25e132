"""Performance cases: the calls that a program built on this library makes,
over the sizes of the repository's own workloads (scenegen.py, bench.py and
the tests).

Every case goes through the public binding (paper_2301_05125_gb300.adgi).
Scene geometry comes from the seeded generators and is kept per process; a
case's seed sets the frame it starts at (lights and occluders move with the
frame), the random numbers of the update, the query points, the rays and the
mesh order.
"""
import functools
import math

import numpy as np
import torch

from paper_2301_05125_gb300 import adgi
from paper_2301_05125_gb300 import scenegen as S

RING = 16  # frames of lights and occluder positions a state holds


def _update(name, **kw):
    """an update case: the generator's defaults, then the given values"""
    c = dict(kind="update", scene="city", n_boxes=15000, dx=32, dy=16, dz=32, spacing=4.0, avg=64, lo=8, hi=256,
             fp16=0, sampler=0, dyn_ratio=0, blend=0, camera=False, graph=True, move=True)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest volume: one room, one light, static geometry, plain calls; launches and latency count
        _update("room", scene="room", n_boxes=0, dx=4, dy=4, dz=4, spacing=2.0, graph=False, move=False),
        # one client of a serving mix: an odd-sized grid, half atlases, moving occluders, graph replays
        _update("client_fp16", n_boxes=5000, dx=19, dy=9, dz=19, spacing=5.0, fp16=1),
        # the tunnel + city workload: few probes, many rays each
        _update("tunnel", avg=256, hi=1024),
        # the largest volume: 131,072 probes, about 2 million triangles, plain calls
        _update("scaled", scene="scaled", n_boxes=165000, dx=64, dy=32, dz=64, lo=4, hi=512, graph=False),
        # the packed 32-bit atlases under a moving camera with clip volumes
        _update("packed_camera", n_boxes=15000, dx=33, dy=15, dz=31, fp16=3, camera=True),
        # the Metropolis sampler with dynamic chains on the tunnel + city workload
        _update("metropolis", avg=256, hi=1024, sampler=1, dyn_ratio=4),
        # the cosine-gather blend on the tunnel + city workload
        _update("cosine", avg=256, hi=1024, blend=1),
        # several volumes of uneven size updated by one call per frame (half atlases)
        dict(name="batch", kind="batch", volumes=6, scenes=2, tri_lo=20000, tri_hi=120000, dmax=40, fp16=1, tick=False),
        # the shading query of a frame: 960 x 540 surface points in screen order
        dict(name="query", kind="query", n=518400, dx=32, dy=16, dz=32, fp16=0, tile=32),
        # a program's own rays (visibility, picking, audio): unordered, an odd count
        dict(name="rays", kind="rays", n_boxes=15000, n=1000003, coherent=False, move=False),
        # the linear BVH of a mesh that deforms every frame
        dict(name="rebuild", kind="rebuild", n_boxes=8000),
        # a level is loaded and first used: host arrays in, one batch of rays out
        dict(name="load", kind="load", n_boxes=15000, n=65536, coherent=True, move=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["update"] * 6 + ["batch", "query", "query", "rays", "rebuild", "load"])
    if kind == "update":
        form = rng.choice(["plain", "plain", "plain", "packed", "metropolis", "cosine"])
        a = _log(rng, 4, 40)
        dims = [max(4, int(a * rng.uniform(0.7, 1.3))), max(4, a // 2 + rng.randrange(0, 3)),
                max(4, int(a * rng.uniform(0.7, 1.3)))]
        avg = _log(rng, 16, 128)
        while dims[0] * dims[1] * dims[2] * avg > 4000000:
            avg = max(12, avg // 2)
            dims[0] = max(4, dims[0] * 3 // 4)
        c = _update(None, n_boxes=_log(rng, 300, 40000), dx=dims[0], dy=dims[1], dz=dims[2],
                    spacing=rng.choice([2.0, 3.0, 4.0, 5.0, 8.0]), avg=avg, hi=rng.choice([160, 256, 512]),
                    lo=rng.choice([4, 8]), graph=rng.random() < 0.7, move=rng.random() < 0.7)
        if form == "plain":
            c["fp16"] = rng.choice([0, 0, 1, 2])
            c["camera"] = rng.random() < 0.3
        elif form == "packed":
            c["fp16"] = 3
            c["camera"] = rng.random() < 0.5
        elif form == "metropolis":
            c["sampler"] = 1
            c["dyn_ratio"] = rng.choice([0, 2, 4])
        else:
            c["blend"] = 1
            c["fp16"] = rng.choice([0, 1])
        return c
    if kind == "batch":
        return dict(kind="batch", volumes=rng.randrange(2, 7), scenes=rng.randrange(1, 3), tri_lo=12000 + rng.randrange(9000),
                    tri_hi=40000 + rng.randrange(60000), dmax=rng.randrange(10, 34), fp16=rng.choice([0, 1]),
                    tick=rng.random() < 0.5)
    if kind == "query":
        return dict(kind="query", n=_log(rng, 64, 1000000), dx=rng.randrange(4, 40), dy=rng.randrange(4, 20),
                    dz=rng.randrange(4, 40), fp16=rng.choice([0, 0, 1]), tile=rng.choice([1, 8, 32]))
    if kind == "rays":
        return dict(kind="rays", n_boxes=_log(rng, 300, 40000), n=_log(rng, 500, 2000000),
                    coherent=rng.random() < 0.5, move=rng.random() < 0.5)
    if kind == "rebuild":
        return dict(kind="rebuild", n_boxes=_log(rng, 20, 40000))
    return dict(kind="load", n_boxes=_log(rng, 300, 30000), n=_log(rng, 5000, 200000), coherent=True,
                move=rng.random() < 0.5)


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=3)
def _scene(kind, n_boxes):
    if kind == "room":
        return S.box_room(1)
    return S.scaled(1, n_boxes) if kind == "scaled" else S.tunnel_city(1, n_boxes)


@functools.lru_cache(maxsize=2)
def _batch_scenes(volumes, scenes, tri_lo, tri_hi, dmax, fp16):
    return S.batched(1, volumes, scenes, float(tri_lo), float(tri_hi), (8, 6, 8), (dmax, max(8, dmax // 2), dmax),
                     fp16=fp16)


def _n_tris(c):
    if c["kind"] == "batch":
        return int(0.5 * (c["tri_lo"] + c["tri_hi"]))
    if c.get("scene") == "room":
        return 144
    return int(11.6 * c["n_boxes"]) + (43248 if c.get("scene") == "scaled" else 22768)


def _view_proj(eye, target, fov_deg=60.0, near=0.5, far=500.0):
    eye, target = np.asarray(eye, np.float64), np.asarray(target, np.float64)
    f = target - eye
    f /= np.linalg.norm(f)
    r = np.cross(f, [0.0, 1.0, 0.0])
    r /= np.linalg.norm(r)
    u = np.cross(r, f)
    view = np.eye(4)
    view[0, :3], view[1, :3], view[2, :3] = r, u, -f
    view[:3, 3] = -view[:3, :3] @ eye
    t = 1.0 / np.tan(np.radians(fov_deg) / 2)
    proj = np.zeros((4, 4))
    proj[0, 0], proj[1, 1] = t, t
    proj[2, 2], proj[2, 3] = -(far + near) / (far - near), -2 * far * near / (far - near)
    proj[3, 2] = -1.0
    return (proj @ view).astype(np.float32)


def _ring(w, f0, move):
    """the lights (and occluder positions) of RING frames from f0 on"""
    lights = [w.lights_at(f0 + k) for k in range(RING)]
    verts = None
    if move:
        verts = [torch.from_numpy(np.ascontiguousarray(w.dyn_at(f0 + k), np.float32)).cuda() for k in range(RING)]
    return lights, verts


def _tiles(vol):
    """device buffers for the volume's whole state: weights and both atlases"""
    return {which: torch.empty(adgi.adgi_slab_bytes(vol.h, which, 0, vol.P) // size, dtype=dt, device="cuda")
            for which, dt, size in (
                ("W", torch.int32, 4),
                ("IRR", torch.int32 if vol.packed else torch.float16 if vol.fp16 else torch.float32,
                 2 if vol.fp16 and not vol.packed else 4),
                ("DEP", torch.int32 if vol.packed else torch.float16 if vol.fp16 else torch.float32,
                 2 if vol.fp16 and not vol.packed else 4),
                ("DEP_N", torch.uint8, 1))
            if not (vol.packed and which == "DEP_N")}


def _copy_tiles(vol, out):
    for which, buf in out.items():
        adgi.adgi_slab_copy(vol.h, which, 0, vol.P, buf, 0)
    return out


def _prepare_update(c, seed):
    w = _scene(c["scene"], c["n_boxes"])
    d = (c["dx"], c["dy"], c["dz"])
    sp = c["spacing"]
    origin = (1.0, 1.0, 1.0) if c["scene"] == "room" else (-0.5 * sp * (d[0] - 1), 1.0, -0.5 * sp * (d[2] - 1))
    vol = adgi.Volume(origin=origin, spacing=(sp, sp, sp), dims=d, rays_avg=c["avg"], rays_min=c["lo"],
                      rays_max=c["hi"], atlas_fp16=c["fp16"], sampler=c["sampler"], dyn_ratio=c["dyn_ratio"],
                      blend_mode=c["blend"])
    vol.set_scene(w.verts, w.idx, w.albedo)
    f0 = 2 * (seed % 499)
    lights, verts = _ring(w, f0, c["move"])
    cameras = [None] * RING
    if c["camera"]:
        for k in range(RING):  # a camera sweeping past the grid
            a = 0.13 * k + 0.01 * (seed % 600)
            eye = (-0.45 * sp * max(d) * math.cos(a), 14.0, -0.45 * sp * max(d) * math.sin(a))
            cameras[k] = (eye, 0.5 * sp * max(d) + 10.0, _view_proj(eye, (0.0, 6.0, 5.0 * math.sin(3.0 * a))))
    st = dict(kind="update", vol=vol, f=f0, f0=f0, seed=seed, lights=lights, verts=verts, cameras=cameras, sky=w.sky,
              first=w.dyn_first, step=vol.update_graph if c["graph"] else vol.update, out=_tiles(vol))
    for _ in range(2):  # a program in its run: both BVH parts built, the first frames blended
        _run_update(st)
    return st


def _run_update(st):
    f = st["f"]
    k = (f - st["f0"]) % RING
    if st["verts"] is not None:
        st["vol"].move_vertices(st["first"], st["verts"][k])
    st["step"](f, st["seed"], st["lights"][k], st["sky"], st["cameras"][k])
    st["f"] = f + 1
    return _copy_tiles(st["vol"], st["out"])


def _prepare_batch(c, seed):
    ws = _batch_scenes(c["volumes"], c["scenes"], c["tri_lo"], c["tri_hi"], c["dmax"], c["fp16"])
    stream = torch.cuda.Stream()
    vols, rings = [], []
    f0 = 2 * (seed % 499)
    for w in ws:
        v = adgi.Volume(stream=stream.cuda_stream, **w.volume)
        v.set_scene(w.verts, w.idx, w.albedo)
        vols.append(v)
        rings.append(_ring(w, f0, True))
    torch.cuda.synchronize()
    st = dict(kind="batch", stream=stream, ws=ws, vols=vols, rings=rings, f=f0, f0=f0, seed=seed,
              batch=(adgi.Tick if c["tick"] else adgi.Batch)(vols, stream.cuda_stream), out=[_tiles(v) for v in vols])
    for _ in range(2):
        _run_batch(st)
    return st


def _run_batch(st):
    f = st["f"]
    k = (f - st["f0"]) % RING
    frames = []
    for w, v, (lights, verts) in zip(st["ws"], st["vols"], st["rings"]):
        v.move_vertices(w.dyn_first, verts[k])
        frames.append(adgi.make_frame(f, st["seed"], lights[k], w.sky))
    st["batch"].update(frames)
    st["f"] = f + 1
    return [_copy_tiles(v, out) for v, out in zip(st["vols"], st["out"])]


def _fold(t, n):
    """fill the border of octahedral tiles [P, n + 2, n + 2, C] from their interior"""
    t[:, 0, 1:n + 1] = t[:, 1, 1:n + 1].flip(1)
    t[:, n + 1, 1:n + 1] = t[:, n, 1:n + 1].flip(1)
    t[:, 1:n + 1, 0] = t[:, 1:n + 1, 1].flip(1)
    t[:, 1:n + 1, n + 1] = t[:, 1:n + 1, n].flip(1)
    t[:, 0, 0], t[:, 0, n + 1] = t[:, n, n].clone(), t[:, n, 1].clone()
    t[:, n + 1, 0], t[:, n + 1, n + 1] = t[:, 1, n].clone(), t[:, 1, 1].clone()
    return t


def _query_inputs(c, seed):
    """atlases as a frame leaves them, and surface points in screen order
    (tiles of tile x tile pixels on one plane each) with their normals"""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    d = (c["dx"], c["dy"], c["dz"])
    P, sp = d[0] * d[1] * d[2], 4.0
    origin = (-2.0 * (d[0] - 1), 1.0, -2.0 * (d[2] - 1))
    dt = torch.float16 if c["fp16"] else torch.float32
    irr = torch.empty(P, 8, 8, 4, device="cuda").exponential_(1.0, generator=g) * 0.8
    irr[..., 3] = 255.0
    base = 0.3 + 2.5 * torch.rand(P, 1, 1, device="cuda", generator=g)
    mean = sp * base * (0.6 + 0.8 * torch.rand(P, 16, 16, device="cuda", generator=g))
    var = (mean * (0.02 + 0.3 * torch.rand(P, 16, 16, device="cuda", generator=g))) ** 2
    irr, dep = _fold(irr, 6).to(dt), _fold(torch.stack([mean, var], -1), 14).to(dt)
    n, tile = c["n"], c["tile"]
    nt = -(-n // (tile * tile))
    lo = torch.tensor(origin, device="cuda")
    ext = torch.tensor([sp * (k - 1) for k in d], device="cuda")
    anchor = lo + ext * torch.rand(nt, 3, device="cuda", generator=g)
    nrm = torch.nn.functional.normalize(torch.randn(nt, 3, device="cuda", generator=g), dim=1)
    t0 = torch.nn.functional.normalize(torch.linalg.cross(nrm, nrm.roll(1, 1) + 0.1), dim=1)
    t1 = torch.linalg.cross(nrm, t0)
    uv = (torch.arange(tile, device="cuda") - 0.5 * tile + 0.37) * 0.05
    pos = anchor[:, None, None] + t0[:, None, None] * uv[None, :, None, None] + t1[:, None, None] * uv[None, None, :, None]
    nrm = nrm[:, None, None].expand(nt, tile, tile, 3)
    return (d, origin, sp, irr, dep, pos.reshape(-1, 3)[:n].contiguous(), nrm.reshape(-1, 3)[:n].contiguous())


def _prepare_query(c, seed):
    d, origin, sp, irr, dep, pos, nrm = _query_inputs(c, seed)
    vol = adgi.Volume(origin=origin, spacing=(sp, sp, sp), dims=d, rays_avg=16, rays_min=8, rays_max=32,
                      atlas_fp16=c["fp16"])
    vol.write_atlas(irr.cpu().numpy(), dep.cpu().numpy())
    return dict(kind="query", vol=vol, pos=pos, nrm=nrm, out=torch.empty_like(pos))


def _rays(n, coherent, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
    if coherent:  # one camera's pixels, row by row
        a = 0.01 * (seed % 600)
        eye = torch.tensor([60.0 * math.cos(a), 18.0, 60.0 * math.sin(a)], device="cuda")
        wid = max(1, int(math.sqrt(1.78 * n)))
        i = torch.arange(n, device="cuda")
        u, v = (i % wid) / wid - 0.5, 0.35 - (i // wid) / max(1.0, n / wid) * 0.9
        f = torch.nn.functional.normalize(-eye, dim=0)
        r = torch.nn.functional.normalize(torch.linalg.cross(f, torch.tensor([0.0, 1.0, 0.0], device="cuda")), dim=0)
        up = torch.linalg.cross(r, f)
        dirs = f + 1.2 * u[:, None] * r + 0.9 * v[:, None] * up
        return eye.expand(n, 3).contiguous(), torch.nn.functional.normalize(dirs, dim=1).contiguous()
    o = torch.rand(n, 3, device="cuda", generator=g) * torch.tensor([160.0, 24.0, 160.0], device="cuda")
    o -= torch.tensor([80.0, -1.0, 80.0], device="cuda")
    dirs = torch.nn.functional.normalize(torch.randn(n, 3, device="cuda", generator=g), dim=1)
    return o.contiguous(), dirs.contiguous()


def _prepare_rays(c, seed):
    w = _scene("city", c["n_boxes"])
    vol = adgi.Volume(origin=(-8.0, 1.0, -8.0), spacing=(4.0, 4.0, 4.0), dims=(4, 4, 4))
    o, d = _rays(c["n"], c["coherent"], seed)
    n = c["n"]
    st = dict(kind=c["kind"], vol=vol, o=o, d=d, t=torch.empty(n, device="cuda"),
              tri=torch.empty(n, dtype=torch.int32, device="cuda"), moves=None)
    if c["move"]:
        st["moves"] = (w.dyn_first, torch.from_numpy(np.ascontiguousarray(w.dyn_at(seed % 499), np.float32)).cuda())
    if c["kind"] == "load":
        st["scene"] = (np.ascontiguousarray(w.verts, np.float32), np.ascontiguousarray(w.idx, np.int32),
                       np.ascontiguousarray(w.albedo, np.float32))
    else:
        vol.set_scene(w.verts, w.idx, w.albedo)
        if st["moves"]:
            vol.move_vertices(*st["moves"])
        _trace(st)
    return st


def _trace(st):
    adgi.adgi_trace_closest(st["vol"].h, st["o"], st["d"], 1e-3, 1e30, st["t"], st["tri"])
    return {"t": st["t"], "tri": st["tri"]}


def _run_load(st):
    st["vol"].set_scene(*st["scene"])
    if st["moves"]:
        st["vol"].move_vertices(*st["moves"])
    return _trace(st)


def _prepare_rebuild(c, seed):
    w = _scene("city", c["n_boxes"])
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    v = torch.from_numpy(w.verts).cuda()
    v = v + 0.05 * torch.randn(v.shape, device="cuda", generator=g)
    idx = torch.from_numpy(w.idx).cuda()
    nt = idx.shape[0]
    return dict(kind="rebuild", v=v.contiguous(), idx=idx.contiguous(), eps=adgi.scene_eps(w.verts),
                nodes=torch.zeros(nt - 1, 16, dtype=torch.int32, device="cuda"),
                tris=torch.zeros(nt, 12, dtype=torch.int32, device="cuda"))


def _run_rebuild(st):
    adgi.adgi_build_bvh(st["v"], st["idx"], st["eps"], st["nodes"], st["tris"],
                        torch.cuda.current_stream().cuda_stream)
    return {"nodes": st["nodes"], "tris": st["tris"]}


def prepare(case, seed):
    return {"update": _prepare_update, "batch": _prepare_batch, "query": _prepare_query, "rays": _prepare_rays,
            "load": _prepare_rays, "rebuild": _prepare_rebuild}[case["kind"]](case, int(seed))


def run(state):
    kind = state["kind"]
    if kind == "update":
        return _run_update(state)
    if kind == "batch":
        return _run_batch(state)
    if kind == "query":
        state["vol"].query(state["pos"], state["nrm"], state["out"])
        return state["out"]
    if kind == "rays":
        return _trace(state)
    if kind == "load":
        return _run_load(state)
    return _run_rebuild(state)


# ------------------------------------------------------------------ work
def _trace_flops(rays, tris):
    # one path of four-box visits (13 operations a box) to the depth of a 4-ary tree, and one triangle test
    return rays * (52.0 * math.log(max(tris, 4), 4) + 55.0)


def work(case):
    c = case
    k = c["kind"]
    if k == "query":
        per = 8 * 64 * 4 + 256 * (2 if c["fp16"] else 4) * 2 if c["fp16"] else 64 * 16 + 256 * 8
        tiles = c["dx"] * c["dy"] * c["dz"] * per
        return {"bytes": 36.0 * c["n"] + min(tiles, c["n"] * 8 * 128), "flops": c["n"] * 8 * 90.0}
    if k in ("rays", "load"):
        T = _n_tris(c)
        scene = 60.0 * T if k == "load" else 48.0 * T
        return {"bytes": 32.0 * c["n"] + scene, "flops": _trace_flops(c["n"], T)}
    if k == "rebuild":
        T = _n_tris(c)
        return {"bytes": T * (36.0 + 12.0 + 48.0 + 64.0), "flops": 60.0 * T}
    if k == "batch":
        P = c["volumes"] * (0.35 * c["dmax"]) ** 3
        avg, fp16, lights, cos = 64, c["fp16"], 4, False
    else:
        P, avg, fp16 = c["dx"] * c["dy"] * c["dz"], c["avg"], c["fp16"]
        lights, cos = (1 if c["scene"] == "room" else 4), c["blend"] == 1
    T = _n_tris(c)
    per = {0: 64 * 16 + 256 * 9, 1: 64 * 8 + 256 * 5, 2: 64 * 8 + 256 * 5, 3: 320 * 4}[fp16]
    R = P * avg * (2.0 if c.get("sampler") else 1.0)
    flops = _trace_flops(R, T) + _trace_flops(0.4 * R * lights, T) + R * 8 * 90.0
    if cos:
        flops += 0.5 * P * avg * (36 + 196) * 16.0
    return {"bytes": 2.0 * P * per + 48.0 * T, "flops": flops}


# ------------------------------------------------------------------ 64-bit values
def _oct(v):
    l1 = v.abs().sum(-1)
    x, y = v[..., 0] / l1, v[..., 1] / l1
    sx = torch.where(x >= 0, 1.0, -1.0).double()
    sy = torch.where(y >= 0, 1.0, -1.0).double()
    neg = v[..., 2] < 0
    return torch.where(neg, (1 - y.abs()) * sx, x), torch.where(neg, (1 - x.abs()) * sy, y)


def _corners(px, py, n):
    fx, fy = 0.5 + (px + 1) * 0.5 * n, 0.5 + (py + 1) * 0.5 * n
    x0, y0 = fx.floor().clamp(0, n), fy.floor().clamp(0, n)
    ax, ay = (fx - x0).clamp(0, 1), (fy - y0).clamp(0, 1)
    i = (y0 * (n + 2) + x0).long()
    return [(i, (1 - ax) * (1 - ay)), (i + 1, ax * (1 - ay)), (i + n + 2, (1 - ax) * ay), (i + n + 3, ax * ay)]


def exact(case, seed):
    """The shading query in 64 bits: eight probes, trilinear weights times the
    one-sided Chebyshev bound.  The other calls' outputs have no closed form
    that plain torch gives in seconds (whole scenes are traced)."""
    if case["kind"] != "query":
        return None
    d, origin, sp, irr, dep, pos, nrm = _query_inputs(case, int(seed))
    irr = irr.double().reshape(-1, 64, 4)
    dep = dep.double().reshape(-1, 256, 2)
    x, nrm = pos.double(), nrm.double()
    lo = torch.tensor(origin, dtype=torch.float64, device="cuda")
    dims = torch.tensor(d, device="cuda")
    b = torch.minimum(((x - lo) / sp).floor().clamp(min=0).long(), dims - 2)
    al = ((x - (lo + b * sp)) / sp).clamp(0, 1)
    var_min = 1e-6 * 3.0 * sp * sp
    px, py = _oct(nrm)
    ic = _corners(px, py, 6)
    sums = torch.zeros_like(x)
    plain = torch.zeros_like(x)
    sw = torch.zeros(x.shape[0], dtype=torch.float64, device="cuda")
    for c in range(8):
        o = torch.tensor([c & 1, (c >> 1) & 1, (c >> 2) & 1], device="cuda")
        wt = torch.where(o.bool(), al, 1 - al).prod(1)
        cell = b + o
        p = cell[:, 0] + d[0] * (cell[:, 1] + d[1] * cell[:, 2])
        v = x - (lo + cell * sp)
        dist = v.norm(dim=1)
        qx, qy = _oct(torch.where(dist[:, None] > 0, v, torch.ones_like(v)))
        dc = [(dep[p, i], w) for i, w in _corners(qx, qy, 14)]
        mu = sum(w * t[:, 0] for t, w in dc)
        var = sum(w * (t[:, 1] + (t[:, 0] - mu) ** 2) for t, w in dc)
        mu, var = torch.where(dist > 0, mu, 0.0), torch.where(dist > 0, var, 0.0).clamp(min=var_min)
        wc = torch.where(dist > mu, var / (var + (dist - mu) ** 2), 1.0)
        E = sum(w[:, None] * irr[p, i, :3] for i, w in ic)
        sums += (wt * wc)[:, None] * E
        plain += wt[:, None] * E
        sw += wt * wc
    return torch.where(sw[:, None] >= 1e-12, sums / sw[:, None].clamp(min=1e-12), plain)
