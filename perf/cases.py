"""Workloads of the radar scan library, each one pass through its public entry points.

The scenes and sensors are the repository's own configurations (tiny room, ~200k-triangle campus,
~1M-triangle campus of the batched scans, ~5M-triangle city, the 50k campus of the served scans)
with seeded poses, sensor settings and vertex corrections.  A case is a dict of plain values:

  path     which call is made: scan, static, step (vertex update and scan), batch, serve, returns, db
  scene    room, campus or city; tris is the triangle target of a campus
  az, rays, bounces, bins   the sensor (batch and serve draw rays, bounces and bins per scan)
  post     0: plain image; 1: speckle, noise, range blur; 2: the same with Perlin noise, the beam
           pattern across azimuths, an elliptic beam and a minimum ray energy
"""
import functools
import math
import random

import numpy as np
import torch

from paper_2310_03505_gb300 import rr, scenes

BIN = 0.0438


def listed():
    return [
        # the smallest scan a robot simulation asks for, at its sensor rate: latency and launches
        dict(name="tiny_scan", path="scan", scene="room", tris=0, az=400, rays=8, bounces=3, bins=1142, post=0),
        # the same room through the call that never allocates (real-time loops), odd sizes, full post pass
        dict(name="tiny_static_post", path="static", scene="room", tris=0, az=397, rays=11, bounces=3, bins=1013, post=2),
        # the medium scan on a resident scene
        dict(name="campus_scan", path="scan", scene="campus", tris=200_000, az=400, rays=200, bounces=5, bins=2000, post=0),
        # a map correction arrives (pinned host vertices), the hierarchy is rebuilt, one scan, image back on the host
        dict(name="campus_step_host", path="step", scene="campus", tris=200_000, az=400, rays=200, bounces=5, bins=2000,
             post=0, host=True),
        # ragged sensor with every option of the model on: the minimum energy makes visibility run before shading
        dict(name="campus_post", path="scan", scene="campus", tris=200_000, az=333, rays=97, bounces=7, bins=3001, post=2),
        # the medium scan over the 8-wide quantised nodes (the autotuner's other node format)
        dict(name="campus_wide8", path="scan", scene="campus", tris=200_000, az=400, rays=200, bounces=5, bins=2000,
             post=0, wide=True),
        # a trajectory's scans of uneven ray counts in shared launch sequences (dataset generation)
        dict(name="batch_1m", path="batch", scene="campus", tris=1_000_000, az=400, rays=512, bounces=5, bins=2000,
             post=0, scans=24),
        # the large scene: rebuild and scan, and the scan alone on the resident scene
        dict(name="city_step", path="step", scene="city", tris=0, az=400, rays=1000, bounces=8, bins=4000, post=0,
             host=False),
        dict(name="city_scan", path="scan", scene="city", tris=0, az=400, rays=1000, bounces=8, bins=4000, post=0),
        # a burst of requests from several robots over two resident scenes
        dict(name="serve_burst", path="serve", scene="campus", tris=50_000, az=400, rays=256, bounces=6, bins=4000,
             post=1, scans=24),
        # binning of returns that a user's own tracer made
        dict(name="returns", path="returns", az=400, bins=2000, n=1_500_000),
        # display images of a recorded drive
        dict(name="display_db", path="db", n=256 * 400 * 2000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    path = rng.choice(["scan", "scan", "scan", "static", "step", "step", "batch", "serve", "returns", "db"])
    if path == "returns":
        return dict(path=path, az=_log(rng, 16, 1600), bins=_log(rng, 200, 8000), n=_log(rng, 20_000, 1_500_000))
    if path == "db":
        return dict(path=path, n=_log(rng, 100_000, 200_000_000))
    c = dict(path=path, scene=rng.choice(["room", "campus", "campus", "city"]), tris=0, az=_log(rng, 90, 800),
             rays=_log(rng, 4, 500), bounces=rng.randint(2, 8), bins=_log(rng, 300, 4000), post=rng.choice([0, 0, 1, 2]))
    if path == "static":
        c.update(scene="room", az=_log(rng, 90, 500), rays=_log(rng, 4, 40), bounces=rng.randint(2, 5))
    if path in ("batch", "serve"):
        c.update(scene="campus", az=rng.choice([200, 360, 400]), rays=_log(rng, 24, 256), bounces=rng.randint(3, 6),
                 scans=rng.randint(3, 24), post=rng.choice([0, 1]))
    if path == "scan":
        c["wide"] = rng.random() < 0.2
    if path == "step":
        c["host"] = rng.random() < 0.5
    if c["scene"] == "campus":
        c["tris"] = _log(rng, 50_000, 1_000_000)
    return c


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=None)
def _mesh(kind, tris):
    """A scene of the repository's generators (fixed geometry) and its arrays on the GPU."""
    if kind == "room":
        sc = scenes.tiny_room()
    elif kind == "city":
        sc = scenes.city()
    elif tris <= 100_000:   # the small served campus
        sc = scenes.campus(target_tris=tris, seed=0x5EED0004, n_buildings=60, n_cylinders=150, extent=80.0)
    else:
        sc = scenes.campus(target_tris=tris)
    return sc, [torch.from_numpy(np.ascontiguousarray(a)).cuda()
                for a in (sc.vertices, sc.triangles.view(np.int32), sc.material_ids.view(np.int16))]


class _Scene:
    """A resident scene, freed with its owner."""

    def __init__(self, kind, tris):
        self.mesh, arrays = _mesh(kind, tris)
        self.h = rr.rr_scene_create(*arrays, self.mesh.materials)

    def __del__(self):
        rr.rr_scene_destroy(self.h)


class _Server:
    def __init__(self, scenes_used, **config):
        self.scenes = scenes_used   # they outlive the server
        self.h = rr.rr_serve_create(**config)

    def __del__(self):
        rr.rr_serve_destroy(self.h)


def _corrected(vertices, rng):
    """The vertices after a smooth map correction of a few centimetres (neighbours move together)."""
    x, y, z = vertices.unbind(1)
    phase = rng.uniform(0.0, 2.0 * math.pi, 4)
    k = 2.0 * math.pi / rng.uniform(15.0, 40.0)
    dz = 0.03 * torch.sin(k * x + phase[0]) * torch.sin(k * y + phase[1])
    dx = 0.02 * torch.sin(k * y + phase[2]) * torch.cos(k * z + phase[3])
    return torch.stack([x + dx, y, z + dz], 1).contiguous()


def _pose(case, mesh, rng):
    if case["scene"] == "room":
        return scenes.pose(*(float(v) for v in rng.uniform(-0.5, 0.5, 2)), 0.5, yaw=float(rng.uniform(-math.pi, math.pi)))
    extent = 60.0 if case["scene"] == "campus" and case["tris"] <= 100_000 else 100.0
    return scenes.random_pose(mesh, rng, extent=extent)


def _sensor(case, rng, **kw):
    options = {}
    if case["post"]:
        options.update(speckle=True, noise=True, noise_sys=1e-4, noise_amb=5e-5, blur_sigma_bins=1.5)
    if case["post"] == 2:
        options.update(perlin=True, az_pattern_sigma=1.2, beam_aspect=2.0, min_energy=1e-7, range_falloff=1.0)
    if case["scene"] == "room":
        options.update(beam_width=math.radians(scenes.TINY_BEAM_WIDTH_DEG))
    size = dict(n_azimuth=case["az"], rays_per_beam=case["rays"], max_bounces=case["bounces"], n_bins=case["bins"])
    return scenes.sensor(**{**size, "bin_size": BIN, **options, **kw}, seed=int(rng.integers(1, 1 << 40)),
                         scan_id=int(rng.integers(0, 1 << 20)))


def prepare(case, seed):
    path, rng = case["path"], np.random.Generator(np.random.PCG64(seed))
    if path == "returns":
        g = torch.Generator(device="cuda").manual_seed(seed)
        n, az, bins = case["n"], case["az"], case["bins"]
        column = torch.randint(0, az, (n,), generator=g, device="cuda", dtype=torch.int32).sort().values
        # returns cluster in range around a wall of each column, the rest is spread out
        wall = torch.rand(az, generator=g, device="cuda")[column.long()]
        far = torch.where(torch.rand(n, generator=g, device="cuda") < 0.7,
                          wall + 0.01 * torch.randn(n, generator=g, device="cuda"),
                          torch.rand(n, generator=g, device="cuda")).abs()
        energy = torch.exp(4.0 * torch.randn(n, generator=g, device="cuda") - 12.0)
        return dict(path=path, column=column, bin=(far * bins).to(torch.int32), energy=energy,
                    out=torch.zeros(az, bins, device="cuda"))
    if path == "db":
        g = torch.Generator(device="cuda").manual_seed(seed)
        polar = torch.exp(6.0 * torch.randn(case["n"], generator=g, device="cuda") - 15.0)
        polar[torch.rand(case["n"], generator=g, device="cuda") < 0.4] = 0.0   # pixels without a return
        return dict(path=path, polar=polar, out=torch.zeros(case["n"], dtype=torch.uint8, device="cuda"))

    scene = _Scene(case["scene"], case["tris"])
    s = dict(path=path, scene=scene)
    if path in ("batch", "serve"):
        if path == "batch":
            s["poses"] = scenes.trajectory(scene.mesh, case["scans"], step=0.25, seed=seed, extent=60.0)
        else:   # half of the robots drive in the room
            s["room"] = _Scene("room", 0)
            s["poses"] = [_pose(case if i % 2 else dict(case, scene="room"), scene.mesh, rng)
                          for i in range(case["scans"])]
        s["params"] = []
        sizes = np.random.Generator(np.random.PCG64(case["scans"]))   # the mix of sensors belongs to the case
        for _ in s["poses"]:
            kw = dict(rays_per_beam=int(sizes.integers(16, case["rays"] + 1)))
            if path == "serve":
                kw.update(max_bounces=int(sizes.integers(min(3, case["bounces"]), case["bounces"] + 1)),
                          n_bins=int(sizes.integers(min(500, case["bins"]), case["bins"] + 1)))
            s["params"].append(_sensor(case, rng, **kw))
        s["out"] = [torch.zeros(p["n_azimuth"], p["n_bins"], device="cuda") for p in s["params"]]
        if path == "serve":
            s["server"] = _Server([scene, s["room"]], slots=4, memory_budget=32 << 30)
        return s

    s["pose"], s["params"] = _pose(case, scene.mesh, rng), _sensor(case, rng)
    shape = (case["az"], case["bins"])
    s["out"] = torch.zeros(shape, pin_memory=True) if case.get("host") else torch.zeros(shape, device="cuda")
    if case.get("wide"):
        rr.rr_batch_config_set(scene.h, node_format=rr.RR_NODES_WIDE8)
    if path == "step":
        # a scene that is rebuilt for every scan uses the cheaper build
        rr.rr_batch_config_set(scene.h, bvh_build=rr.RR_BVH_LBVH)
        v = _corrected(_mesh(case["scene"], case["tris"])[1][0], rng)
        s["vertices"] = v.cpu().pin_memory() if case["host"] else v
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    path = s["path"]
    if path == "returns":
        rr.rr_accumulate_returns(s["column"], s["bin"], s["energy"], *s["out"].shape, s["out"])
    elif path == "db":
        rr.rr_polar_to_db_u8(s["polar"], 60.0, s["out"])
    elif path == "batch":
        rr.rr_scan_batch_async(s["scene"].h, s["poses"], s["params"], s["out"])
    elif path == "serve":
        where = (s["room"].h, s["scene"].h)
        tickets = [rr.rr_serve_submit(s["server"].h, where[i % 2], q, p, o)
                   for i, (q, p, o) in enumerate(zip(s["poses"], s["params"], s["out"]))]
        for t in tickets:
            rr.rr_serve_wait(s["server"].h, t)
            rr.rr_serve_result(s["server"].h, t)
    elif path == "static":
        rr.rr_scan_static(s["scene"].h, s["pose"], s["params"], s["out"])
    else:
        if path == "step":
            rr.rr_scene_update_vertices(s["scene"].h, s["vertices"])
        rr.rr_scan(s["scene"].h, s["pose"], s["params"], s["out"])
    return s["out"]


# ------------------------------------------------------------------ least work
def work(case):
    """Inputs read once, outputs written once; operations: per ray and bounce one descent of a
    hierarchy over the triangles (a box test is about 12 operations) and one shading."""
    if case["path"] == "returns":
        return dict(bytes=12 * case["n"] + 4 * case["az"] * case["bins"], flops=3 * case["n"])
    if case["path"] == "db":
        return dict(bytes=5 * case["n"], flops=4 * case["n"])
    tris = dict(room=1_904, city=5_000_000).get(case["scene"], case["tris"])
    scans = case.get("scans", 1)
    many = scans > 1
    rays = scans * case["az"] * ((16 + case["rays"]) / 2 if many else case["rays"])
    pixels = scans * case["az"] * case["bins"]
    # 14 bytes of indices and material per triangle, about half a vertex each
    return dict(bytes=20 * tris + 4 * pixels, flops=rays * case["bounces"] * (24 * math.log2(tris) + 100))


def exact(case, seed):
    """64-bit results where they can be had: a scan's image depends on discrete decisions of every
    traced path, so only the binning and the display map have a value here."""
    if case["path"] == "returns":
        s = prepare(case, seed)
        flat = s["column"].long() * case["bins"] + s["bin"].long()
        inside = (s["bin"] >= 0) & (s["bin"] < case["bins"])
        out = torch.zeros(case["az"] * case["bins"], dtype=torch.float64, device="cuda")
        out.index_add_(0, flat[inside], s["energy"][inside].double())
        return out.reshape(case["az"], case["bins"])
    if case["path"] == "db":
        e = prepare(case, seed)["polar"].double()
        v = torch.where(e > 0, (255.0 * (10.0 * torch.log10(e) + 60.0) / 60.0).clamp(0.0, 255.0), torch.zeros_like(e))
        return torch.floor(v + 0.5).to(torch.uint8)
    return None
