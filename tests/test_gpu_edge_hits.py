"""Rays aimed at edges that two triangles share, from every side: none may
pass between the two, and the node formats and builds agree on the distance
up to rounding and on the triangle up to the choice between the two.  Needs
a GPU."""
import numpy as np
import pytest

from paper_2310_03505_gb300 import rr, scenes
from tests import parity as P
from tests.test_gpu_wide_bvh import segments_with

pytestmark = pytest.mark.gpu

N_AZ = 720
SENSOR = np.array([1.3, -0.7, 2.1])
TURNS = {   # the sensor's quaternion: beams through all azimuths of a tilted plane
    "level": (1.0, 0.0, 0.0, 0.0),
    "about x": (np.sqrt(0.5), np.sqrt(0.5), 0.0, 0.0),
    "about y": (np.sqrt(0.5), 0.0, np.sqrt(0.5), 0.0),
    "skew": tuple(np.array([0.8, 0.3, -0.4, 0.33166247903554])),
}


def rotate(q, v):
    w, u = q[0], np.asarray(q[1:])
    return v + 2.0 * w * np.cross(u, v) + 2.0 * np.cross(u, np.cross(u, v))


def folds(quat, far):
    """One fold (two triangles with a common edge, folded away from the
    sensor) in each beam, the beam's axis through its edge; a closed box around
    them; far: and a triangle that reaches 1,000 km (nodes with float boxes)."""
    rng = np.random.Generator(np.random.PCG64(20))
    a = 2.0 * np.pi * np.arange(N_AZ) / N_AZ
    d = rotate(quat, np.stack([np.cos(a), np.sin(a), np.zeros(N_AZ)], 1))
    dist = np.exp(rng.uniform(np.log(5.0), np.log(20.0), N_AZ))
    e = np.cross(d, rng.normal(size=(N_AZ, 3)))
    e /= np.linalg.norm(e, axis=1, keepdims=True)
    s = np.cross(e, d)
    at = SENSOR + dist[:, None] * d
    up, t = rng.uniform(0.1, 0.9, (2, N_AZ, 1))
    ends = np.stack([at - 0.01 * t * e, at + 0.01 * (1.0 - t) * e], 1)   # the edge
    wings = np.stack([at + w * 0.012 * s + 0.006 * d + 0.004 * (up - 0.5) * e for w in (-1.0, 1.0)], 1)
    v = np.concatenate([ends, wings], 1).reshape(-1, 3)
    i = 4 * np.arange(N_AZ)[:, None]
    tri = np.concatenate([i + [0, 1, 2], i + [1, 0, 3]], 1).reshape(-1, 3)
    c = 50.0 * (np.array([[x, y, z] for x in (-1, 1) for y in (-1, 1) for z in (-1, 1)]))
    q = [(0, 1, 3, 2), (4, 6, 7, 5), (0, 4, 5, 1), (2, 3, 7, 6), (0, 2, 6, 4), (1, 5, 7, 3)]
    box = len(v) + np.array([t for k in q for t in ((k[0], k[1], k[2]), (k[0], k[2], k[3]))])
    v, tri = np.concatenate([v, c]), np.concatenate([tri, box])
    if far:
        g = 1e6 * np.array([[1, 0, 0], [-0.5, 0.8, 0], [-0.5, -0.8, 0]]) - [0, 0, 60.0]
        v, tri = np.concatenate([v, g]), np.concatenate([tri, [[len(v), len(v) + 1, len(v) + 2]]])
    sc = scenes.Scene("folds", v.astype(np.float32), tri.astype(np.uint32), np.zeros(len(tri), np.uint16),
                      [scenes.MATERIALS["metal"]])
    return sc, dist


@pytest.mark.parametrize("far", [False, True])
@pytest.mark.parametrize("turn", TURNS)
def test_no_ray_passes_a_shared_edge(rrlib, turn, far):
    quat = TURNS[turn]
    sc, dist = folds(quat, far)
    pz = dict(p=tuple(np.float32(SENSOR)), q=tuple(np.float32(quat)))
    params = scenes.sensor(n_azimuth=N_AZ, rays_per_beam=1, max_bounces=1, n_bins=2000, bin_size=0.05, beam_width=0.0,
                           elevation=0.0)
    h = P.gpu_scene(sc)
    try:
        got = []
        for build in (rr.RR_BVH_LBVH, rr.RR_BVH_SAH_TOP):
            rr.rr_batch_config_set(h, bvh_build=build)
            got += [segments_with(h, pz, params, f)[1] for f in (rr.RR_NODES_BINARY, rr.RR_NODES_WIDE8)]
        for s in got:
            assert np.array_equal(s["az"], np.arange(N_AZ))
            assert np.array_equal(s["tri"] // 2, np.arange(N_AZ)), "a ray passed its fold's edge"
            # the edge lies within 4 half ulps of coordinates below 32 m (its ends, the direction, the hit)
            # across the beam or along it, the faces at 63 degrees to it: far below a tenth of a millimetre
            assert np.max(np.abs(s["t"] - dist)) <= 1e-4
            same = s["tri"] == got[0]["tri"]
            assert np.array_equal(s["t"][same], got[0]["t"][same])
            # the other triangle of the edge: both distances round the same point
            assert np.all(np.abs(s["t"] - got[0]["t"]) <= 32 * 2.0 ** -24 * 32.0)
    finally:
        rr.rr_scene_destroy(h)
