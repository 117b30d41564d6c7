"""Binary nodes on the scene-wide 16-bit grid: a box decoded from the grid
contains the child's float box, so every query finds the hit that the 8-wide
nodes (their own grid per node) find, whatever the scene's size, place and
proportions.  Needs a GPU."""
import numpy as np
import pytest

from paper_2310_03505_gb300 import rr, scenes
from tests import parity as P
from tests.test_gpu_wide_bvh import assert_same_hits, segments_with

pytestmark = pytest.mark.gpu


def placed(scale, offset, rays=8):
    """The tiny room scaled per axis and moved, with a sensor to match."""
    sc, _, p = scenes.config_tiny()
    scale, offset = np.asarray(scale, np.float64), np.asarray(offset, np.float64)
    sc.vertices = (sc.vertices.astype(np.float64) * scale + offset).astype(np.float32)
    s = float(max(scale))
    at = np.array([0.0, 0.0, 0.5]) * scale + offset
    params = scenes.sensor(**{**p, "rays_per_beam": rays, "bin_size": p["bin_size"] * s, "t_min": p["t_min"] * s})
    return sc, scenes.pose(*(float(x) for x in at), yaw=0.3), params


@pytest.mark.parametrize("scale,offset", [
    ((1, 1, 1), (0, 0, 0)),
    ((1e-3, 1e-3, 1e-3), (0, 0, 0)),
    ((1e3, 1e3, 1e3), (0, 0, 0)),
    ((1, 1, 1), (3e4, -2e4, 500)),          # far from the origin: coordinates of a few mm resolution
    ((50, 50, 0.02), (0, 0, 0)),            # extents of 500 m and 6 cm
    ((0.01, 100, 1), (-7, 2e3, 0)),
])
def test_grid_and_wide_nodes_give_the_same_hits(rrlib, scale, offset):
    sc, pz, params = placed(scale, offset)
    h = P.gpu_scene(sc)
    try:
        _, sw, _ = segments_with(h, pz, params, rr.RR_NODES_WIDE8)
        _, sb, _ = segments_with(h, pz, params, rr.RR_NODES_BINARY)
        assert len(sb) >= params["n_azimuth"] * params["rays_per_beam"]
        assert_same_hits(sb, sw)
    finally:
        rr.rr_scene_destroy(h)


@pytest.mark.parametrize("n_tris", [1, 2, 3, 33])
@pytest.mark.parametrize("flat_axis", [0, 1, 2])
def test_flat_and_tiny_scenes(rrlib, n_tris, flat_axis):
    """Triangles of one plane (no extent along an axis), each in a cell of its
    own (overlapping ones would tie up to rounding), seen from beside it."""
    rng = np.random.Generator(np.random.PCG64(7 + n_tris + 100 * flat_axis))
    cell = np.stack(np.divmod(np.arange(36)[:n_tris], 6), 1).repeat(3, 0) - 3.0
    v = np.zeros((3 * n_tris, 3))
    v[:, [k for k in range(3) if k != flat_axis]] = 1.3 * (cell + rng.uniform(0.0, 1.0, (3 * n_tris, 2)))
    v[:, flat_axis] = 2.5
    sc = scenes.Scene("flat", v.astype(np.float32), np.arange(3 * n_tris, dtype=np.uint32).reshape(-1, 3),
                      np.zeros(n_tris, np.uint16), [scenes.MATERIALS["dielectric"]])
    params = scenes.sensor(n_azimuth=90, rays_per_beam=16, max_bounces=2, n_bins=400, bin_size=0.05,
                           beam_width=1.5 if flat_axis == 2 else 0.5)
    h = P.gpu_scene(sc)
    try:
        _, sw, _ = segments_with(h, scenes.pose(0.1, -0.2, 0.3), params, rr.RR_NODES_WIDE8)
        _, sb, _ = segments_with(h, scenes.pose(0.1, -0.2, 0.3), params, rr.RR_NODES_BINARY)
        assert_same_hits(sb, sw)
    finally:
        rr.rr_scene_destroy(h)


def test_the_grid_follows_moved_vertices(rrlib):
    """A rebuild that grows the scene tenfold lays a new grid."""
    sc, _, _ = placed((1, 1, 1), (0, 0, 0))
    big, pz, params = placed((10, 10, 10), (40, 0, 0))
    h, ref = P.gpu_scene(sc), P.gpu_scene(big)
    try:
        rr.rr_scene_update_vertices(h, big.vertices)
        _, s0, _ = segments_with(h, pz, params, rr.RR_NODES_BINARY)
        _, s1, _ = segments_with(ref, pz, params, rr.RR_NODES_BINARY)
        assert_same_hits(s0, s1)
        assert np.array_equal(s0["visits"], s1["visits"])
    finally:
        rr.rr_scene_destroy(h)
        rr.rr_scene_destroy(ref)
