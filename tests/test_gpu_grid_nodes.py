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


def with_ground(reach):
    """The tiny room with one more triangle 2 m below it that reaches `reach`
    metres: its centroid, the hierarchy's place for it, stays in the room, but
    the grid has to cover it."""
    sc, pz, params = scenes.config_tiny()
    n = len(sc.vertices)
    g = np.array([[reach, 0, -2], [-reach / 2, 0.75 * reach, -2], [-reach / 2, -0.75 * reach, -2]], np.float32)
    sc = scenes.Scene("grounded", np.concatenate([sc.vertices, g]),
                      np.concatenate([sc.triangles, np.array([[n, n + 1, n + 2]], np.uint32)]),
                      np.concatenate([sc.material_ids, sc.material_ids[:1]]), sc.materials)
    return sc, pz, params


def triangle_tests(h, pz, params):
    out = np.zeros((params["n_azimuth"], params["n_bins"]), np.float32)
    rr.rr_scene_stats(h, reset=True)
    rr.rr_scan(h, pz, {**params, "count_traversal": True}, out)
    st = rr.rr_scene_stats(h, reset=True)
    return st["tris_tested"] / st["closest_queries"]


@pytest.mark.parametrize("build", [rr.RR_BVH_LBVH, rr.RR_BVH_SAH_TOP])
def test_far_geometry_does_not_coarsen_the_boxes(rrlib, build):
    """Next to a triangle that reaches 100 km the grid's cell is as large as
    the room, and a query on the grid tests most of its triangles; with float
    boxes it tests what it tests without that triangle.  The hits are those of
    the 8-wide nodes, before and after rebuilds that move the triangle in and
    out (the form follows at the build after the next finished scan)."""
    near, pz, params = with_ground(20.0)
    far, _, _ = with_ground(1e5)
    h = P.gpu_scene(far)
    try:
        rr.rr_batch_config_set(h, bvh_build=build)
        ref = P.gpu_scene(near)
        rr.rr_batch_config_set(ref, bvh_build=build)
        few = triangle_tests(ref, pz, params)
        rr.rr_scene_destroy(ref)
        for verts in (None, near.vertices, near.vertices, far.vertices, far.vertices):
            if verts is not None:
                rr.rr_scene_update_vertices(h, verts)
            _, sb, _ = segments_with(h, pz, params, rr.RR_NODES_BINARY)
            _, sw, _ = segments_with(h, pz, params, rr.RR_NODES_WIDE8)
            assert_same_hits(sb, sw)
        # the triangle's own box holds every query: one more test each
        assert triangle_tests(h, pz, params) <= 1.5 * few + 1.0
    finally:
        rr.rr_scene_destroy(h)


@pytest.mark.parametrize("block,rays,cut,count", [(64, 8, 0.0, False), (64, 16, 0.0, False), (128, 3, 1e-7, False),
                                                  (256, 16, 0.0, True), (64, 2, 1e-7, False), (64, 40, 1e-7, True)])
def test_float_boxes_through_every_kernel(rrlib, block, rays, cut, count):
    """The kernels for nodes with float boxes (few and whole warps, the block
    sizes, the counting ones, visibility before and after the shading): the
    images of the 8-wide nodes up to the rounding of the bin sums, and those of
    rr_scan_static, split scans and batches."""
    import torch
    sc, pz, base = with_ground(1e5)
    p = scenes.sensor(**{**base, "rays_per_beam": rays, "min_energy": cut, "count_traversal": count})
    h = P.gpu_scene(sc)
    try:
        out = torch.zeros(p["n_azimuth"], p["n_bins"], device="cuda")
        rr.rr_batch_config_set(h, trace_block=block, node_format=rr.RR_NODES_WIDE8)
        rr.rr_scan(h, pz, p, out)
        ref = out.cpu().numpy()
        assert ref.max() > 0
        rr.rr_batch_config_set(h, node_format=rr.RR_NODES_BINARY)
        for run in ("scan", "split", "batch", "static"):
            out.zero_()
            rr.rr_batch_config_set(h, split_streams=3 if run == "split" else 0)
            if run == "batch":
                rr.rr_scan_batch(h, [pz, pz], [p, p], [out, torch.zeros_like(out)])
            elif run == "static":
                rr.rr_scan_static(h, pz, p, out)
            else:
                rr.rr_scan(h, pz, p, out)
            assert np.max(np.abs(out.cpu().numpy() - ref)) <= 1e-5 * ref.max(), run
    finally:
        rr.rr_scene_destroy(h)


@pytest.mark.parametrize("n_tris", [2, 3, 33])
def test_small_triangles_far_apart(rrlib, n_tris):
    """Millimetre triangles on a circle of 30 m around the sensor: float boxes
    from the smallest hierarchy on."""
    a = 2.0 * np.pi * np.arange(n_tris) / n_tris
    c = np.stack([30.0 * np.cos(a), 30.0 * np.sin(a), np.zeros(n_tris)], 1)
    up, side = np.array([0.0, 0.0, 2e-3]), np.stack([-np.sin(a), np.cos(a), np.zeros(n_tris)], 1) * 2e-3
    v = np.stack([c - up - side, c - up + side, c + up], 1).reshape(-1, 3).astype(np.float32)
    sc = scenes.Scene("specks", v, np.arange(3 * n_tris, dtype=np.uint32).reshape(-1, 3), np.zeros(n_tris, np.uint16),
                      [scenes.MATERIALS["dielectric"]])
    params = scenes.sensor(n_azimuth=99, rays_per_beam=8, max_bounces=2, n_bins=900, bin_size=0.05, beam_width=1e-4)
    h = P.gpu_scene(sc)
    try:
        _, sw, _ = segments_with(h, scenes.pose(), params, rr.RR_NODES_WIDE8)
        _, sb, _ = segments_with(h, scenes.pose(), params, rr.RR_NODES_BINARY)
        assert np.count_nonzero(sb["tri"] != rr.RR_NO_HIT) > 0
        assert_same_hits(sb, sw)
    finally:
        rr.rr_scene_destroy(h)
