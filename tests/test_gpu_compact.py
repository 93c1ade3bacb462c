"""The compact 4-ary nodes that traces walk (needs a GB300): closest hits equal the
brute-force definition (oracle.trace_brute) where the grid's arithmetic is at its
limits, and the other layouts' nodes take over where it does not apply."""
import numpy as np
import pytest

import oracle
from paper_2305_16652_gb300 import gen, hcc
from parity import compare_hits
from test_gpu_layouts import _rays, _trace

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = hcc.hcc_create(0)
    yield c
    hcc.hcc_destroy(c)


def _check(ctx, tris, org, dir_, layout="exact"):
    """Closest and any hits against brute force, by each walk: four lanes per ray (auto, for this
    many rays), one thread per ray, and warps that take new rays."""
    bvh = gen.build_bvh(tris)
    h = hcc.hcc_bvh_upload(ctx, bvh, layout=layout)
    try:
        ref = oracle.trace_brute(tris, org, dir_)
        for schedule in ("auto", "per_ray", "refill"):
            hcc.hcc_set_trace_schedule(ctx, schedule)
            compare_hits(_trace(ctx, h, org, dir_), ref)
            occl = _trace(ctx, h, org, dir_, any_hit=True)["prim"] >= 0
            assert np.array_equal(occl, ref["prim"] >= 0), schedule
        return ref
    finally:
        hcc.hcc_set_trace_schedule(ctx, "auto")
        hcc.hcc_bvh_destroy(h)


@pytest.mark.parametrize("n", [1, 2, 7, 31, 32, 33, 1000, 38912, 50000, 50001, 70000, 70001, 80000, 155649, 160000])
def test_partial_warps_and_first_refills(ctx, n):
    """Wavefronts that end inside a warp, on both sides of the sizes where four lanes per ray give way
    to one (50,000 for any hit, 70,000 for closest), and around the first slots taken by refilling."""
    tris = gen.random_tris(3, 60, mu=-1.5)
    org, dir_ = _rays(n, n, tris)
    _check(ctx, tris, org, dir_)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("distance", [0.0, 3.0, 6.0, 100.0])
def test_axis_parallel_and_distant_rays(ctx, axis, distance):
    """Directions with two zero components, from inside, within and beyond the grid's reach
    (where a ray is measured from its entry into the scene)."""
    tris = gen.random_tris(5, 400, mu=-1.5)
    rng = np.random.default_rng(axis)
    n = 1500
    o = rng.random((n, 3))
    d = np.zeros((n, 3))
    d[:, axis] = np.where(rng.random(n) < 0.5, 1.0, -1.0)
    if distance:
        o[:, axis] = 0.5 - d[:, axis] * (distance + 0.5)
    d[n // 2:] += rng.normal(scale=1e-3, size=(n - n // 2, 3))  # and nearly parallel ones
    org = np.concatenate([o, np.full((n, 1), 1e-4)], 1).astype(np.float32)
    dir_ = np.concatenate([d, np.full((n, 1), np.inf)], 1).astype(np.float32)
    ref = _check(ctx, tris, org, dir_)
    assert (ref["prim"] >= 0).sum() > 100


@pytest.mark.parametrize("scale", [1e-6, 1.0, 1e5])
def test_direction_and_scene_scales(ctx, scale):
    tris = (gen.random_tris(9, 300, mu=-1.5) * np.float32(scale)).astype(np.float32)
    org, dir_ = _rays(11, 2000, tris)
    org[:, 3] = 0.0
    dir_[:, :3] *= np.float32(37.0)  # not normalised
    dir_[::3, 3] = np.float32(0.02 * scale)  # short intervals, and empty ones
    dir_[1::7, 3] = 0.0
    _check(ctx, tris, org, dir_)


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_flat_scene(ctx, axis):
    tris = gen.random_tris(13, 200, mu=-1.5).reshape(-1, 3, 3)
    tris[:, :, axis] = 0.25
    tris = np.ascontiguousarray(tris.reshape(-1, 9))
    org, dir_ = _rays(17, 2000, tris)
    org[: 200, axis] = 0.25  # rays in the plane itself
    _check(ctx, tris, org, dir_)


def test_negative_and_late_intervals(ctx):
    tris = gen.random_tris(19, 400, mu=-1.5)
    org, dir_ = _rays(23, 2000, tris)
    org[:1000, 3] = -1.0
    org[1000:, 3] = 0.7
    _check(ctx, tris, org, dir_)


@pytest.mark.parametrize("layout", ["quantised", "exact", "wide"])
def test_negative_intervals_over_the_layouts_nodes(ctx, layout):
    """Hits behind the origin, where distances and the best hit are negative."""
    tris = gen.random_tris(19, 2000, mu=-2.0)
    org, dir_ = _rays(23, 4000, tris)
    org[:, 3] = -10.0
    dir_[::2, 3] = 0.0
    try:
        hcc.hcc_set_trace_nodes(ctx, "layout")
        ref = _check(ctx, tris, org, dir_, layout)
        assert (ref["t"] < 0).sum() > 200
    finally:
        hcc.hcc_set_trace_nodes(ctx, "auto")


@pytest.mark.parametrize("layout", ["quantised", "exact", "wide"])
def test_scene_that_does_not_suit_the_grid(ctx, layout):
    """Detail far below the grid's step (a cloud of 1e-6 units in a scene of 1): the layout's nodes are walked."""
    small = (gen.random_tris(29, 300, mu=-1.5) * np.float32(1e-6)).astype(np.float32)
    far = np.array([[0, 0, 1, 1, 0, 1, 0, 1, 1]], np.float32)
    tris = np.ascontiguousarray(np.concatenate([small, far]))
    org, dir_ = _rays(31, 2000, small)
    org[:, 3] = 0.0
    ref = _check(ctx, tris, org, dir_, layout)
    assert (ref["prim"] >= 0).any()


def _rays_in_walls(tmin, tmax):
    """A room with a few triangles in it, and rays that run exactly in the planes of its walls."""
    box = np.array([[x, y, z] for x in (0, 10) for y in (0, 3) for z in (0, 8)], np.float32)
    quads = [(0, 1, 3, 2), (4, 5, 7, 6), (0, 1, 5, 4), (2, 3, 7, 6), (0, 2, 6, 4), (1, 3, 7, 5)]
    walls = [box[[a, b, c]].reshape(9) for q in quads for a, b, c in (q[:3], (q[0], q[2], q[3]))]
    tris = np.ascontiguousarray(np.concatenate([np.array(walls, np.float32), gen.random_tris(9, 100, mu=-1.5)]))
    rng = np.random.default_rng(17)
    axis, side = rng.integers(0, 3, 2000), rng.integers(0, 2, 2000)
    o, d = rng.random((2000, 3)) * [8, 2, 6] + [1, 0.5, 1], rng.normal(size=(2000, 3))
    rows = np.arange(2000)
    o[rows, axis] = np.array([10.0, 3.0, 8.0])[axis] * side
    d[rows, axis] = 0.0
    org = np.concatenate([o, np.full((2000, 1), tmin)], 1).astype(np.float32)
    dir_ = np.concatenate([d, np.full((2000, 1), tmax)], 1).astype(np.float32)
    ref = oracle.trace_brute(tris, org, dir_)
    assert (ref["prim"] >= 0).sum() > 500
    return tris, org, dir_, ref


@pytest.mark.parametrize("n", [2000, 100_000])
def test_rays_in_the_planes_of_walls(ctx, n):
    """Rays that run exactly in the plane of a room's wall, a face of the boxes above it, meet the
    walls at its ends as the definition says (a slab test that takes 0 times the reciprocal of a
    zero direction for an exit at t = 0 drops them)."""
    tris, org, dir_, ref = _rays_in_walls(1e-4, np.inf)
    h = hcc.hcc_bvh_upload(ctx, gen.build_bvh(tris), layout="exact")
    try:
        got = _trace(ctx, h, np.tile(org, (n // 2000, 1)), np.tile(dir_, (n // 2000, 1)))
        assert np.array_equal(got.view(np.int32), np.tile(ref, n // 2000).view(np.int32))
    finally:
        hcc.hcc_bvh_destroy(h)


@pytest.mark.parametrize("nodes", ["auto", "layout"])
@pytest.mark.parametrize("layout", ["quantised", "exact", "wide"])
@pytest.mark.parametrize("tmin,tmax", [(1e-4, np.inf), (-50.0, 0.0), (-50.0, np.inf)])
def test_rays_in_the_planes_of_walls_over_every_node(ctx, nodes, layout, tmin, tmax):
    tris, org, dir_, ref = _rays_in_walls(tmin, tmax)
    h = hcc.hcc_bvh_upload(ctx, gen.build_bvh(tris), layout=layout)
    try:
        hcc.hcc_set_trace_nodes(ctx, nodes)
        for schedule in ("auto", "per_ray"):
            hcc.hcc_set_trace_schedule(ctx, schedule)
            assert np.array_equal(_trace(ctx, h, org, dir_).view(np.int32), ref.view(np.int32))
            got = _trace(ctx, h, org, dir_, any_hit=True)
            assert np.array_equal(got["prim"] >= 0, ref["prim"] >= 0)
    finally:
        hcc.hcc_set_trace_nodes(ctx, "auto")
        hcc.hcc_set_trace_schedule(ctx, "auto")
        hcc.hcc_bvh_destroy(h)


def _axis_parallel(rng, n, zeros, o):
    """Rays from o in directions with `zeros` zero components, of either sign, and either sign of zero."""
    d = rng.normal(size=(n, 3))
    order = np.argsort(rng.random((n, 3)), axis=1)
    for k in range(zeros):
        d[np.arange(n), order[:, k]] = np.where(rng.random(n) < 0.5, 0.0, -0.0)
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    org = np.concatenate([o, np.zeros((n, 1))], 1).astype(np.float32)
    return org, np.concatenate([d, np.full((n, 1), np.inf)], 1).astype(np.float32)


@pytest.mark.parametrize("zeros", [1, 2])
@pytest.mark.parametrize("scale", [1e-4 * 2.0**k for k in range(11)])
def test_zero_components_in_small_scenes(ctx, scale, zeros):
    """The far side of the scene lies 1e-4 to 0.1 ahead: the ray's scale is large, and the
    reciprocal of a zero component must not go to infinity with it."""
    tris = (gen.random_tris(37, 400, mu=-1.5) * np.float32(scale)).astype(np.float32)
    rng = np.random.default_rng(zeros)
    org, dir_ = _axis_parallel(rng, 2000, zeros, rng.random((2000, 3)) * scale)
    ref = _check(ctx, tris, org, dir_)
    assert (ref["prim"] >= 0).sum() > 300


@pytest.mark.parametrize("zeros", [1, 2])
@pytest.mark.parametrize("length", [1e-6, 1e-3, 1e3, 2e3, 4e3, 1e4, 1e5, 1e6])
def test_zero_components_and_direction_lengths(ctx, length, zeros):
    tris = (gen.random_tris(41, 400, mu=-1.5) * np.float32(10)).astype(np.float32)
    rng = np.random.default_rng(zeros)
    org, dir_ = _axis_parallel(rng, 2000, zeros, rng.random((2000, 3)) * 10)
    dir_[:, :3] *= np.float32(length)
    ref = _check(ctx, tris, org, dir_)
    assert (ref["prim"] >= 0).sum() > 300


@pytest.mark.parametrize("zeros", [1, 2])
@pytest.mark.parametrize("ahead", [0.0005, 0.001, 0.002, 0.004, 0.006, 0.01])
def test_zero_components_just_before_an_outer_wall(ctx, ahead, zeros):
    """A wall at the edge of a scene of one unit, a little ahead of the rays."""
    rng = np.random.default_rng(zeros)
    wall = np.array([[1, -1, -1, 1, 2, -1, 1, 2, 2], [1, -1, -1, 1, 2, 2, 1, -1, 2]], np.float32)
    tris = np.ascontiguousarray(np.concatenate([np.clip(gen.random_tris(43, 400, mu=-1.5), 0, 0.9), wall])).astype(np.float32)
    o = rng.random((2000, 3))
    o[:, 0] = 1 - ahead
    org, dir_ = _axis_parallel(rng, 2000, zeros, o)
    dir_[:, 0] = np.abs(dir_[:, 0])
    ref = _check(ctx, tris, org, dir_)
    assert (ref["prim"] >= 400).sum() > 300


def test_zero_components_in_a_batch_and_a_server(ctx):
    scales = (0.002, 0.004, 1.0)
    rng = np.random.default_rng(47)
    tris = [(gen.random_tris(51 + k, 400, mu=-1.5) * np.float32(s)).astype(np.float32) for k, s in enumerate(scales)]
    rays = [_axis_parallel(rng, 1000, 1, rng.random((1000, 3)) * s) for s in scales]
    refs = [oracle.trace_brute(t, *r) for t, r in zip(tris, rays)]
    bvhs = [hcc.hcc_bvh_upload(ctx, gen.build_bvh(t), layout="exact") for t in tris]
    cuts = [hcc.hcc_select_cut(ctx, b, 16, 0.125) for b in bvhs]
    batch = hcc.hcc_batch_create(ctx, bvhs, cuts, [0, 1000, 2000, 3000])
    server = hcc.hcc_server_create(0, bvhs, cuts, slots=2, method="hcc", key_bits=16)
    try:
        o, d = (torch.from_numpy(np.concatenate([r[k] for r in rays])).to("cuda:0") for k in (0, 1))
        hits = torch.zeros((3000, 4), dtype=torch.int32, device="cuda:0")
        hcc.hcc_batch_run(ctx, batch, "hcc", o, d, 16, hits)
        hcc.hcc_sync(ctx)
        compare_hits(hcc.hits_to_numpy(hits), np.concatenate(refs))
        for k, (r, ref) in enumerate(zip(rays, refs)):
            for any_hit in (False, True):
                got = np.zeros(1000, oracle.HIT_DTYPE)
                hcc.hcc_server_wait(server, hcc.hcc_server_submit(server, k, *r, got, any_hit=any_hit))
                if any_hit:
                    assert np.array_equal(got["prim"] >= 0, ref["prim"] >= 0)
                else:
                    compare_hits(got, ref)
    finally:
        hcc.hcc_server_destroy(server)
        hcc.hcc_batch_destroy(batch)
        for c in cuts:
            hcc.hcc_cut_destroy(c)
        for b in bvhs:
            hcc.hcc_bvh_destroy(b)


@pytest.mark.parametrize("size", [1.0, 10.0])
@pytest.mark.parametrize("tmin", [-1e2, -3e2, -1e3, -1e4, -1e5, -1e6, -1e8, -1e30, -np.inf])
def test_intervals_that_start_far_behind_the_origin(ctx, tmin, size):
    """Rays measured from a tmin far below zero meet what they meet from a nearer one."""
    tris = (gen.random_tris(61, 2000, mu=-3.0) * np.float32(size)).astype(np.float32)
    org, dir_ = _rays(67, 6000, tris)
    org[:, 3] = tmin
    dir_[::2, 3] = 0.0  # nothing ahead of the origin
    dir_[1::3, 0] = 0.0
    dir_[2::9, :2] = 0.0
    ref = _check(ctx, tris, org, dir_)
    assert (ref["prim"] >= 0).sum() > 300 and (ref["t"] < 0).sum() > 100


def _aimed(seed, n, size, distance, length, zeros):
    """Rays at a scene of `size` units from `distance` scene sizes away, directions of the given length."""
    rng = np.random.default_rng(seed)
    o = rng.random((n, 3))
    d = rng.random((n, 3)) - o
    axis = rng.integers(0, 3, n)
    for k in range(zeros):
        d[np.arange(n), (axis + k) % 3] = 0
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    org = np.concatenate([(o - d * distance) * size, np.zeros((n, 1))], 1).astype(np.float32)
    return org, np.concatenate([d * length, np.full((n, 1), np.inf)], 1).astype(np.float32)


# beyond 10^5 scene sizes the triangle test itself tells apart nothing smaller than the scene's
# triangles on the axes that a ray moves along, so there only rays along an axis have answers that
# do not hang on the last bits of every box test; from 10^9 on every triangle is tested
@pytest.mark.parametrize("distance,zeros", [(1e2, 0), (1e4, 0), (1e9, 0), (1e4, 2), (1e6, 2), (1e7, 2), (1e8, 2), (1e9, 2)])
def test_rays_from_very_far_away(ctx, distance, zeros):
    tris = gen.random_tris(73, 600, mu=-1.5)
    org, dir_ = _aimed(79, 3000, 1.0, distance, 1.0, zeros)
    ref = _check(ctx, tris, org, dir_)
    assert (ref["prim"] >= 0).sum() > (20 if distance == 1e9 and not zeros else 2500)


@pytest.mark.parametrize("size,length", [(1.0, 1e-36), (1.0, 1e-34), (1.0, 1e-19), (1.0, 1e-17), (1.0, 1e30), (1.0, 1e38),
                                         (1e8, 1e-28), (1e8, 1e-20), (1e-8, 1e20), (1e-3, 1e28), (1e-3, 1e37)])
@pytest.mark.parametrize("zeros", [0, 1])
def test_direction_lengths_at_the_ends_of_the_range(ctx, size, length, zeros):
    tris = (gen.random_tris(83, 600, mu=-1.5) * np.float32(size)).astype(np.float32)
    org, dir_ = _aimed(89, 3000, size, 0.5, length, zeros)
    ref = _check(ctx, tris, org, dir_)
    assert (ref["prim"] >= 0).sum() > 2500


def _trace_us(ctx, h, org, dir_, nodes, any_hit):
    hits = torch.zeros((org.shape[0], 4), dtype=torch.int32, device="cuda:0")
    hcc.hcc_set_trace_nodes(ctx, nodes)
    times = []
    for _ in range(7):
        start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        start.record()
        for _ in range(5):
            hcc.hcc_trace(ctx, h, org, dir_, hits, any_hit=any_hit)
        end.record()
        end.synchronize()
        times.append(start.elapsed_time(end) * 200)
    hcc.hcc_set_trace_nodes(ctx, "auto")
    hcc.hcc_sync(ctx)
    return float(np.median(times)), hits.cpu().numpy()


def _detail(ground):
    """An object of 0.3 units (a bumpy ball of 100,000 triangles) on a ground of the given size, and rays
    at it from about 0.6 units away."""
    rng = np.random.default_rng(71)
    m = 224
    a, b = np.meshgrid(np.linspace(0, 2 * np.pi, m + 1), np.linspace(0.02, np.pi - 0.02, m + 1), indexing="ij")
    r = 0.15 * (1 + 0.004 * rng.normal(size=a.shape))
    p = np.stack([r * np.cos(a) * np.sin(b), 0.15 + r * np.cos(b), r * np.sin(a) * np.sin(b)], -1)
    q = [p[:-1, :-1], p[1:, :-1], p[1:, 1:], p[:-1, 1:]]
    g = ground / 2
    plane = [[-g, 0, -g, g, 0, -g, g, 0, g], [-g, 0, -g, g, 0, g, -g, 0, g]]
    tris = np.concatenate([np.concatenate([q[0], q[i], q[i + 1]], -1).reshape(-1, 9) for i in (1, 2)] + [np.array(plane)])
    o = rng.normal(size=(500_000, 3))
    o *= 0.6 / np.linalg.norm(o, axis=1, keepdims=True)
    o[:, 1] = 0.15 + np.abs(o[:, 1])
    d = rng.normal(scale=0.07, size=o.shape) + [0, 0.15, 0] - o
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    pad = [np.full((o.shape[0], 1), x) for x in (1e-4, np.inf)]
    return tris.astype(np.float32), *(np.concatenate([x, y], 1).astype(np.float32) for x, y in zip((o, d), pad))


@pytest.mark.parametrize("ground", [1.0, 30.0, 100.0, 1000.0])
def test_small_detail_in_large_scenes_costs_no_more_than_the_layouts_nodes(ctx, ground):
    """The grid spans the scene, so its step grows with it; rays at an object that the step is coarse
    for must not pay for it (exact nodes: 1.3 times slower on the smallest ground, as on rooms)."""
    tris, org, dir_ = _detail(ground)
    h = hcc.hcc_bvh_upload(ctx, gen.build_bvh(tris), layout="exact")
    try:
        o, d = torch.from_numpy(org).to("cuda:0"), torch.from_numpy(dir_).to("cuda:0")
        for any_hit in (False, True):
            (t_auto, hit), (t_layout, ref) = (_trace_us(ctx, h, o, d, x, any_hit) for x in ("auto", "layout"))
            assert np.array_equal(hit[:, 0] >= 0, ref[:, 0] >= 0)
            assert any_hit or (hit != ref).any(axis=1).sum() <= 5  # ties on an edge
            assert t_auto < 1.15 * t_layout
            if ground == 1.0:
                assert t_auto < t_layout
    finally:
        hcc.hcc_bvh_destroy(h)


def test_traces_that_overlap_after_a_change_of_stream(ctx):
    """Each stream's persistent trace hands out every ray, and so do the traces after them."""
    w = gen.room_workload(1, target_tris=60_000, W=480, H=270, spp=4)
    n = w.rays.n
    o, d = torch.from_numpy(w.rays.org).to("cuda:0"), torch.from_numpy(w.rays.dir).to("cuda:0")
    streams = [torch.cuda.Stream() for _ in range(3)]
    hits = [torch.empty((n, 4), dtype=torch.int32, device="cuda:0") for _ in range(12)]
    h = hcc.hcc_bvh_upload(ctx, w.bvh, layout="exact")
    c = hcc.hcc_create(0, streams[0])
    try:
        ref = torch.empty_like(hits[0])
        hcc.hcc_trace(ctx, h, o, d, ref)
        hcc.hcc_sync(ctx)
        for x in hits:
            x.zero_()
        torch.cuda.synchronize()
        for k, x in enumerate(hits):
            hcc.hcc_set_stream(c, streams[k % 3])
            hcc.hcc_trace(c, h, o, d, x)
        torch.cuda.synchronize()
        hcc.hcc_sync(c)
        assert all(torch.equal(x, ref) for x in hits)
        for s in streams:
            hits[0].zero_()
            torch.cuda.synchronize()
            hcc.hcc_set_stream(c, s)
            hcc.hcc_trace(c, h, o, d, hits[0])
            hcc.hcc_sync(c)
            assert torch.equal(hits[0], ref)
    finally:
        hcc.hcc_destroy(c)
        hcc.hcc_bvh_destroy(h)
