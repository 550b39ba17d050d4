"""Branches that depend on the size of a call, at the sizes where they change: the piece height of
pic_render_static, its list of survivors and its batches of records."""
import numpy as np
import pytest

from scenes import custom_scene, make_rig

pytestmark = pytest.mark.gpu
CAR = (4.5, 1.9, 1.5)


def soup(seed, n_tris, E, A, H, W, K=2, spread=25.0):
    """E x A agents in a soup of n_tris small triangles; camera 1 looks back from another mount."""
    rng = np.random.default_rng(seed)
    c = np.stack([rng.uniform(-spread, spread, n_tris), rng.uniform(-spread, spread, n_tris), rng.uniform(0.0, 4.0, n_tris)], axis=1)
    tris = (c[:, None, :] + rng.uniform(-3, 3, size=(n_tris, 3, 3))).astype(np.float32)
    rig = make_rig(tuple(np.arange(K) * 170.0), 80.0, 70.0, W, H, mount=(1.0, 0.2, 1.4))
    poses = rng.uniform(-10, 10, size=(E, A, 3)).astype(np.float32)
    return custom_scene(tris, rng.integers(0, 200, n_tris).astype(np.uint8), poses, np.tile(np.array(CAR, np.float32), (E, A, 1)), rig, H, W)


@pytest.mark.parametrize("n_tris,E,A,H,W,offset", [
    (1, 1, 1, 17, 33, 0),            # one triangle, pieces of 16 rows, the last of one row
    (127, 1, 2, 64, 64, 0),          # one round of tests less a thread
    (257, 1, 3, 70, 100, 1),         # two rounds and a thread; outputs that allow no vector store
    (1500, 1, 2, 64, 80, 0),         # several hundred survivors per tile: the list is emptied more than once
    (300, 2, 60, 96, 64, 0),         # more CTAs than two per multiprocessor: pieces of 64 rows
])
def test_static_pieces_lists_and_alignment(n_tris, E, A, H, W, offset):
    import torch
    import paper_2607_26005_b200 as pic
    from tests.gpu_util import CudaRun
    s = soup(n_tris, n_tris, E, A, H, W)
    dev = torch.device("cuda", 0)
    g = CudaRun(s)
    try:
        want = g.render(brute=True)
    finally:
        g.close()
    n = E * A * s.K * H * W
    cls = torch.full((n + offset,), 255, dtype=torch.uint8, device=dev)[offset:]
    dep = torch.full((n + offset,), -1.0, dtype=torch.float16, device=dev)[offset:]
    put = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    pic.render_static(E, A, s.K, H, W, s.near, s.far, put(s.tri_xyz), put(s.tri_class), put(s.poses), put(s.dims), s.rig, cls, dep)
    V = E * A * s.K
    c, d = cls.cpu().numpy().reshape(V, H, W), dep.cpu().numpy().reshape(V, H, W)
    assert (c == want[0]).all()
    assert (np.abs(d.view(np.uint16).astype(int) - want[1].view(np.uint16).astype(int)) <= 1).all()
    assert pic.static_status() == 0


@pytest.mark.parametrize("n_tris,E,A,H,W,K,spread", [
    (40, 1, 1, 8, 16, 1, 25.0),           # one tile of one strip
    (300, 1, 3, 17, 33, 2, 25.0),         # ragged in both directions
    (300, 8, 37, 64, 64, 4, 200.0),       # 1 184 tiles: the most that take one CTA each (on 148 multiprocessors) ...
    (300, 79, 15, 64, 64, 1, 200.0),      # ... and one more
    (3000, 1, 2, 130, 70, 2, 12.0),       # more survivors than the record pool holds
    (20, 1, 120, 64, 64, 1, 25.0),        # more visible box faces than their list holds, all around the cameras
    (4000, 1, 4, 64, 64, 2, 90.0),        # a map of small cells: more grid rows in view than one pass takes
])
def test_calls_with_few_tiles(n_tris, E, A, H, W, K, spread):
    from tests.gpu_util import CudaRun
    from tests.util import assert_same_as_exhaustive
    s = soup(n_tris + A, n_tris, E, A, H, W, K=K, spread=spread)
    g = CudaRun(s)
    try:
        V = E * A * K
        n = min(V, 300)
        a = g.render()
        b = g.render(brute=True, view_first=V - n, view_count=n)
        assert_same_as_exhaustive(a, b, slice(V - n, V))
        c = g.render(depth32=False)
        assert (a[0] == c[0]).all() and (a[1].view(np.uint16) == c[1].view(np.uint16)).all()
    finally:
        g.close()


@pytest.mark.parametrize("n_tris,E,A,H,W,K,spread", [
    (60, 6, 50, 20, 30, 4, 30.0),         # rows of no whole groups of four pixels: scalar stores
    (200, 2, 100, 36, 76, 4, 60.0),       # groups of four but not of sixteen; a second tile narrower than a cell
    (200, 2, 100, 65, 48, 4, 60.0),       # a second tile of a single row
    (3000, 1, 60, 130, 80, 4, 12.0),      # (1 440 tiles) more records and more fragments than a tile's lists hold
    (60, 13, 24, 64, 64, 4, 6.0),         # large primitives around the cameras: cells wholly inside, range tests
])
def test_calls_with_many_tiles(n_tris, E, A, H, W, K, spread):
    test_calls_with_few_tiles(n_tris, E, A, H, W, K, spread)


@pytest.mark.parametrize("side", [15.0, 15.5, 16.0, 40.0])      # pixels: boxes of 16 x 16 and 17 x 17, around the limit of 256, and a large one
@pytest.mark.parametrize("far", [100.0, 10.3])                  # wholly in the depth range, cut by the far plane
def test_antialiased_primitives_around_the_size_limit(side, far):
    import oracle
    from scenes import default_palette
    from tests.gpu_util import CudaRun
    from tests.test_gpu_colour import compare_colour
    H, W = 70, 100
    rig = make_rig((0.0,), 90.0, 80.0, W, H, mount=(0.0, 0.0, 1.5))
    z, fx = 10.0, rig[0, 5]
    tris = []
    for k, (u, v, tilt) in enumerate([(-30.3, -20.2, 0.0), (12.6, -18.4, 0.5), (-9.7, 5.1, 1.0), (30.2, 12.4, 0.3)]):   # tilted squares, pixels off the axis
        h = 0.5 * side * z / fx
        c, y0, z0 = np.array([z, 0.0, 1.5]), -u * z / fx, -v * z / fx
        corners = [c + np.array([tilt * a, y0 + a, z0 + b]) for a, b in ((-h, -h), (h, -h), (h, h), (-h, h))]
        tris += [[corners[0], corners[1], corners[2]], [corners[0], corners[2], corners[3]]]
    s = custom_scene(np.asarray(tris, np.float32), np.repeat([2, 3, 4, 5], 2).astype(np.uint8), np.zeros((1, 1, 3), np.float32),
                     np.array([[CAR]], np.float32), rig, H, W, far=far)
    pal = default_palette()
    g = CudaRun(s)
    try:
        got, flags = g.render_rgb(pal, True)
    finally:
        g.close()
    ref = oracle.render_rgb(s, pal, True)
    assert flags == 0
    compare_colour(ref, got)


@pytest.mark.parametrize("n_tris,E,A,H,W,K,spread", [
    (300, 4, 50, 65, 129, 4, 60.0),       # 800 views of 6 tiles, the last row and column of one pixel: culled a warp per view
    (300, 8, 50, 64, 70, 4, 60.0),        # 1 600 views of 2 tiles
    (300, 37, 14, 64, 70, 4, 60.0),       # 2 072 of them: the fewest that are culled as a whole (on 148 multiprocessors)
    (100, 5, 26, 250, 500, 1, 40.0),      # 130 views of 32 tiles: as many tiles
    (40, 2, 75, 30, 1990, 4, 6.0),        # the most tiles a view can have there (32), large primitives under the cameras
    (2000, 4, 38, 130, 80, 4, 10.0),      # tiles whose survivor lists overflow ...
    (2000, 5, 38, 130, 80, 4, 10.0),      # ... in views culled as a whole
])
def test_views_of_several_tiles(n_tris, E, A, H, W, K, spread):
    test_calls_with_few_tiles(n_tris, E, A, H, W, K, spread)


@pytest.mark.parametrize("E,A,H,W", [
    (1, 2, 128, 320),                     # 10 tiles: their frusta and the image's are 121 entries, one block of the set-up kernel
    (1, 2, 64, 700),                      # 11 tiles: 132, two blocks
    (1, 3, 700, 1300),                    # 231 tiles: 20 blocks; 1 386 tiles in all, culled a warp per tile
    (1, 2, 700, 1300),                    # ... 924 of them: a CTA per tile
])
def test_images_of_many_tiles(E, A, H, W):
    import oracle
    from scenes import default_palette
    from tests.test_gpu_colour import compare_colour
    from tests.gpu_util import CudaRun
    test_calls_with_few_tiles(120, E, A, H, W, 2, 40.0)
    s = soup(120 + A, 120, E, A, H, W, K=2, spread=40.0)
    g = CudaRun(s)
    try:
        got, flags = g.render_rgb(default_palette(), False)
        assert flags == 0
        compare_colour(oracle.render_rgb(s, default_palette(), False, [1, 2 * E * A - 1]), got[[1, 2 * E * A - 1]])
    finally:
        g.close()


@pytest.mark.parametrize("E,A", [(1, 2), (37, 12), (38, 12), (37, 14), (38, 14)])       # 4 tiles per view: one per CTA up to 2 072 tiles (148 multiprocessors), else four
def test_antialiased_calls_with_few_and_many_tiles(E, A):
    from scenes import default_palette
    from tests.gpu_util import CudaRun
    s = soup(A, 80, E, A, 70, 100, K=1, spread=40.0)
    g = CudaRun(s)
    try:
        pal = default_palette()
        whole, flags = g.render_rgb(pal, True)
        part, _ = g.render_rgb(pal, True, view_first=E * A - 2, view_count=2)        # the same views in a call of few tiles
        assert flags == 0
        assert (np.abs(whole[-2:].astype(int) - part[-2:].astype(int)) <= 1).all()
    finally:
        g.close()


@pytest.mark.parametrize("E,A,H,W", [(1, 5, 40, 40), (1, 11, 500, 384), (2, 24, 250, 300)])    # one part, two parts of an odd number of views, five parts
def test_host_images_in_parts(E, A, H, W):
    from tests.gpu_util import CudaRun
    s = soup(E * A, 200, E, A, H, W, K=3, spread=30.0)
    g = CudaRun(s)
    try:
        want = g.render(depth32=False)
        for _ in range(2):
            cls, dep = np.full((E, A, 3, H, W), 255, np.uint8), np.full((E, A, 3, H, W), -1, np.float16)
            g.scene.render_host(np.ascontiguousarray(s.poses), np.ascontiguousarray(s.dims), s.rig, cls, dep)
            assert (cls.reshape(want[0].shape) == want[0]).all()
            assert (dep.reshape(want[1].shape).view(np.uint16) == want[1].view(np.uint16)).all()
    finally:
        g.close()


@pytest.mark.parametrize("E,A,H,W,K", [
    (4, 3, 40, 64, 2),                    # few tiles
    (64, 12, 40, 64, 2),                  # a warp per tile
    (64, 14, 130, 96, 2),                 # culled a warp per view
])
def test_poses_far_outside_the_map(E, A, H, W, K):
    """Finite poses more than 2^31 grid cells from the map, in every direction: nothing but other agents at the same place is in view."""
    from tests.gpu_util import CudaRun
    from tests.util import assert_same_as_exhaustive
    s = soup(E + A, 200, E, A, H, W, K=K, spread=40.0)
    poses = s.poses.copy()
    far = np.array([1e9, 1e11, 1e12, 1e30, 3e38], np.float32)
    for i in range(E * A // 2):
        poses.reshape(-1, 3)[2 * i, i % 2] = far[i % 5] * (1 if (i // 2) % 2 else -1)
    g = CudaRun(s)
    try:
        V = E * A * K
        n = min(V, 300)
        a = g.render(poses=poses)
        assert_same_as_exhaustive(a, g.render(poses=poses, brute=True, view_first=V - n, view_count=n), slice(V - n, V))
    finally:
        g.close()


@pytest.mark.parametrize("E,A,H,W", [(40, 12, 64, 64), (60, 12, 70, 130)])       # culled a warp per tile, a warp per view
def test_antialiased_depth_ties_are_the_same_every_time(E, A, H, W):
    """Large triangles of many classes in one plane: equal depths everywhere, so the image shows the order of the lists."""
    from scenes import default_palette
    from tests.gpu_util import CudaRun
    rng = np.random.default_rng(W)
    n = 150
    yz = rng.uniform(-30.0, 30.0, size=(n, 1, 2)) + rng.uniform(-12.0, 12.0, size=(n, 3, 2))
    tris = np.concatenate([np.full((n, 3, 1), 20.0), yz], axis=2).astype(np.float32)
    poses = np.zeros((E, A, 3), np.float32)
    poses[..., 0] = rng.uniform(-10.0, 5.0, (E, A)); poses[..., 1] = rng.uniform(-20.0, 20.0, (E, A))
    dims = np.tile(np.array(CAR, np.float32), (E, A, 1))
    s = custom_scene(tris, rng.integers(2, 9, n).astype(np.uint8), poses, dims, make_rig((0.0,), 90.0, 70.0, W, H), H, W, env_map_id=np.zeros(E, np.int32))
    g = CudaRun(s)
    try:
        first, _ = g.render_rgb(default_palette(), True)
        for _ in range(4):
            again, _ = g.render_rgb(default_palette(), True)
            assert (first == again).all()
    finally:
        g.close()


def crowd(A, H, W, K, hfov, vfov, spacing, size, walls=0):
    """A agents on a lattice in one environment, each seeing up to all the others; `walls`: so many large primitives around them."""
    rng = np.random.default_rng(A + walls)
    n = int(np.ceil(np.sqrt(A)))
    xy = np.stack(np.meshgrid(np.arange(n), np.arange(n)), axis=-1).reshape(-1, 2)[:A] * spacing + rng.uniform(-0.3, 0.3, (A, 2))
    xy -= xy.mean(0)
    poses = np.concatenate([xy, rng.uniform(-3.1, 3.1, (A, 1))], axis=1)[None].astype(np.float32)
    tris = []
    r, a = 35.0, 0.0
    for _ in range(walls):                                 # upright 9 m walls on rings 2 m apart: too large for the cells of a map of this many
        c, d = np.array([r * np.cos(a), r * np.sin(a), 0.0]), np.array([-4.5 * np.sin(a), 4.5 * np.cos(a), 0.0])
        p = [c - d, c + d, c + d + [0, 0, 2.0], c - d + [0, 0, 2.0]]
        tris += [[p[0], p[1], p[2]], [p[0], p[2], p[3]]]
        a += 10.0 / r
        if a > 2 * np.pi - 10.0 / r:
            r, a = r + 2.0, 0.0
    s = custom_scene(np.asarray(tris, np.float32).reshape(-1, 3, 3), np.repeat(rng.integers(2, 9, walls), 2).astype(np.uint8), poses,
                     np.tile(np.array(size, np.float32), (1, A, 1)), make_rig(tuple(np.arange(K) * 360.0 / K), hfov, vfov, W, H), H, W)
    # how many agents and walls each view has within its horizontal field
    at = np.concatenate([poses[0, :, :2]] + [np.asarray(t)[:, :2].mean(0)[None] for t in tris[::2]])
    rel = at[None] - poses[0, :, None, :2]
    ang = (np.arctan2(rel[..., 1], rel[..., 0])[:, None] - poses[0, :, None, None, 2] - s.rig[None, :, None, 3] + np.pi) % (2 * np.pi) - np.pi
    return s, (np.abs(ang) < np.radians(hfov / 2)).sum(-1).reshape(-1)


@pytest.mark.parametrize("A,H,W,K,hfov,vfov,spacing,size,walls,modes", [
    (320, 64, 64, 1, 120.0, 120.0, 7.5, (2.0, 1.0, 1.2), 0, (False,)),            # a tile per view: some 600 box faces in sight
    (300, 72, 512, 2, 110.0, 30.0, 5.0, (2.5, 1.2, 1.5), 0, (False, True)),       # culled a warp per view
    (100, 64, 1024, 6, 120.0, 40.0, 2.0, (0.6, 0.6, 1.0), 1100, (False, True)),   # large primitives, with the faces
])
def test_views_with_more_items_than_the_cull_list(A, H, W, K, hfov, vfov, spacing, size, walls, modes):
    import oracle
    from scenes import default_palette
    from tests.gpu_util import CudaRun
    from tests.test_gpu_colour import compare_colour
    from tests.util import assert_same_as_exhaustive
    s, seen = crowd(A, H, W, K, hfov, vfov, spacing, size, walls)
    busiest = np.sort(np.argsort(seen)[-3:])
    pal = default_palette()
    g = CudaRun(s)
    try:
        for aa in modes:
            got, flags = g.render_rgb(pal, aa)
            assert flags == 0, f"antialias {aa}: status {flags}"
            # (a mismatch has to lie on a flagged pixel, so the share of those bounds the share of mismatches)
            compare_colour(oracle.render_rgb(s, pal, aa, busiest), got[busiest], max_mismatch_frac=2e-2, max_flag_frac=2e-2)
            for v in busiest:                              # the same views culled a warp per tile
                alone, _ = g.render_rgb(pal, aa, view_first=int(v), view_count=1)
                assert (alone[v] == got[v]).all()
        a = g.render()
        n = min(len(seen), 100)
        assert_same_as_exhaustive(a, g.render(brute=True, view_first=0, view_count=n), slice(0, n))
    finally:
        g.close()


@pytest.mark.parametrize("length,near,hfov,H,W,pitch", [
    (300.0, 0.1, 46.0, 100, 384, 0.0),
    (1000.0, 0.1, 90.0, 100, 192, 0.0),
    (1000.0, 0.02, 46.0, 100, 384, 12.0),
    (3000.0, 0.1, 46.0, 100, 384, -20.0),
])
def test_long_primitives_cut_at_the_near_plane(length, near, hfov, H, W, pitch):
    """Triangles of hundreds of metres that pass the cameras at centimetres: where float32 puts their edges depends on focal length,
    length and distance, and views culled as a whole must not lose a pixel of them."""
    from scenes import default_palette
    from tests.gpu_util import CudaRun
    from tests.util import assert_same_as_exhaustive
    rng = np.random.default_rng(int(length))
    E, A, n = 44, 16, 40
    unit = lambda v: v / np.linalg.norm(v)
    tris = []
    for _ in range(n):
        along, side = unit(rng.normal(size=3) * [1, 1, 0.15]), unit(rng.normal(size=3) * [1, 1, 0.3])
        o = np.array([rng.uniform(-3, 3), rng.uniform(-3, 3), 1.5 + rng.uniform(-0.6, 0.6)])
        a, b = o + along * length * rng.uniform(0.3, 1.0), o - along * length * rng.uniform(0.3, 1.0)
        tris.append([a, b, b + side * rng.uniform(0.2, 3.0)])
    poses = rng.uniform(-3.0, 3.0, (E, A, 3)).astype(np.float32)
    dims = np.full((E, A, 3), 0.01, np.float32)
    rig = make_rig((0.0,), hfov, hfov * H / W, W, H, mount=(0.0, 0.0, 1.5), pitch_deg=pitch)
    s = custom_scene(np.asarray(tris, np.float32), rng.integers(2, 9, n).astype(np.uint8), poses, dims, rig, H, W, near, 200.0, env_map_id=np.zeros(E, np.int32))
    g = CudaRun(s)
    try:
        assert_same_as_exhaustive(g.render(), g.render(brute=True))
        whole, flags = g.render_rgb(default_palette(), True)
        part, flags_part = g.render_rgb(default_palette(), True, view_first=0, view_count=50)       # culled a warp per tile
        assert flags == flags_part == 0 and (np.abs(whole[:50].astype(int) - part[:50].astype(int)) <= 1).all()
    finally:
        g.close()


@pytest.mark.parametrize("copies,step,n_side,dots,dot", [
    (1, 0.375, 3, 8, 0.25),      # primitives of a few pixels: fragments only
    (2, 1.5, 3, 8, 0.25),        # fragments and records at the same depth, each primitive twice
    (3, 2.5, 3, 8, 0.25),        # 27 records
    (8, 4.0, 2, 8, 0.25),        # 32 records, the most a tile holds, and 40 survivors: set up in two passes
    (9, 4.0, 2, 8, 0.25),        # one more than it holds
    (7, 4.0, 2, 10, 0.75),       # 28 records and 90 fragments, which fit the memory they share ...
    (7, 4.0, 2, 16, 0.75),       # ... and 144, which do not
    (1, 0.75, 1, 26, 0.75),      # 243 fragments and hardly a record
])
def test_equal_depths_and_pixel_centres_on_edges(copies, step, n_side, dots, dot):
    """Walls of squares that share their edges, facing the camera at whole distances, so that depths are exactly equal and edges run
    through pixel centres: the lower index wins, and a shared edge belongs to one side."""
    from tests.gpu_util import CudaRun
    from tests.util import assert_same_as_exhaustive
    rng = np.random.default_rng(copies + dots)
    squares = [(8.0, y, z, step) for y in range(n_side) for z in range(n_side)] * copies + [(8.0, 0.25 * i, 0.25, dot) for i in range(dots)]
    tris = []
    for i in rng.permutation(len(squares)):
        x, iy, iz, d = squares[i]
        y0, z0 = (iy - n_side / 2) * d, 1.5 + (iz - n_side / 2) * d
        p = [(x, y0, z0), (x, y0 + d, z0), (x, y0 + d, z0 + d), (x, y0, z0 + d)]
        tris += [[p[0], p[1], p[2]], [p[0], p[2], p[3]]]
    E, A, K = 80, 16, 1
    poses = np.zeros((E, A, 3), np.float32)
    poses[..., 0] = rng.choice([-8.0, 0.0, 4.0], (E, A))
    poses[..., 1] = rng.integers(-8, 9, (E, A)) * 0.125
    s = custom_scene(np.asarray(tris, np.float32), rng.integers(2, 200, len(squares)).repeat(2).astype(np.uint8), poses, np.full((E, A, 3), 0.01, np.float32),
                     make_rig((0.0,), 90.0, 90.0, 64, 64, mount=(0.0, 0.0, 1.5)), 64, 64, env_map_id=np.zeros(E, np.int32))
    g = CudaRun(s)
    try:
        want = g.render(brute=True)
        assert_same_as_exhaustive(g.render(), want)
        few = g.render(view_first=0, view_count=100)
        assert (few[0][:100] == want[0][:100]).all()
    finally:
        g.close()


# (rows of groups of four pixels take this order, and with occlusion counts all)
@pytest.mark.parametrize("H,W,mode", [(70, 100, "class"), (70, 100, "occlusion"), (40, 90, "occlusion"), (40, 92, "rgb"), (130, 68, "class"), (130, 68, "rgb")])
def test_tiles_with_the_horizon_first_up_to_a_number_of_tiles(H, W, mode):
    """Calls at both sides of the line up to which the tiles with the horizon come first give the same images and counts, from the first view
    or a later one on, into the batch's images or the views' own, and the same as the exhaustive kernel or the oracle."""
    import torch
    import oracle
    import paper_2607_26005_b200 as pic
    from scenes import default_palette
    from tests.gpu_util import CudaRun
    from tests.test_gpu_colour import compare_colour
    from tests.util import f16_ulp_distance
    tiles, A, K, skip = -(-H // 64) * -(-W // 64), 16, 4, 37
    line = 160 * torch.cuda.get_device_properties(0).multi_processor_count // tiles      # the most views that take this order
    E = (line + skip) // (A * K) + 1
    V = E * A * K
    s = soup(H + W, 150, E, A, H, W, K=K, spread=40.0)
    g = CudaRun(s)

    def run(first, n, relative):
        """The images (and counts) of `n` views from `first` on (0: all), one array per view."""
        views = slice(first, first + n) if n else slice(0, V)
        g.scene.set_option(pic.OPT_OUT_RELATIVE, 1 if relative else 0)
        try:
            if mode == "rgb":
                return [g.render_rgb(default_palette(), False, view_first=first, view_count=n)[0][slice(0, n) if relative else views]]
            counts = torch.zeros((E, A, K, A, 2), dtype=torch.int32, device=g.dev)
            g.scene.set_option(pic.OPT_OCCLUSION, counts if mode == "occlusion" else 0)
            cls, d16, _ = g.render(depth32=False, view_first=first, view_count=n)
            return [a[slice(0, n) if relative else views] for a in (cls, d16.view(np.uint16))] + [counts.cpu().numpy().reshape(V, A, 2)[views]]
        finally:
            g.scene.set_option(pic.OPT_OUT_RELATIVE, 0)
            g.scene.set_option(pic.OPT_OCCLUSION, 0)

    try:
        whole = run(0, 0, False)                           # more tiles than the line: in order
        for first, n, relative in ((0, line, False), (skip, line, False), (skip, line, True), (skip, line - 1, False)):
            for got, want in zip(run(first, n, relative), whole):
                assert (got == want[first:first + n]).all(), (first, n, relative)
        last = run(skip, line, False)
        if mode == "rgb":
            ids = np.array([skip, skip + line // 2, skip + line - 1])
            compare_colour(oracle.render_rgb(s, default_palette(), False, ids), last[0][ids - skip])
        else:
            n = 40
            cls, d16, _ = g.render(brute=True, depth32=False, view_first=skip + line - n, view_count=n)
            assert (last[0][-n:] == cls[skip + line - n:skip + line]).all()
            assert (f16_ulp_distance(last[1][-n:], d16[skip + line - n:skip + line]) <= 1).all()
    finally:
        g.close()


@pytest.mark.parametrize("copies,step,n_side,dots,dot", [
    (8, 4.0, 2, 8, 0.25),        # 32 records, the most a tile holds
    (9, 4.0, 2, 8, 0.25),        # one more than it holds
    (7, 4.0, 2, 10, 0.75),       # 28 records and 90 fragments, which fit the memory they share ...
    (7, 4.0, 2, 16, 0.75),       # ... and 144, which do not
    (1, 0.75, 1, 26, 0.75),      # 243 fragments and hardly a record
])
def test_limits_of_a_tiles_lists_in_colour_and_with_counts(copies, step, n_side, dots, dot):
    """The squares above as plain colours, which are the class image's, and with other agents among them and occlusion counts, which are the same
    when every tile is left to the cooperative kernel."""
    import torch
    import paper_2607_26005_b200 as pic
    from scenes import default_palette
    from tests.gpu_util import CudaRun
    rng = np.random.default_rng(copies + dots)
    squares = [(8.0, y, z, step) for y in range(n_side) for z in range(n_side)] * copies + [(8.0, 0.25 * i, 0.25, dot) for i in range(dots)]
    tris = []
    for x, iy, iz, d in squares:
        y0, z0 = (iy - n_side / 2) * d, 1.5 + (iz - n_side / 2) * d
        p = [(x, y0, z0), (x, y0 + d, z0), (x, y0 + d, z0 + d), (x, y0, z0 + d)]
        tris += [[p[0], p[1], p[2]], [p[0], p[2], p[3]]]
    classes = rng.integers(2, 200, len(squares)).repeat(2).astype(np.uint8)
    E, A, K = 80, 16, 1
    poses = np.zeros((E, A, 3), np.float32)
    poses[..., 0] = rng.choice([-8.0, 0.0, 4.0], (E, A))
    poses[..., 1] = rng.integers(-8, 9, (E, A)) * 0.125
    rig = make_rig((0.0,), 90.0, 90.0, 64, 64, mount=(0.0, 0.0, 1.5))
    for size in ((0.01, 0.01, 0.01), (0.3, 0.3, 1.2)):       # the cameras look over the boxes
        s = custom_scene(np.asarray(tris, np.float32), classes, poses, np.tile(np.array(size, np.float32), (E, A, 1)), rig, 64, 64, env_map_id=np.zeros(E, np.int32))
        g = CudaRun(s)
        try:
            cls, d16, _ = g.render(depth32=False)
            palette = np.asarray(default_palette())
            rgb, flags = g.render_rgb(palette, False)
            of_map = cls != s.agent_class                    # (boxes are shaded)
            assert flags == 0 and of_map.mean() > 0.5 and (rgb[of_map] == palette[cls[of_map]]).all()
            results = []
            for debug in (0, 4):                             # 4: the cooperative kernel alone
                counts = torch.zeros((E, A, K, A, 2), dtype=torch.int32, device=g.dev)
                g.scene.set_option(pic.OPT_OCCLUSION, counts)
                c, d, _ = g.render(depth32=False, debug_flags=debug)
                g.scene.set_option(pic.OPT_OCCLUSION, 0)
                assert (c == cls).all() and (d.view(np.uint16) == d16.view(np.uint16)).all()
                results.append(counts.cpu().numpy())
            assert (results[0] == results[1]).all() and (size[0] < 0.1 or results[0][..., 0].any())
        finally:
            g.close()
