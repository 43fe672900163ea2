"""Kernel variants at the sizes where they can go wrong, against the oracle or a
plain reference of the same step."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2603_15186_gb300 import Renderer
    r = Renderer(cut_capacity=1 << 22, record_capacity=1 << 22, pair_capacity=1 << 24)
    yield r
    r.close()


# one cell, one row, one column; rows of one word, of whole words and with a
# remainder; fewer rows than the CTAs' halos and rows that do not divide evenly; one,
# two and four words per thread at their largest; the first map beyond, by its words
# and by its row length; one of corridors off one corridor (levels up to 900, wide
# frontiers)
NAV_MAPS = [(1, 1), (33, 1), (1, 70), (32, 9), (64, 40), (31, 33), (97, 65), (61, 129), (528, 276),
            (511, 384), (511, 385), (511, 896), (511, 1920), (511, 1928), (5247, 64), (6000, 64),
            (700, 900)]


@pytest.mark.parametrize("nx,ny", NAV_MAPS)
def test_nav_fields_and_paths_of_all_map_sizes(R, nx, ny):
    import oracle as O
    rng = np.random.default_rng(nx * 7919 + ny)
    occ = (rng.random((2, ny, nx)) < 0.14).astype(np.uint8)
    if (nx, ny) == (700, 900):
        occ[:] = 0
        occ[:, :, ::3] = 1
        occ[:, ny // 2] = 0
    goals = [(nx // 2, ny // 2), (nx - 1, ny - 1), (0, 0), (nx, 0)]
    for x, y in goals[:3]:
        occ[:, y, x] = 0
    blocked, dist = R.nav_fields(torch.from_numpy(occ).cuda(), goals, 0, 1, 0)
    b_ref = O.nav_blocked(occ, 0, 1, 0)
    assert np.array_equal(blocked.cpu().numpy(), b_ref)
    got = dist.cpu().numpy().view(np.uint32)
    refs = [O.nav_field(b_ref, g) for g in goals]
    for k in range(len(goals)):
        assert np.array_equal(got[k], refs[k]), k
    starts = [(int(rng.integers(nx)), int(rng.integers(ny)), int(rng.integers(4))) for _ in range(40)]
    for max_len in (1, 32, 1500):
        paths, lens = (t.cpu().numpy() for t in R.nav_paths(dist, starts, max_len))
        for a, (i, j, g) in enumerate(starts):
            ref = O.nav_path(refs[g], (i, j), max_len)
            assert lens[a] == len(ref) and np.array_equal(paths[a, :lens[a]], ref), (a, max_len)
            assert not paths[a, lens[a]:].any()


# one, two and four words per thread: the most goals that search on bits and one more
# (152 SMs), which the queue takes
@pytest.mark.parametrize("nx,ny,n", [(64, 40, 190), (64, 40, 191), (300, 200, 228), (300, 200, 229),
                                     (511, 385, 152), (511, 385, 153), (511, 900, 76), (511, 900, 77)])
def test_nav_fields_of_many_goals(R, nx, ny, n):
    """Every goal's field is the one that it has in a call of its own."""
    rng = np.random.default_rng(n)
    occ = torch.from_numpy((rng.random((2, ny, nx)) < 0.12).astype(np.uint8)).cuda()
    goals = np.stack([rng.integers(-1, nx + 1, n), rng.integers(0, ny, n)], 1)
    blocked, dist = R.nav_fields(occ, goals, 0, 1, 0)
    for k in range(0, n, 10):
        b1, d1 = R.nav_fields(occ, goals[k:k + 1], 0, 1, 0)
        assert torch.equal(b1, blocked) and torch.equal(d1[0], dist[k]), k


def test_nav_paths_of_other_fields(R):
    """A field that no breadth-first search gave is followed by the same rule: the
    first neighbour one less than the count so far, else stay and count on."""
    rng = np.random.default_rng(5)
    ny, nx, max_len = 150, 170, 400
    # plateaus and gaps: steps towards the left, some cells off by a few
    dist = (np.arange(nx)[None, :] + rng.integers(0, 3, (ny, nx)) * (rng.random((ny, nx)) < 0.2)).astype(np.uint32)
    dist[:, 60] += 2
    starts = np.stack([rng.integers(0, nx, 60), rng.integers(0, ny, 60), np.zeros(60, int)], 1)
    got = R.nav_paths(torch.from_numpy(dist.view(np.int32))[None].cuda(), starts, max_len)
    paths, lens = (t.cpu().numpy() for t in got)
    for a, (i, j, _) in enumerate(starts):
        d, cells = int(dist[j, i]), []
        while True:
            cells.append((i, j))
            if d == 0 or len(cells) == max_len:
                break
            for x, y in ((i + 1, j), (i - 1, j), (i, j + 1), (i, j - 1)):
                if 0 <= x < nx and 0 <= y < ny and dist[y, x] == d - 1:
                    i, j = x, y
                    break
            d -= 1
        assert lens[a] == len(cells) and np.array_equal(paths[a, :len(cells)], cells), a


@pytest.mark.parametrize("n", [4256, 4257, 20_001])
@pytest.mark.parametrize("plateaus", [False, True])
def test_paths_of_many_agents(R, n, plateaus):
    """Of 4256 agents (152 SMs) a CTA each, of more a thread: the paths that the agents
    have in calls of a few hundred, on distance fields and on others, with starts outside
    the map, on blocked cells and without such a goal among them."""
    rng = np.random.default_rng(n)
    ny, nx, max_len = 120, 170, 90
    occ = torch.from_numpy((rng.random((1, ny, nx)) < 0.2).astype(np.uint8)).cuda()
    dist = R.nav_fields(occ, [(5, 5), (100, 60), (169, 119)], 0, 0, 0)[1]
    if plateaus:
        dist = dist + torch.from_numpy(rng.integers(0, 2, (3, ny, nx)).astype(np.int32)).cuda()
    starts = np.stack([rng.integers(-1, nx + 1, n), rng.integers(-1, ny + 1, n), rng.integers(-1, 4, n)], 1)
    paths, lens = R.nav_paths(dist, starts, max_len)
    assert int(lens.max()) == max_len and int(lens.min()) == 0
    for k in range(0, n, n // 5):
        p1, l1 = R.nav_paths(dist, starts[k:k + 300], max_len)
        assert torch.equal(l1, lens[k:k + 300]) and torch.equal(p1, paths[k:k + 300]), k


@pytest.mark.parametrize("cell,nx,ny,nz", [(0.05, 90, 85, 31), (0.004, 1000, 900, 3), (0.5, 9, 7, 2), (0.03, 1, 40, 40)])
def test_slice_boxes_of_all_sizes(R, cell, nx, ny, nz):
    """Boxes from none or one cell to more than a warp takes at once (leaves of up to
    half a metre on 4 mm cells), and warps whose leaves lie on different planes."""
    from types import SimpleNamespace
    import oracle as O
    from scenegen import make_uniform_box_scene
    scene = make_uniform_box_scene(700, seed=9)
    big = np.flatnonzero(scene.child_count == 0)[::50]
    scene.log_scale[big] = np.log(np.float32(0.5)) - np.float32(0.3) * np.arange(3, dtype=np.float32)
    R.load_scene(scene)
    g = SimpleNamespace(x0=0.1, y0=0.05, cell=cell, nx=nx, ny=ny, z0=0.02, dz=0.09, nz=nz, threshold=0.3)
    got, occ = (t.cpu().numpy() for t in R.slice_occupancy(g))
    want, want_occ = O.slice_occupancy(scene, g)
    # within 1e-3, but for cells at the 1/255 cut-off on one side only
    exempt = (np.minimum(got, want) <= 1.0 / 255.0 + 1e-3) & (np.abs(got - want) > 1e-3)
    assert exempt.mean() < 0.01
    assert np.abs(got - want)[~exempt].max() <= 1e-3
    near = np.abs(want - g.threshold) <= 1e-3
    assert np.array_equal(occ[~near], want_occ[~near])
    assert (want > 0).any()


@pytest.fixture(scope="module")
def floor_views(small_floor):
    from scenegen import walk_cameras
    taus = np.random.default_rng(3).uniform(0.0, 40.0, 110)
    return walk_cameras(small_floor, 110, seed=8, width=320, height=240, taus=taus)


# record_capacity: 2^22 holds the masks of every call here, 2^16 those of four cameras of
# this scene (calls cut in slices), 2^12 none (single-pass kernels)
@pytest.mark.parametrize("records", [1 << 22, 1 << 16, 1 << 12])
def test_cuts_by_masks_equal_single_pass_cuts(small_floor, floor_views, records):
    from paper_2603_15186_gb300 import Renderer
    R = Renderer(cut_capacity=1 << 22, record_capacity=records, pair_capacity=1 << 20)
    R.load_scene(small_floor)
    cams = floor_views

    def lists(ids, off):
        off = off.cpu().numpy()
        return np.split(ids[:off[-1]].cpu().numpy(), off[1:-1])

    plain = [lists(*R.select_cut([c]))[0] for c in cams[:70]]
    for n in (4, 5, 8, 9, 16, 17, 32, 33, 70):
        got = lists(*R.select_cut(cams[:n]))
        assert len(got) == n and all(np.array_equal(a, b) for a, b in zip(got, plain)), n
    rng = np.random.default_rng(2)
    for frustum, guard in ((True, 0.0), (True, 24.0), (False, 0.0)):
        for sizes in ([1] * 40, [4], [3, 5], [7, 9, 1], [32, 1, 31], list(rng.integers(1, 20, 7))):
            n = int(sum(sizes))
            gb = [0] + list(np.cumsum(sizes))
            got = lists(*R.select_cut_shared(cams[:n], gb, frustum, guard))
            # a group of 33 sends the whole call to the single-pass kernel
            want = lists(*R.select_cut_shared(cams[:n + 33], gb + [n + 33], frustum, guard))[:-1]
            assert all(np.array_equal(a, b) for a, b in zip(got, want)), (frustum, guard, sizes)
            assert any(len(a) for a in got)
    R.close()


# this scene's masks take 0.6 MB an array, its words 10 KB a unit; records of 48 bytes.
# 2^16: all words and three arrays; 2^15: one array, several slices; 1: a buffer of the cut's own
@pytest.mark.parametrize("records", [1 << 16, 1 << 15, 1])
def test_cuts_in_slices_equal_cuts_at_once(small_floor, floor_views, records):
    from paper_2603_15186_gb300 import NgsError, Renderer
    pair = [Renderer(cut_capacity=1 << 22, record_capacity=k, pair_capacity=1 << 20) for k in (1 << 22, records)]
    for r in pair:
        r.load_scene(small_floor)
    rng = np.random.default_rng(6)

    def same(call):
        (ids, off), (ids1, off1) = (call(r) for r in pair)
        assert torch.equal(off, off1)
        assert torch.equal(ids[:int(off[-1])], ids1[:int(off[-1])]) and int(off[-1]) > 0

    for n in (4, 32, 33, 110):
        same(lambda r: r.select_cut(floor_views[:n]))
        with pytest.raises(NgsError):
            pair[1].select_cut(floor_views[:n], cap=100)
    for frustum in (True, False):
        for sizes in ([1] * 40, [20] * 5, list(rng.integers(1, 33, 6))):
            n = int(sum(sizes))
            gb = [0] + list(np.cumsum(sizes))
            same(lambda r: r.select_cut_shared((floor_views * 2)[:n], gb, frustum))
    for r in pair:
        r.close()


@pytest.fixture(scope="module")
def larger_floor():
    from scenegen import make_floor_scene, walk_cameras
    scene = make_floor_scene(600_000, seed=12, size=(14.0, 10.0, 3.0), n_clusters=8, cluster_size=4000)
    taus = np.random.default_rng(3).uniform(0.0, 40.0, 110)
    return scene, walk_cameras(scene, 110, seed=8, width=320, height=240, taus=taus)


# chunks of 8, 16 and 32 cameras, one and several; 2^13 records: slices in the cut's own buffer
@pytest.mark.parametrize("records", [1 << 22, 1 << 13])
def test_cuts_by_masks_of_a_larger_scene(larger_floor, records):
    """A scene of enough nodes for masks at any number of cameras: the lists of the
    single-pass kernels, which a group of 33 sends the whole call to."""
    from paper_2603_15186_gb300 import Renderer
    scene, cams = larger_floor
    R = Renderer(cut_capacity=1 << 22, record_capacity=records, pair_capacity=1 << 20)
    R.load_scene(scene)
    for frustum, guard in ((True, 0.0), (True, 24.0), (False, 0.0)):
        for sizes in ([1] * 4, [1] * 9, [1] * 16, [1] * 40, [3, 5], [3, 12, 1], [20, 30, 7], [32, 1, 31]):
            n = int(sum(sizes))
            gb = [0] + list(np.cumsum(sizes))
            ids, off = R.select_cut_shared(cams[:n], gb, frustum, guard)
            want, w_off = R.select_cut_shared(cams[:n + 33], gb + [n + 33], frustum, guard)
            assert torch.equal(off, w_off[:len(off)]) and int(off[-1]) > 0
            assert torch.equal(ids[:int(off[-1])], want[:int(off[-1])]), (frustum, guard, sizes)
            if not frustum and len(sizes) == n:
                plain, p_off = R.select_cut(cams[:n])
                assert torch.equal(p_off, off) and torch.equal(plain[:int(off[-1])], ids[:int(off[-1])])
            del ids, want
    R.close()


# one key into a second partition (4096 or 8192 keys), the keys that the histogram's
# CTAs take at once (2048) and one more, several rounds of all its CTAs
@pytest.mark.parametrize("key_bytes,n", [(4, 2048), (4, 2049), (4, 8193), (4, 311_297), (4, 6_000_001),
                                         (8, 2049), (8, 4097), (8, 700_001)])
def test_sort_histogram_sizes(R, key_bytes, n):
    g = torch.Generator(device="cuda").manual_seed(n)
    # few distinct high digits, as depths have
    keys = torch.randint(0, 1 << 27, (n,), generator=g, device="cuda", dtype=torch.int64)
    if key_bytes == 8:
        keys |= torch.randint(0, 3, (n,), generator=g, device="cuda", dtype=torch.int64) << 40
    else:
        keys = keys.to(torch.int32)
    vals = torch.arange(n, device="cuda", dtype=torch.int32)
    want, order = torch.sort(keys, stable=True)
    R.sort_pairs(keys, vals)
    torch.cuda.synchronize()
    assert torch.equal(keys, want) and torch.equal(vals, order.to(torch.int32))


# partitions of 256 elements up to 2^20, of 2048 beyond; chains of more partitions than CTAs
@pytest.mark.parametrize("n", [255, 256, 257, 8_193, 311_297, 1 << 20, (1 << 20) + 1, 4_000_001])
def test_scan_partition_sizes(R, n):
    x = torch.randint(0, 1000, (n,), device="cuda", dtype=torch.int32)
    out, total = R.scan_u32(x)
    torch.cuda.synchronize()
    want = torch.cumsum(x.to(torch.int64), 0)
    assert int(total) == int(want[-1]) & 0xffffffff or int(total) == int(want[-1])
    assert torch.equal(out.to(torch.int64) & 0xffffffff, (want - x) & 0xffffffff)


def test_scans_on_a_context_of_small_capacities():
    """A context of few records, without a scene, scans as many elements as any: its
    look-back words are sized for what it accepts (1024 partitions of 2048, or the 4096
    of 256 that 2^20 elements take)."""
    from paper_2603_15186_gb300 import NgsError, Renderer
    r = Renderer(cut_capacity=1 << 14, record_capacity=1 << 14, pair_capacity=1 << 14)
    for n in (1, 262_145, 524_289, 1 << 20, (1 << 20) + 1, 1 << 21):
        x = torch.randint(0, 1000, (n,), device="cuda", dtype=torch.int32)
        out, total = r.scan_u32(x)
        torch.cuda.synchronize()
        want = torch.cumsum(x.to(torch.int64), 0)
        assert int(total) == int(want[-1]) and torch.equal(out.to(torch.int64), want - x)
    x = torch.zeros((1 << 21) + 1, device="cuda", dtype=torch.int32)
    with pytest.raises(NgsError):
        r.scan_u32(x)
    r.close()


@pytest.mark.parametrize("dtype,tile", [("f32", 16), ("f16", 8)])
def test_tall_rects_next_to_small_ones(R, dtype, tile):
    """A view from among large Gaussians: rects of one to all of the tile rows in one
    warp, several hundred thousand pairs; pixels as on tiles of one row of rects."""
    from scenegen import look_camera, make_uniform_box_scene, quantize_attributes
    scene = make_uniform_box_scene(3000, seed=4)
    leaves = np.flatnonzero(scene.child_count == 0)
    scene.log_scale[leaves[::9]] += np.float32(2.0)
    cam = look_camera((2.0, 2.0, 1.2), 0.4, 640, 480, tau=0.0)
    stored = None if dtype == "f32" else quantize_attributes(scene, dtype)[0]
    R.load_scene(scene, attr_dtype=dtype, stored=stored)
    images = []
    for t in (tile, 32):
        R.set_tile(t, t)
        images.append(R.render([cam])[0].clone())
        ranges, pairs = R.tile_ranges(0, -(-640 // t) * -(-480 // t), 1 << 23)
        assert pairs == R.stats()["pair_total"] == int((ranges[:, 1] - ranges[:, 0]).sum())
    R.set_tile(16, 16)
    assert pairs > 20_000 and torch.equal(images[0], images[1])


def test_sort_key_widths_share_the_scratch():
    """64-bit keys after as many 32-bit keys (and the other way round): the context's
    scratch is large enough for either."""
    from paper_2603_15186_gb300 import Renderer
    r = Renderer(cut_capacity=1 << 20, record_capacity=1 << 22, pair_capacity=1 << 22)
    n = 3_000_000
    for dtype in (torch.int32, torch.int64, torch.int32):
        keys = torch.randint(0, 1 << 30, (n,), device="cuda", dtype=dtype)
        vals = torch.arange(n, device="cuda", dtype=torch.int32)
        want, order = torch.sort(keys, stable=True)
        r.sort_pairs(keys, vals)
        torch.cuda.synchronize()
        assert torch.equal(keys, want) and torch.equal(vals, order.to(torch.int32))
    r.close()


@pytest.mark.parametrize("mode", ["batched", "plain"])
def test_depths_beyond_the_short_keys(mode):
    """Three passes over 27 bits of depth while no mean can lie 13.1 km away, four over
    all bits otherwise: large Gaussians 20 and 30 km away are blended behind the near
    ones and in their order, and the near ones as without them."""
    import oracle as O
    from paper_2603_15186_gb300 import Renderer
    from scenegen import camera_c0, make_uniform_box_scene
    from scenegen.scene import build_hierarchy
    near = make_uniform_box_scene(600, seed=12)
    leaf = near.child_count == 0
    cam = camera_c0(0.0)
    r = Renderer(cut_capacity=1 << 20, record_capacity=1 << 20, pair_capacity=1 << 22)
    r.set_mode(mode)
    for far in (0, 2):
        pos = np.concatenate([near.pos[leaf], np.float32([[30_000, 2, 1.2], [20_000, 2, 1.2]])[:far]])
        quat = np.concatenate([near.quat[leaf], np.float32([[1, 0, 0, 0]] * far).reshape(far, 4)])
        logs = np.concatenate([near.log_scale[leaf], np.full((far, 3), np.log(4000.0), np.float32)])
        opac = np.concatenate([near.opacity[leaf], np.full(far, 0.8, np.float32)])
        sh = np.concatenate([near.sh[leaf], np.zeros((far, 16, 3), np.float32)])
        for k in range(far):
            sh[600 + k, 0, k] = 1.5          # red behind green
        scene = build_hierarchy(pos, quat, logs, opac, sh)
        r.load_scene(scene)
        got = r.render([cam])[0].cpu().numpy().astype(np.float64)
        ref = O.render(scene, cam)
        ok = ref.flags == 0
        assert ok.mean() > 0.5 and np.abs(got - ref.image)[:, ok].max() <= 2e-3
        if far:
            assert ref.image[1].mean() > ref.image[0].mean()
    r.close()


@pytest.mark.parametrize("per", [1, 3, 40])
def test_sub_batches_of_as_many_cameras_as_the_records_hold(small_floor, floor_views, per):
    """Record slots for so many cameras' whole cuts, which the partition tables are sized
    for too: the views come in sub-batches of at most that many, with the pixels of each alone."""
    from paper_2603_15186_gb300 import Renderer
    leaves = int((small_floor.child_count == 0).sum())
    r = Renderer(cut_capacity=1 << 20, record_capacity=per * leaves, pair_capacity=1 << 26)
    r.load_scene(small_floor)
    cams = floor_views[:50]
    images = [x.clone() for x in r.render(cams)]
    assert r.stats()["sub_batches"] >= -(-50 // per)   # the pairs' estimate may split them further
    r.set_mode("plain")
    for k in range(0, 50, 7):
        assert torch.equal(r.render([cams[k]])[0], images[k]), k
    r.close()


def test_views_that_reach_far_depths_and_others_share_a_graph():
    """Views along the axis of a Gaussian 30 km away (four passes over the depth) and across
    it (three would do), in turn: one capture each way at most, the pixels of the plain path."""
    from paper_2603_15186_gb300 import Renderer
    from scenegen import look_camera, make_uniform_box_scene
    from scenegen.scene import build_hierarchy
    near = make_uniform_box_scene(600, seed=12)
    leaf = near.child_count == 0
    scene = build_hierarchy(np.concatenate([near.pos[leaf], np.float32([[30_000, 2, 1.2]])]),
                            np.concatenate([near.quat[leaf], np.float32([[1, 0, 0, 0]])]),
                            np.concatenate([near.log_scale[leaf], np.full((1, 3), np.log(400.0), np.float32)]),
                            np.concatenate([near.opacity[leaf], np.full(1, 0.8, np.float32)]),
                            np.concatenate([near.sh[leaf], np.zeros((1, 16, 3), np.float32)]))
    r = Renderer(cut_capacity=1 << 20, record_capacity=1 << 20, pair_capacity=1 << 22)
    r.load_scene(scene)
    cams = [look_camera((2.0, 2.0, 1.2), a, 160, 120, tau=0.0) for a in (np.pi / 2, 0.0)]
    r.set_mode("plain")
    want = [r.render([c])[0].clone() for c in cams]
    r.set_mode("batched")
    replayed = []
    for k in (0, 0, 1, 0, 1, 0):
        assert torch.equal(r.render([cams[k]])[0], want[k])
        replayed.append(r.stats()["graph_replayed"])
    assert replayed == [0, 1, 0, 1, 1, 1]
    r.load_scene(near)
    r.render([cams[1]])
    r.render([cams[1]])
    assert r.stats()["graph_replayed"] == 1
    r.close()


# pairs: less than a partition of the last tile pass; partitions with one value of the
# tiles' low digit and with several; three passes over 76800 tiles
@pytest.mark.parametrize("leaves,grow,width,height", [(40, 0.0, 640, 480), (3000, 1.0, 640, 480),
                                                      (20_000, 1.5, 640, 480), (3000, 1.5, 2560, 1920)])
def test_tile_ranges_from_the_last_pass(leaves, grow, width, height):
    from paper_2603_15186_gb300 import Renderer
    from scenegen import look_camera, make_uniform_box_scene
    R = Renderer(cut_capacity=1 << 22, record_capacity=1 << 20, pair_capacity=1 << 27)
    scene = make_uniform_box_scene(leaves, seed=leaves)
    scene.log_scale[scene.child_count == 0] += np.float32(grow)
    R.load_scene(scene)
    cam = look_camera((2.0, 2.0, 1.2), 0.4, width, height, tau=0.0)
    images = []
    for t in (8, 32):
        R.set_tile(t, t)
        images.append(R.render([cam])[0].clone())
        ranges, pairs = R.tile_ranges(0, -(-width // t) * -(-height // t), 1 << 27)
        some = ranges[ranges[:, 1] > ranges[:, 0]]
        # the tiles' runs lie end to end in tile order
        assert some[0, 0] == 0 and some[-1, 1] == pairs == R.stats()["pair_total"]
        assert np.array_equal(some[1:, 0], some[:-1, 1])
    assert torch.equal(*images)
    R.close()


@pytest.mark.parametrize("n", [2, 16, 64, 70, 140, 290])
def test_camera_groups_of_all_sizes(R, n):
    """Cut + preprocess in groups of one to sixteen cameras of a node block (the fewer the
    cameras, the smaller): the pixels are those of each view alone."""
    from scenegen import look_camera, make_uniform_box_scene
    if not hasattr(R, "box120k"):
        R.box120k = make_uniform_box_scene(120_000, seed=4)
    R.load_scene(R.box120k)
    cams = [look_camera((1.0 + 2.0 * k / n, 2.0, 1.2), 0.37 * k, 64, 48, tau=4.0 + k % 5) for k in range(n)]
    images = [x.clone() for x in R.render(cams)]
    for k in range(0, n, max(1, n // 12)):
        assert torch.equal(R.render([cams[k]])[0], images[k]), k


@pytest.mark.parametrize("sizes", [[1] * 5, [1] * 16, [1] * 40, [2, 5], [3, 12, 1], [8] * 8, [20, 30, 7]])
def test_frustum_cuts_of_scattered_cameras(small_floor, sizes):
    """Cameras that look everywhere, so that none to all of a chunk's keep a word of
    nodes: the lists of the single-pass kernel."""
    from paper_2603_15186_gb300 import Renderer
    from scenegen import look_camera
    R = Renderer(cut_capacity=1 << 22, record_capacity=1 << 22, pair_capacity=1 << 20)
    R.load_scene(small_floor)
    rng = np.random.default_rng(sum(sizes))
    n = int(sum(sizes))
    cams = [look_camera((rng.uniform(0.5, 7.5), rng.uniform(0.5, 5.5), 1.2), rng.uniform(-3.1, 3.1), 320,
                        240, tau=float(rng.uniform(0.0, 30.0))) for _ in range(n + 33)]
    gb = [0] + list(np.cumsum(sizes))
    for guard in (0.0, 24.0):
        ids, off = (t.cpu().numpy() for t in R.select_cut_shared(cams[:n], gb, True, guard))
        # a group of 33 sends the whole call to the single-pass kernel
        want, w_off = (t.cpu().numpy() for t in R.select_cut_shared(cams, gb + [n + 33], True, guard))
        assert np.array_equal(off, w_off[:len(off)]) and np.array_equal(ids[:off[-1]], want[:off[-1]])
        assert off[-1] > 0
    R.close()
