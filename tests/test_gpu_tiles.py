"""The downsampling by occupied tiles against the oracle and against the sorted form: the same bits in the same order
(downsampling tile, cell, label).  Routes: the frame of max_range (marked before the counters are read), the frame
fitted to the hits (a max_range whose frame is too large), and the sorted form (a scratch without room for the tiles).
Scans: random clouds on both sides of the coordinate planes, one point, rays along the axes with coordinates too small
for the sums' unit (points of the gathered mean), hits next to the ground plane (noted fractions, and more of them than
the list holds), a cell of more than 2^15 members, all 32 classes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sb():
    import paper_1909_04631_gb300 as sbm
    sbm.load()
    return sbm


def _pose(x, y, z, yaw=0.0):
    T = np.eye(4)
    T[:2, :2] = [[np.cos(yaw), -np.sin(yaw)], [np.sin(yaw), np.cos(yaw)]]
    T[:3, 3] = (x, y, z)
    return T


def _scan(kind, rng):
    if kind == "one":
        return np.array([[3.2, -1.1, 0.4]], np.float32), _pose(0.1, 0.2, 0.3)
    if kind == "cloud":
        return rng.uniform(-9, 9, (3000, 3)).astype(np.float32), _pose(0.7, -0.4, 0.2, 0.3)
    if kind == "axes":  # directions whose other coordinates are rounding residues, from the origin
        a = np.repeat(np.arange(4) * (np.pi / 2), 40)
        r = rng.uniform(1, 20, len(a))
        p = np.stack([r * np.cos(a), r * np.sin(a), r * 1e-18], 1)
        q = rng.uniform(-8, 8, (200, 3))
        q[:, 2] = 3e-41
        return np.concatenate([p, q]).astype(np.float32), _pose(0, 0, 0)
    if kind in ("few", "many"):  # hits within the sums' unit of the ground plane: noted one by one, or too many for it
        p = rng.uniform(-8, 8, (900, 3))
        k = 40 if kind == "few" else 700
        p[:k, 2] = rng.uniform(-4e-8, 4e-8, k) - 1.5
        p[:k, 0] = np.where(np.arange(k) % 7 == 0, -0.25 + rng.uniform(-2e-8, 2e-8, k), p[:k, 0])
        return p.astype(np.float32), _pose(0.25, 0.1, 1.5)
    assert kind == "dense"  # members of the cells next to the sensor and along the rays: more than 2^15
    p = np.array([1.5, 0.7, -0.6]) + 0.03 * rng.random((40000, 3))
    return p.astype(np.float32), _pose(3.33, -2.2, 1.15)


def _order_key(xyz, lab, res):
    c = np.floor(xyz * np.float32(1 / res)).astype(np.int64)
    t, l = c >> 3, c & 7
    return list(zip(t[:, 0], t[:, 1], t[:, 2], l[:, 2], l[:, 1], l[:, 0], lab))


@pytest.mark.parametrize("kind", ["one", "cloud", "axes", "few", "many", "dense"])
@pytest.mark.parametrize("K", [1, 5, 31])
def test_routes_give_the_oracles_bits(sb, orc, kind, K):
    rng = np.random.default_rng(len(kind) * 100 + K)
    pts, T = _scan(kind, rng)
    lab = rng.integers(1, K + 1, len(pts)).astype(np.int32)
    sets = []
    for max_range, cap in ((50.0, 1 << 22), (400.0, 1 << 22), (50.0, None)):
        prm = dict(res=0.1, length_scale=0.3, sigma0=0.4, alpha0=0.001, free_step=0.3, num_classes=K,
                   max_range=max_range)
        ox, ol, st = orc.training_set(orc.params(**prm), pts, lab, T)
        if cap is None:  # just enough for the items: the directory does not fit
            cap = st["hits"] + st["free"]
        with sb.Map(sb.default_params(**prm, pool_blocks=1 << 12, sample_capacity=cap)) as m:
            gx, gl = m.training_set(pts, lab, T)
        assert len(gx) == st["train"]
        sets.append((gx, gl))
        if kind not in ("axes", "few", "many"):  # a centroid next to a cell's face can round onto it
            key = _order_key(gx, gl, 0.1)
            assert sum(a > b for a, b in zip(key, key[1:])) <= len(key) // 1000
        o, g = np.lexsort((ol, *ox.T)), np.lexsort((gl, *gx.T))
        np.testing.assert_array_equal(gl[g], ol[o])
        np.testing.assert_array_equal(gx[g], ox[o])
    for gx, gl in sets[1:]:
        np.testing.assert_array_equal(gx, sets[0][0])
        np.testing.assert_array_equal(gl, sets[0][1])


def test_errors_and_recovery(sb):
    """A label outside the range and a scan beyond the capacity are refused as before, and the map works after."""
    rng = np.random.default_rng(3)
    pts = rng.uniform(-9, 9, (500, 3)).astype(np.float32)
    lab = np.ones(500, np.int32)
    with sb.Map(sb.default_params(num_classes=3, pool_blocks=1 << 13, sample_capacity=1 << 15)) as m:
        bad = lab.copy()
        bad[77] = 4
        with pytest.raises(sb.SbkiError) as e:
            m.insert_scan(pts, bad, np.eye(4))
        assert e.value.status == sb.ERR_LABEL_RANGE
        far = np.tile(pts * 5, (12, 1))
        with pytest.raises(sb.SbkiError) as e:
            m.insert_scan(far, np.ones(len(far), np.int32), np.eye(4))
        assert e.value.status == sb.ERR_CAPACITY
        st = m.insert_scan(pts, lab, np.eye(4))
        assert st["hits"] == 500 and st["train_points"] > 0


def test_items_outside_the_frame_of_a_batch_are_refused(sb):
    """A pose whose 3x3 part scales by ten puts items outside the frame of max_range on every side: a batch says so
    (the error is set while CTAs of the same launch still start), no map changes, and the handle works after."""
    rng = np.random.default_rng(11)
    pts = rng.uniform(-9, 9, (3000, 3)).astype(np.float32)
    lab = np.ones(len(pts), np.int32)
    wide = np.eye(4)
    wide[:3, :3] *= 10
    with sb.Map(sb.default_params(num_classes=3, max_range=50.0, pool_blocks=1 << 15, sample_capacity=1 << 22)) as m:
        m.insert_batch([dict(points=pts, labels=lab, pose=np.eye(4), map_id=0)] * 2)
        before = m.export()
        with pytest.raises(sb.SbkiError) as e:
            m.insert_batch([dict(points=pts, labels=lab, pose=T, map_id=0) for T in (np.eye(4), wide)])
        assert e.value.status == sb.ERR_INVALID_ARG
        for a, b in zip(before[:2], m.export()[:2]):
            np.testing.assert_array_equal(a, b)
        st = m.insert_scan(pts, lab, np.eye(4))
        assert st["hits"] == len(pts)


def _affine(kind):
    T = _pose(0.4, -0.3, 0.2, 0.7)
    if kind == "scaled":
        T[:3, :3] *= 8
    elif kind == "sheared":
        T[:3, :3] = T[:3, :3] @ np.array([[5.0, 3.0, 0], [0, 6.0, -2.0], [0, 0, 7.0]])
    elif kind == "mirrored":
        T[:3, :3] = T[:3, :3] @ np.diag([-9.0, 1.0, 1.0])
    else:  # "far": one axis beyond 2^22 cells
        T = np.eye(4)
        T[0, 0] = 1e5
    return T


@pytest.mark.parametrize("kind", ["scaled", "sheared", "mirrored", "far"])
def test_poses_that_leave_the_frame_of_max_range(sb, orc, kind):
    """A pose is any affine transform: hits within max_range of the sensor may lie further off in the world.  The
    training set is the oracle's, whether the frame of max_range fits the directory (50 m) or not (400 m)."""
    rng = np.random.default_rng(len(kind))
    T = _affine(kind)
    if kind == "far":
        pts = np.array([[5.0, 0.7, -0.6]], np.float32)
    else:
        pts = rng.uniform(-9, 9, (1500, 3)).astype(np.float32)
    lab = rng.integers(1, 4, len(pts)).astype(np.int32)
    for max_range in (50.0, 400.0):
        prm = dict(res=0.1, length_scale=0.3, sigma0=0.4, alpha0=0.001, free_step=0.3, num_classes=3, max_range=max_range)
        ox, ol, st = orc.training_set(orc.params(**prm), pts, lab, T)
        with sb.Map(sb.default_params(**prm, pool_blocks=1 << 12, sample_capacity=1 << 22)) as m:
            gx, gl = m.training_set(pts, lab, T)
        assert len(gx) == st["train"]
        o, g = np.lexsort((ol, *ox.T)), np.lexsort((gl, *gx.T))
        np.testing.assert_array_equal(gl[g], ol[o])
        np.testing.assert_array_equal(gx[g], ox[o])


def test_a_scan_too_wide_for_the_keys_is_refused(sb):
    pts = np.array([[5.0, 5.0, 5.0]], np.float32)
    T = np.diag([1e5, 1e5, 1e5, 1.0])
    for max_range in (50.0, 400.0):
        with sb.Map(sb.default_params(num_classes=3, max_range=max_range, pool_blocks=1 << 12, sample_capacity=1 << 22)) as m:
            with pytest.raises(sb.SbkiError) as e:
                m.training_set(pts, np.ones(1, np.int32), T)
            assert e.value.status == sb.ERR_INVALID_ARG
            assert len(m.training_set(pts, np.ones(1, np.int32), np.eye(4))[0]) > 0


def test_batch_with_items_past_the_frame_but_within_the_keys(sb):
    """Tiles are counted up to the frame of max_range (131 per axis here), keys hold 256: a batch with items between
    the two is taken, as two updates would be."""
    rng = np.random.default_rng(5)
    prm = dict(num_classes=3, max_range=50.0, pool_blocks=1 << 16, sample_capacity=1 << 22, track_pairs=1)
    wide = np.diag([8.0, 8.0, 8.0, 1.0])
    scans = [dict(points=rng.uniform(1, 9, (300, 3)).astype(np.float32), labels=np.ones(300, np.int32), pose=T, map_id=0)
             for T in (wide, np.eye(4))]
    with sb.Map(sb.default_params(**prm)) as mb, sb.Map(sb.default_params(**prm)) as ms:
        mb.insert_batch(scans)
        for s in scans:
            ms.insert_scan(s["points"], s["labels"], s["pose"])
        (kb, ab, pb), (ks, as_, ps) = mb.export(pairs=True), ms.export(pairs=True)
    np.testing.assert_array_equal(kb, ks)
    np.testing.assert_array_equal(pb, ps)
    np.testing.assert_allclose(ab, as_, rtol=1e-5)  # sums in another order


def _beams(kind, rng):
    """Directions and ranges: lone beams all over a 60 m or 30 m scene, a dense fan of beams close by, or five."""
    n, r1 = {"lone60": (200, 59), "lone30": (4000, 29), "fan": (4000, 12), "few": (5, 49)}[kind]
    az, el = rng.uniform(0, 2 * np.pi, n), rng.uniform(-0.3, 0.3, n)
    if kind == "fan":
        az = np.linspace(0, 0.4, n)
    r = rng.uniform(5, r1, n)
    return np.stack([r * np.cos(el) * np.cos(az), r * np.cos(el) * np.sin(az), r * np.sin(el)], 1).astype(np.float32)


@pytest.mark.parametrize("kind,max_range,tiles", [("fan", 50.0, True), ("lone60", 60.0, False), ("lone30", 30.0, False),
                                                  ("few", 50.0, False)])
def test_sparse_scans_take_the_sorted_form(sb, orc, kind, max_range, tiles):
    """Scans with hardly more items than occupied tiles, or a few long beams: declined before or while their tiles are
    marked, and the oracle's training set either way, alone and in a batch."""
    rng = np.random.default_rng(17)
    pts = _beams(kind, rng)
    lab = rng.integers(1, 4, len(pts)).astype(np.int32)
    T = _pose(0.3, -1.75, 1.73)
    prm = dict(res=0.1, length_scale=0.3, sigma0=0.4, alpha0=0.001, free_step=0.3, num_classes=3, max_range=max_range)
    ox, ol, st = orc.training_set(orc.params(**prm), pts, lab, T)
    with sb.Map(sb.default_params(**prm, pool_blocks=1 << 12, sample_capacity=1 << 24)) as m:
        before = m.profile_read()["launches"]
        gx, gl = m.training_set(pts, lab, T)
        launches = m.profile_read()["launches"] - before
    o, g = np.lexsort((ol, *ox.T)), np.lexsort((gl, *gx.T))
    np.testing.assert_array_equal(gl[g], ol[o])
    np.testing.assert_array_equal(gx[g], ox[o])
    # begin, transform, clear, mark, then eight more; or offsets, emit, digit counts, a pass per byte of the key, three
    tile = np.floor(np.concatenate([pts @ T[:3, :3].T + T[:3, 3], T[None, :3, 3]]) / 0.1).astype(int) >> 3
    bits = sum(int(np.ceil(np.log2(e))) for e in tile.max(0) - tile.min(0) + 3) + 9 + 2
    assert launches == (12 if tiles else 4 + 3 + -(-bits // 8) + 3)
    with sb.Map(sb.default_params(**prm, pool_blocks=1 << 18, sample_capacity=1 << 24, sensor_model=1)) as m:
        s = m.insert_batch([dict(points=pts, labels=lab, pose=T, map_id=0)] * 2)
        assert s["train_points"] == 2 * st["train"]


def _crowd(n, at, rng):
    """n hits within 3 cm of `at`: one cell of them, and one of their free samples at each place along the beams."""
    return (np.asarray(at) + 0.03 * rng.random((n, 3))).astype(np.float32)


@pytest.mark.parametrize("kind", ["counts in their own word", "128-bit sums from a corner", "gathered"])
def test_crowded_cells(sb, orc, kind):
    """Branches that only a crowd of members reaches: more points than the counts that ride on the sums allow
    (2^19 / 18 at this free-sample spacing), 2^15 members and more in cells off the corner of a tile at a coordinate
    plane (both sides of it), and 2^18 of them, whose points are gathered."""
    rng = np.random.default_rng(23)
    step = 0.3
    if kind == "counts in their own word":
        pts, T, step = _crowd(30000, (0.3, 0.2, -0.15), rng), _pose(3.33, -2.2, 1.15), 0.01
    elif kind == "128-bit sums from a corner":
        pts, T = np.concatenate([_crowd(34000, (0.33, 0.53, 0.63), rng), _crowd(34000, (-0.37, -0.57, -0.27), rng)]), np.eye(4)
    else:
        pts, T = _crowd(270000, (0.33, 0.53, -0.27), rng), np.eye(4)
    lab = np.ones(len(pts), np.int32)
    prm = dict(res=0.1, length_scale=0.3, sigma0=0.4, alpha0=0.001, free_step=step, num_classes=2, max_range=50.0)
    ox, ol, st = orc.training_set(orc.params(**prm), pts, lab, T)
    with sb.Map(sb.default_params(**prm, pool_blocks=1 << 12, sample_capacity=1 << 22)) as m:
        gx, gl = m.training_set(pts, lab, T)
    o, g = np.lexsort((ol, *ox.T)), np.lexsort((gl, *gx.T))
    np.testing.assert_array_equal(gl[g], ol[o])
    np.testing.assert_array_equal(gx[g], ox[o])


def test_a_batch_without_room_for_its_tiles(sb):
    """Directories that fit and occupied tiles that do not (512 here): the recorded sorted form takes the batch, with
    the map of single updates on a handle with room."""
    rng = np.random.default_rng(29)
    prm = dict(num_classes=3, max_range=15.0, pool_blocks=1 << 15, track_pairs=1)
    scans = []
    for i in range(3):
        d = rng.normal(size=(150, 3))
        pts = (d / np.linalg.norm(d, axis=1)[:, None] * rng.uniform(4, 14.5, (150, 1))).astype(np.float32)
        scans.append(dict(points=pts, labels=rng.integers(1, 4, 150).astype(np.int32), pose=_pose(i, 0.3, -0.2, i), map_id=0))
    with sb.Map(sb.default_params(**prm, sample_capacity=1 << 17)) as mb, \
            sb.Map(sb.default_params(**prm, sample_capacity=1 << 22)) as ms:
        st = mb.insert_batch(scans)
        train = sum(ms.insert_scan(s["points"], s["labels"], s["pose"])["train_points"] for s in scans)
        (kb, ab, pb), (ks, as_, ps) = mb.export(pairs=True), ms.export(pairs=True)
    assert st["train_points"] == train
    np.testing.assert_array_equal(kb, ks)
    np.testing.assert_array_equal(pb, ps)
    np.testing.assert_allclose(ab, as_, rtol=1e-5)  # sums in another order


@pytest.mark.parametrize("order", ["along the rings", "shuffled"])
def test_beams_without_neighbours_decline_sooner(sb, orc, order):
    """A scan wide for its items: ordered beams (whose items meet in runs) take the tile form, the same beams shuffled
    the sorted one; the same bits."""
    rng = np.random.default_rng(31)
    az, el = np.meshgrid(np.arange(1500) * (2 * np.pi / 1500), np.deg2rad(np.linspace(-24, -4, 20)))
    r = np.minimum(1.73 / np.sin(-el.ravel()), 22.0)
    az, el = az.ravel(), el.ravel()
    pts = np.stack([r * np.cos(el) * np.cos(az), r * np.cos(el) * np.sin(az), r * np.sin(el)], 1).astype(np.float32)
    if order == "shuffled":
        pts = pts[rng.permutation(len(pts))]
    lab = np.ones(len(pts), np.int32)
    T = _pose(0.3, -1.75, 1.73)
    prm = dict(res=0.1, length_scale=0.3, sigma0=0.4, alpha0=0.001, free_step=0.1, num_classes=3, max_range=60.0)
    ox, ol, st = orc.training_set(orc.params(**prm), pts, lab, T)
    with sb.Map(sb.default_params(**prm, pool_blocks=1 << 12, sample_capacity=1 << 24)) as m:
        before = m.profile_read()["launches"]
        gx, gl = m.training_set(pts, lab, T)
        launches = m.profile_read()["launches"] - before
    assert (launches == 12) == (order != "shuffled")
    o, g = np.lexsort((ol, *ox.T)), np.lexsort((gl, *gx.T))
    np.testing.assert_array_equal(gl[g], ol[o])
    np.testing.assert_array_equal(gx[g], ox[o])
