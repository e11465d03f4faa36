"""The accumulation by rows at its edges, against the FP64 oracle: supports from just above half the voxel diagonal
to six voxels (one and several rounds of columns, both row shapes, windows of two to four quads), both block edges,
points on voxel centres, faces and corners (pairs at exactly d = l are re-decided in FP64), several maps of a handle,
and every form of the kernel.  Keys and pair counts exact, alpha within relative 1e-5: the bound that the repository
holds the FP32 sums to."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sb():
    import paper_1909_04631_gb300 as sbm
    sbm.load()
    return sbm


def _cloud(rng, n, res, K1):
    x = rng.uniform(-1.7, 1.7, size=(n, 3))
    x[::4] = (np.round(x[::4] / res) + 0.5) * res        # voxel centres
    x[1::4] = np.round(x[1::4] / res) * res              # voxel corners
    x[2::8] += rng.choice([-80.0, 35.0], size=(len(x[2::8]), 1))  # far from the origin, either sign
    return x.astype(np.float32), rng.integers(0, K1, size=n).astype(np.int32)


def _check(m, om, tracked):
    keys, alpha, pairs = m.export(pairs=tracked)
    okeys, oalpha, opairs = om.export()
    np.testing.assert_array_equal(keys, okeys)
    if tracked:
        np.testing.assert_array_equal(pairs, opairs)
    assert (np.abs(alpha.astype(np.float64) - oalpha) / oalpha).max(initial=0.0) <= 1e-5
    return int(opairs.sum())


@pytest.mark.parametrize("lr,edge", [(0.87, 8), (0.87, 4), (1.0, 4), (1.5, 8), (2.0, 4), (2.5, 8), (3.0, 8), (3.0, 4),
                                     (3.45, 8), (3.5, 8), (4.0, 8), (5.25, 8), (6.0, 8)])
@pytest.mark.parametrize("n", [1, 7, 9, 333])
def test_supports_and_edges(sb, orc, lr, edge, n):
    res, K = 0.1, 5
    rng = np.random.default_rng(int(100 * lr) + edge + n)
    xyz, lab = _cloud(rng, n, res, K + 1)
    prm = dict(res=res, length_scale=lr * res, sigma0=0.4, alpha0=0.001, num_classes=K, block_edge=edge)
    for assoc in (0, 1):
        om = orc.OracleMap(orc.params(**prm, association=assoc))
        om.insert_training(xyz, lab)
        for tracked in (0, 1):
            with sb.Map(sb.default_params(**prm, association=assoc, track_pairs=tracked, pool_blocks=1 << 13,
                                          sample_capacity=1 << 14)) as m:
                st = m.insert_training(xyz, lab)
                assert st["pairs"] == _check(m, om, bool(tracked))


@pytest.mark.parametrize("scales", [(1.0, 0.5, 1.15, 0.3, 1.0), (1.9, 0.3, 1.0, 0.45, 1.3)], ids=["narrow", "wide"])
def test_class_supports(sb, orc, scales):
    res, K = 0.1, 4
    rng = np.random.default_rng(7)
    xyz, lab = _cloud(rng, 500, res, K + 1)
    prm = dict(res=res, length_scale=0.3, sigma0=0.4, alpha0=0.001, num_classes=K, l_scale=list(scales))
    om = orc.OracleMap(orc.params(**prm))
    om.insert_training(xyz, lab)
    for tracked in (0, 1):
        with sb.Map(sb.default_params(**prm, track_pairs=tracked, pool_blocks=1 << 13, sample_capacity=1 << 14)) as m:
            st = m.insert_training(xyz, lab)
            assert st["pairs"] == _check(m, om, bool(tracked))


@pytest.mark.parametrize("lr", [2.5, 3.0, 4.5])
def test_soft_labels(sb, orc, lr):
    res, K = 0.1, 6
    rng = np.random.default_rng(int(10 * lr))
    pts = rng.uniform(-2.0, 2.0, size=(400, 3)).astype(np.float32)
    probs = rng.dirichlet(np.full(K, 0.3), size=400).astype(np.float32)
    probs[::3] = np.eye(K, dtype=np.float32)[rng.integers(0, K, len(probs[::3]))]
    pose = np.eye(4)
    pose[:3, 3] = (0.31, -0.2, 0.15)
    prm = dict(res=res, length_scale=lr * res, sigma0=0.4, alpha0=0.001, num_classes=K, max_range=50.0)
    om = orc.OracleMap(orc.params(**prm))
    om.insert_scan_soft(pts, probs, pose)
    with sb.Map(sb.default_params(**prm, track_pairs=1, pool_blocks=1 << 13, sample_capacity=1 << 16)) as m:
        st = m.insert_scan_soft(pts, probs, pose)
        assert st["pairs"] == _check(m, om, True)
