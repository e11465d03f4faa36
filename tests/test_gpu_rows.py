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


def _pairs_reference(prm, scale, xyz, lab, keys, G):
    """FP64 gradients of sum G alpha, and a bound on the FP32 evaluation's error for each: per pair, with e = 2^-24, the
    distance is within 4 e relative, u = 1 - d/l within 8 e, and the degree-10 (7) Horner form of the slope (kernel)
    within 20 e (14 e) of its coefficients' absolute sum, 45 (9); a sum of n terms adds n e of its terms' magnitudes."""
    e = 2.0 ** -24
    l, s0, res = prm["length_scale"], prm["sigma0"], prm["res"]
    c = (keys + 0.5) * res
    gx, bx = np.zeros((len(xyz), 3)), np.zeros(len(xyz))
    gl = gs = bl = bs = 0.0
    gk, bk = np.zeros(len(scale)), np.zeros(len(scale))
    for i, x in enumerate(xyz.astype(np.float64)):
        o = c - x
        d = np.sqrt((o[:, 0] ** 2 + o[:, 1] ** 2) + o[:, 2] ** 2)
        m = (o[:, 0] ** 2 + o[:, 1] ** 2) + o[:, 2] ** 2 < l * l
        o, d, g, s = o[m], d[m], G[m, lab[i]].astype(np.float64), scale[lab[i]]
        u = 1 - d / l
        f = (2 + np.cos(2 * np.pi * (1 - u))) * u / 3 + np.sin(2 * np.pi * (1 - u)) / (2 * np.pi)
        df = (2 - 2 * np.cos(2 * np.pi * u)) / 3 - 2 * np.pi * u * np.sin(2 * np.pi * u) / 3  # -f'(r)
        t = g * s0 * s * df / l
        n = len(d) + 40
        with np.errstate(all="ignore"):
            gx[i] = (t[:, None] * np.where(d[:, None] > 0, o / d[:, None], 0)).sum(0)
        bt = np.abs(g) * (u ** 4 * 900 * e + 4 * u ** 3 * 8 * e * 45 + 16 * e * np.abs(df))  # of g df
        bf = np.abs(g) * (u ** 5 * 126 * e + 5 * u ** 4 * 8 * e * 9 + 16 * e * np.abs(f))    # of g f
        bx[i] = s0 * s / l * (bt.sum() + n * e * np.abs(g * df).sum())
        gs += s * (g * f).sum()
        bs += s * (bf.sum() + n * e * np.abs(g * f).sum())
        gl += s0 * s / l ** 2 * (g * df * d).sum()
        bl += s0 * s / l ** 2 * l * (bt.sum() + n * e * np.abs(g * df).sum())
        gk[lab[i]] += s0 * (g * f).sum()
        bk[lab[i]] += s0 * (bf.sum() + n * e * np.abs(g * f).sum())
    return gl, gs, gx, gk, bl, bs, bx, bk


@pytest.mark.parametrize("lr,edge", [(0.6, 8), (0.87, 4), (1.5, 8), (2.5, 4), (3.0, 8), (3.0, 4), (3.45, 8), (3.6, 8)])
@pytest.mark.parametrize("n", [1, 15, 17, 300])
def test_backward_in_pairs(sb, lr, edge, n):
    import torch
    res, K = 0.1, 5
    rng = np.random.default_rng(int(100 * lr) + edge + n)
    xyz, lab = _cloud(rng, n, res, K + 1)
    scale = [1.0, 0.5, 2.0, 1.25, 0.75, 1.0]
    prm = dict(res=res, length_scale=lr * res, sigma0=0.4, alpha0=0.01, num_classes=K, block_edge=edge)
    with sb.Map(sb.default_params(**prm, sigma0_scale=scale, pool_blocks=1 << 13, sample_capacity=1 << 14)) as m:
        m.insert_training(xyz, lab)
        keys, _, _ = m.export()
        G = rng.normal(size=(len(keys), K + 1)).astype(np.float32)
        m.grad_clear()
        assert m.grad_add_alpha(keys, G) == 0
        xyzl = torch.from_numpy(np.concatenate([xyz, lab[:, None].astype(np.float32)], 1)).cuda()
        gl, gs, gx = m.backward(xyzl)
        gk = m.backward_scales(xyzl)
    rl, rs, rx, rk, bl, bs, bx, bk = _pairs_reference(prm, scale, xyz, lab, keys, G)
    assert (np.abs(gx.cpu().numpy() - rx) <= bx[:, None] + 1e-12).all()
    assert abs(gl - rl) <= bl + 1e-12 and abs(gs - rs) <= bs + 1e-12
    assert (np.abs(gk - rk) <= bk + 1e-12).all()


@pytest.mark.parametrize("lr,edge", [(0.87, 4), (0.87, 8), (2.0, 4), (3.0, 4), (3.0, 8), (3.5, 8)])
@pytest.mark.parametrize("n", [1, 33, 2500])
def test_touched_blocks_by_own_block(sb, lr, edge, n):
    """The touched set of the point-major form (27 neighbour bits per own block) is the block-major form's, which walks
    every point's candidate blocks: equal counts of touched and new blocks and equal blocks, over three updates."""
    res, K = 0.1, 5
    rng = np.random.default_rng(n + edge)
    B = edge * res
    prm = dict(res=res, length_scale=lr * res, sigma0=0.4, alpha0=0.001, num_classes=K, block_edge=edge,
               pool_blocks=1 << 13, sample_capacity=1 << 14)
    for assoc in (0, 1):
        with sb.Map(sb.default_params(**prm, association=assoc)) as m, \
                sb.Map(sb.default_params(**prm, association=assoc, accumulate_mode=1)) as b:
            for _ in range(3):
                xyz, lab = _cloud(rng, n, res, K + 1)
                xyz[::3] = (np.round(xyz[::3] / B) * B + rng.choice([-1, 0, 1], size=xyz[::3].shape)
                            * lr * res * rng.choice([0.5, 1.0, 2 ** -0.5], size=(len(xyz[::3]), 1))).astype(np.float32)
                sm, sbl = m.insert_training(xyz, lab), b.insert_training(xyz, lab)
                assert sm["touched_blocks"] == sbl["touched_blocks"] and sm["new_blocks"] == sbl["new_blocks"]
            km, kb = m.export()[0], b.export()[0]
            np.testing.assert_array_equal(km, kb)
