"""Read-off (Eq. mode, Eq. variance, Sec. V-C) at the edges of its kernel: class counts and point counts around a
warp's 32 rows, and voxels whose concentrations leave the range of the FP32-pair form (tiny, huge, below the prior,
non-finite) or whose occupancy lies on a threshold, against FP64 numpy.

Tolerance: a pair's quotient rounds like the exact one up to 2^-20 of a half ulp, so mean, variance and mode are within
one FP32 rounding (2^-24) of the FP64 value, plus the FP64 reference's own cancellation in S - alpha and S - (K+1)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
A0 = np.float32(0.001)


def _contents(rng, n, K1):
    a = (0.02 * rng.random((n, K1)) ** 3).astype(np.float32)
    a[np.arange(n), rng.integers(0, K1, n)] += (10.0 ** rng.uniform(-2, 4, n)).astype(np.float32)
    a[::5] += 1.5  # every class above one: the mode exists
    a[1::40, 0] = 1e-12 - A0   # alpha below the pairs' range
    a[2::40] *= np.float32(1e25)
    a[3::40, K1 - 1] = -0.5 * A0  # below the prior
    a[4::40] = 0.25  # ties: equal classes
    a[5::40, 0] = np.nan
    a[6::40, K1 - 1] = np.inf
    a[7::40] = 0.0   # no mass
    a[8::40] = 0.0
    a[8::40, 0] = a[8::40, 1] = 3.0
    return a + A0


def _reference(alpha, inc, lo, hi):
    a = alpha.astype(np.float64)
    K1 = a.shape[1]
    with np.errstate(all="ignore"):
        S = a.sum(1, keepdims=True)
        mean, var = a / S, a * (S - a) / (S * S * (S + 1))
        mode = np.where((a > 1).all(1, keepdims=True), (a - 1) / (S - K1), np.nan)
        po = (a[:, 1:] / S).sum(1)
        mass = inc.astype(np.float64).sum(1)
    state = np.where(mass > 0, np.where(po < lo, 0, np.where(po > hi, 2, 1)), 1)
    slack = np.where(np.isfinite(S) & (S > a), 8e-16 * K1 * np.abs(S) / np.maximum(np.abs(S - a), 1e-300), 0)
    return S, mean, var, mode, po, state, slack


@pytest.mark.parametrize("K1,n", [(2, 1), (2, 33), (3, 31), (20, 32), (20, 1000), (31, 257), (32, 64), (32, 4097)])
def test_readoff_against_fp64(K1, n):
    import torch
    import paper_1909_04631_gb300 as sb
    rng = np.random.default_rng(K1 * 10007 + n)
    alpha = _contents(rng, n, K1)
    keys = np.stack([np.arange(n) % 37 - 18, np.arange(n) // 37 - 20, np.arange(n) % 3 - 1], 1).astype(np.int64)
    lo, hi = 0.5, 0.6  # K1 = 2 with equal classes sits exactly on the lower threshold
    m = sb.Map(num_classes=K1 - 1, pool_blocks=1 << 13, sample_capacity=1 << 12, free_thresh=lo, occ_thresh=hi)
    m.import_(keys, alpha)
    inc = alpha - A0  # one FP32 subtraction, as the import does
    pts = torch.from_numpy(((keys + 0.5) * 0.1).astype(np.float32)).cuda()
    out = dict(probs=torch.full((n, K1), -1.0, device="cuda"), var=torch.full((n, K1), -1.0, device="cuda"),
               mode=torch.full((n, K1), -1.0, device="cuda"), p_occ=torch.full((n,), -1.0, device="cuda"),
               label=torch.full((n,), -1, device="cuda", dtype=torch.int32),
               state=torch.full((n,), -1, device="cuda", dtype=torch.int32))
    m.query_device(pts, **out)
    g = {k: v.cpu().numpy() for k, v in out.items()}
    held = A0 + inc
    S, mean, var, mode, po, state, slack = _reference(held, inc, lo, hi)
    tol = 2.0 ** -24 * (1 + 2.0 ** -10)
    fine = np.isfinite(held).all(1)
    assert np.array_equal(np.isnan(g["probs"]), np.isnan(mean.astype(np.float32)))
    tiny = 2.0 ** -149
    for name, ref, sl in (("probs", mean, 0.0), ("var", var, slack)):
        r = ref[fine]
        assert (np.abs(g[name][fine] - r) <= (tol + (sl[fine] if np.ndim(sl) else sl)) * np.abs(r) + tiny).all(), name
    has = fine & (held > 1).all(1)
    assert np.array_equal(np.isnan(g["mode"][fine]), ~np.repeat(has[fine, None], K1, 1))
    cancel = 8e-16 * K1 * S[has] / np.maximum(S[has] - K1, 1e-300)
    assert (np.abs(g["mode"][has] - mode[has]) <= (tol + cancel) * np.abs(mode[has]) + tiny).all()
    assert (np.abs(g["p_occ"][fine] - po[fine]) <= tol * np.abs(po[fine]) + tiny).all()
    assert np.array_equal(g["label"][fine], held[fine].argmax(1))
    assert np.array_equal(g["state"][fine], state[fine])
    m.close()
