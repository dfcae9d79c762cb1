"""The galaxy sum's mode groups and point blocks where they are ragged: shells that cut the
m_z columns into short or split runs, one to a few points, point counts around the block
and chunk sizes, and every l_max, against a plain FP64 sum over the same modes.

Tolerance on A_n's shell means: every term carries a float32 phase factor, product and
weight, a relative error of at most 12 roundings of 2^-24 (7e-7) of its |w|, so
|dP_l| <= c_l 2 (7e-7) (sum |w|)^2 / I for the shell mean of Re A_0 A_n^* (|A_0|, |A_n| <=
sum |w|), c_l the sum of the Legendre combination's absolute coefficients.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
ys = pytest.importorskip("paper_1505_05341_gb300")

pytestmark = pytest.mark.gpu

COEF = {0: 2.0, 2: 10.0, 4: 76.5, 6: 533.0}


@pytest.mark.parametrize("ell", [0, 2, 4, 6])
@pytest.mark.parametrize("n,k_min,n_gal,n_ran", [(4, 0.0, 1, 1), (10, 0.02, 3, 6), (14, 0.031, 255, 2), (18, 0.05, 256, 1027)])
def test_ragged(n, k_min, n_gal, n_ran, ell):
    side, lo = 400.0, np.array([100.0, -50.0, 30.0])
    rng = np.random.default_rng(n + ell)
    pos = (lo + side * rng.random((n_gal + n_ran, 3))).astype(np.float32)
    w = rng.uniform(0.5, 2.0, n_gal + n_ran).astype(np.float32)
    nbar = np.full(n_gal + n_ran, 1e-3, np.float32)
    cat = lambda a, b: tuple(torch.from_numpy(np.ascontiguousarray(v[a:b])).cuda()  # noqa: E731
                             for v in (pos[:, 0], pos[:, 1], pos[:, 2], w, nbar))
    dk, kf = 0.013, 2 * np.pi / side
    res = ys.sum_gal(n, tuple(lo), side, cat(0, n_gal), cat(n_gal, n_gal + n_ran), ell_max=ell, k_min=k_min, dk=dk, n_bins=12)
    x, w64 = pos.astype(np.float64), w.astype(np.float64)
    alpha = w64[:n_gal].sum() / w64[n_gal:].sum()
    sw = np.concatenate([w64[:n_gal], -alpha * w64[n_gal:]])
    norm = alpha * np.sum(w64[n_gal:] ** 2 * nbar[n_gal:].astype(np.float64))
    shot = np.sum(w64[:n_gal] ** 2) + alpha ** 2 * np.sum(w64[n_gal:] ** 2)
    rhat = x / np.linalg.norm(x, axis=1, keepdims=True)
    m = np.array([(a, b, c) for a in range(-n // 2, n // 2) for b in range(-n // 2, n // 2) for c in range(n // 2 + 1)
                  if 0 < a * a + b * b + c * c < (n // 2) ** 2])
    km = kf * np.sqrt((m ** 2).sum(1).astype(np.float64))
    b = np.floor((km - k_min) / dk).astype(int)
    keep = (km >= k_min) & (b < 12)
    m, b = m[keep], b[keep]
    weight = np.where((m[:, 2] > 0) & (m[:, 2] < n // 2), 2.0, 1.0)
    count = np.bincount(b, weight, 12)
    assert np.array_equal(res.n_modes, count)
    has = count > 0
    phase = np.exp(-1j * kf * (m @ (x - lo).T))
    mu = (m / np.linalg.norm(m, axis=1, keepdims=True)) @ rhat.T
    amp = {d: (phase * mu ** d) @ sw for d in range(0, ell + 1, 2)}
    mean = {d: np.bincount(b, weight * (amp[0] * amp[d].conj()).real, 12)[has] / count[has] for d in amp}
    ref = {0: (mean[0] - shot) / norm}
    if ell >= 2:
        ref[2] = 2.5 / norm * (3 * mean[2] - mean[0])
    if ell >= 4:
        ref[4] = 1.125 / norm * (35 * mean[4] - 30 * mean[2] + 3 * mean[0])
    if ell >= 6:
        ref[6] = 0.8125 / norm * (231 * mean[6] - 315 * mean[4] + 105 * mean[2] - 5 * mean[0])
    for l, want in ref.items():
        tol = COEF[l] * 2 * 7e-7 * np.abs(sw).sum() ** 2 / norm
        assert np.max(np.abs(getattr(res, f"p{l}")[has] - want), initial=0.0) <= tol, l
