"""The galaxy sum to the rounding of its terms: ragged mode groups, point blocks and chunks
against a plain FP64 sum, with a bar that a single missing point exceeds (asserted), and the
rms error of the terms themselves.

Bar of test_ragged: a term's rms rounding is below 1e-7 of its weight (twelve roundings of
2^-24 / sqrt 12), so |dA_n| <= 1e-6 sqrt(sum w^2) is ten standard deviations, and
|dP_l| <= c_l 1e-6 sqrt(sum w^2) <|A_0| + max_n |A_n|> / I over a shell's modes, c_l the sum of
the Legendre combination's absolute coefficients.

test_term_rounding: with |A_0|^2 off by 2 Re(A_0^* dA_0), a shell of n modes has P_0 off by
2 s / sqrt(n) of the raw monopole, s the terms' rms rounding.  A float cosine and sine (2.5e-8
rms) of a float angle in [-pi, pi) (4.1e-8) make s = 4.8e-8; 10 % are left for the sample.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
ys = pytest.importorskip("paper_1505_05341_gb300")

COEF = {0: 2.0, 2: 10.0, 4: 76.5, 6: 533.0}
SIDE, LO = 400.0, np.array([100.0, -50.0, 30.0])
KF = 2 * np.pi / SIDE


class Case:
    """Catalogue, modes and FP64 sums; drop leaves that many of the last points out of the sums."""

    def __init__(self, n, k_min, dk, nb, n_gal, n_ran, seed, unit=False):
        rng = np.random.default_rng(seed)
        self.n, self.k_min, self.dk, self.nb, self.n_gal = n, k_min, dk, nb, n_gal
        self.pos = (LO + SIDE * rng.random((n_gal + n_ran, 3))).astype(np.float32)
        self.w = np.ones(n_gal + n_ran, np.float32) if unit else rng.uniform(0.5, 2.0, n_gal + n_ran).astype(np.float32)
        self.nbar = np.full(n_gal + n_ran, 1e-3, np.float32)
        w, g = self.w.astype(np.float64), slice(0, n_gal)
        alpha = w[g].sum() / w[n_gal:].sum()
        self.sw = np.concatenate([w[g], -alpha * w[n_gal:]])
        self.norm = alpha * np.sum(w[n_gal:] ** 2 * self.nbar[n_gal:].astype(np.float64))
        self.shot = np.sum(w[g] ** 2) + alpha ** 2 * np.sum(w[n_gal:] ** 2)
        a = np.arange(-(n // 2), n // 2)
        m = np.stack(np.meshgrid(a, a, np.arange(n // 2 + 1), indexing="ij"), -1).reshape(-1, 3)
        n2 = (m ** 2).sum(1)
        km = KF * np.sqrt(n2.astype(np.float64))
        b = np.floor((km - k_min) / dk).astype(int)
        keep = (n2 > 0) & (n2 < (n // 2) ** 2) & (km >= k_min) & (b < nb)
        self.m, self.b = m[keep], b[keep]
        self.wt = np.where((self.m[:, 2] > 0) & (self.m[:, 2] < n // 2), 2.0, 1.0)
        self.count = np.bincount(self.b, self.wt, nb)

    def sums(self, ell, drop=0):
        x = self.pos.astype(np.float64)[:len(self.pos) - drop]
        sw = self.sw[:len(x)]
        rhat = x / np.linalg.norm(x, axis=1, keepdims=True)
        amp = {d: np.empty(len(self.m), complex) for d in range(0, ell + 1, 2)}
        for s in range(0, len(self.m), 2000):
            q = self.m[s:s + 2000]
            phase = np.exp(-1j * KF * (q @ (x - LO).T))
            mu = (q / np.linalg.norm(q, axis=1, keepdims=True)) @ rhat.T
            for d in amp:
                amp[d][s:s + 2000] = (phase * mu ** d) @ sw
        return amp

    def poles(self, ell, drop=0, amp=None):
        amp = amp or self.sums(ell, drop)
        has = self.count > 0
        mean = {d: np.bincount(self.b, self.wt * (amp[0] * amp[d].conj()).real, self.nb)[has] / self.count[has] for d in amp}
        out = {0: (mean[0] - self.shot) / self.norm}
        if ell >= 2:
            out[2] = 2.5 / self.norm * (3 * mean[2] - mean[0])
        if ell >= 4:
            out[4] = 1.125 / self.norm * (35 * mean[4] - 30 * mean[2] + 3 * mean[0])
        if ell >= 6:
            out[6] = 0.8125 / self.norm * (231 * mean[6] - 315 * mean[4] + 105 * mean[2] - 5 * mean[0])
        return out

    def bar(self, l, amp):
        has = self.count > 0
        size = np.abs(amp[0]) + np.max([np.abs(v) for v in amp.values()], axis=0)
        mean = np.bincount(self.b, self.wt * size, self.nb)[has] / self.count[has]
        return COEF[l] * 1e-6 * np.sqrt(np.sum(self.sw ** 2)) * mean / self.norm

    def gpu(self, ell):
        dev = lambda s: tuple(torch.from_numpy(np.ascontiguousarray(v[s])).cuda()  # noqa: E731
                              for v in (self.pos[:, 0], self.pos[:, 1], self.pos[:, 2], self.w, self.nbar))
        return ys.sum_gal(self.n, tuple(LO), SIDE, dev(slice(0, self.n_gal)), dev(slice(self.n_gal, None)), ell_max=ell,
                          k_min=self.k_min, dk=self.dk, n_bins=self.nb)


RAGGED = [(4, 0.0, 1, 1), (10, 0.02, 3, 6), (14, 0.031, 255, 2), (18, 0.05, 256, 1027)]


def ragged(n, k_min, n_gal, n_ran, ell):
    return Case(n, k_min, 0.013, 12, n_gal, n_ran, n + ell)


@pytest.mark.parametrize("ell", [0, 2, 4, 6])
@pytest.mark.parametrize("n,k_min,n_gal,n_ran", RAGGED)
def test_bar_notices_one_point(n, k_min, n_gal, n_ran, ell):
    c = ragged(n, k_min, n_gal, n_ran, ell)
    amp = c.sums(ell)
    ref, less = c.poles(ell, amp=amp), c.poles(ell, drop=1)
    for l in ref:
        assert np.all(np.abs(ref[l] - less[l]).max() > c.bar(l, amp).max()), l
        assert np.abs(ref[l] + (c.shot / c.norm if l == 0 else 0.0)).max() > c.bar(l, amp).max(), l


@pytest.mark.gpu
@pytest.mark.parametrize("ell", [0, 2, 4, 6])
@pytest.mark.parametrize("n,k_min,n_gal,n_ran", RAGGED)
def test_ragged(n, k_min, n_gal, n_ran, ell):
    c = ragged(n, k_min, n_gal, n_ran, ell)
    res, amp, has = c.gpu(ell), c.sums(ell), c.count > 0
    assert np.array_equal(res.n_modes, c.count)
    for l, want in c.poles(ell, amp=amp).items():
        assert np.all(np.abs(getattr(res, f"p{l}")[has] - want) <= c.bar(l, amp)), l


@pytest.mark.gpu
def test_term_rounding():
    q = []
    for seed in range(3):
        c = Case(40, 0.0, 0.5 * KF, 40, 1000, 4000, seed, unit=True)
        res, amp, has = c.gpu(0), c.sums(0), c.count > 0
        raw = np.bincount(c.b, c.wt * np.abs(amp[0]) ** 2, c.nb)[has] / c.count[has] / c.norm
        q.append((res.p0[has] - c.poles(0, amp=amp)[0]) / raw * np.sqrt(c.count[has]) / 2)
    rms = np.sqrt(np.mean(np.concatenate(q) ** 2))
    print("rms rounding of a term %.2e" % rms)
    assert rms <= 1.1 * 4.8e-8
