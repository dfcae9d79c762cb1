"""The line transforms whose last radix is left to the reader (E2 = 2: 384, 512; E2 = 4: 768,
1024) at every l_max, on shells from the lowest modes to just below the Nyquist frequency,
with the observer away from the nodes and on an occupied one.

Particles sit on nodes (NGP, no window), where the mesh estimate is the galaxy sum; the sum is
taken in FP64 over the modes of a few narrow shells (oracle.direct's point sums over the modes
enumerated here).  Tolerance: |dP_l| <= c_l e P_raw with e = 2.5e-6, the relative rounding of a
mode after three float32 transforms of up to 30 butterfly levels at 2^-24 each with head-room
of 1.4, and c_l the sum of the Legendre combination's absolute coefficients.
"""
import numpy as np
import pytest

from oracle.binning import BinSpec
from oracle.direct import _finish, _point_sums
from oracle.normalization import catalog_sums
from synth.catalogs import Catalog, Geometry

torch = pytest.importorskip("torch")
ys = pytest.importorskip("paper_1505_05341_gb300")

COEF = {0: 2.0, 2: 10.0, 4: 76.5, 6: 533.0}


def shell_modes(n, box_len, bins):
    """Half-grid modes of the shells: m, shell, Hermitian weight, |k|."""
    kf = 2 * np.pi / box_len
    hi = min(n // 2, int((bins.k_min + bins.dk * bins.n_bins) / kf) + 1)
    my, mz = np.arange(-hi, hi + 1)[:, None], np.arange(0, hi + 1)[None, :]
    out = []
    for mx in range(-hi, hi + 1):
        n2 = mx * mx + my * my + mz * mz
        k = kf * np.sqrt(n2.astype(np.float64))
        b = np.floor((k - bins.k_min) / bins.dk)
        iy, iz = np.nonzero((n2 > 0) & (n2 < (n // 2) ** 2) & (b >= 0) & (b < bins.n_bins))
        out.append(np.stack([np.full(iy.size, mx), iy - hi, iz, b[iy, iz]], 1).astype(np.int64))
    m = np.concatenate(out)
    w = np.where((m[:, 2] > 0) & (m[:, 2] < n // 2), 2.0, 1.0)
    return m[:, :3], m[:, 3], w, kf * np.sqrt((m[:, :3] ** 2).sum(1).astype(np.float64))


def test_shell_modes_are_the_oracles():
    from oracle.direct import _valid_modes
    b = BinSpec(0.05, 0.02, 3)
    m, s, w, k = shell_modes(20, 300.0, b)
    M, bidx, wo, kmag, _ = _valid_modes(20, 300.0, b)
    rows = lambda *a: sorted(zip(*(np.asarray(v, float).tolist() for v in a)))  # noqa: E731
    assert rows(m[:, 0], m[:, 1], m[:, 2], s, w) == rows(M[:, 0], M[:, 1], M[:, 2], bidx, wo)


def catalogue(n, at_node, seed):
    rng = np.random.default_rng(seed)
    lo = np.array([-0.5 * n, -0.25 * n, 0.125 * n])  # H = 1: every node is exact in float32

    def cat(m, heavy):
        p = rng.integers(0, n, (m, 3)) + lo
        w = rng.uniform(0.5, 1.5, m).astype(np.float32)
        if heavy:
            p[0], w[0] = (3.0, -7.0, 0.125 * n + 5.0), 12.0
        return Catalog(*(np.ascontiguousarray(p[:, i], dtype=np.float32) for i in range(3)), w, np.full(m, m / n ** 3, np.float32))

    observer = (3.0, -7.0, 0.125 * n + 5.0) if at_node else (3.3, -7.6, 0.125 * n + 5.2)
    return cat(120, True), cat(400, False), Geometry(tuple(lo), float(n), observer)


@pytest.mark.gpu
@pytest.mark.parametrize("n,ell,at_node", [
    (384, 0, False), (384, 2, True), (384, 4, False), (384, 6, True),
    (512, 0, False), (512, 2, False), (512, 4, True), (512, 6, False), (512, 6, True),
    (768, 0, False), (768, 2, True), (768, 4, False),
    (1024, 0, False), (1024, 2, False), (1024, 4, True),
])
def test_large_lines(n, ell, at_node):
    gal, ran, geo = catalogue(n, at_node, n + ell)
    kf = 2 * np.pi / geo.box_len
    norm = catalog_sums(gal, ran)
    pos = np.concatenate([gal.positions(), ran.positions()]).astype(np.float64)
    wts = np.concatenate([gal.w.astype(np.float64), -norm.alpha * ran.w.astype(np.float64)])
    dev = lambda c: tuple(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (c.x, c.y, c.z, c.w, c.nbar))  # noqa: E731
    dgal, dran = dev(gal), dev(ran)
    for k_min, dk, nb in ((0.0, 3.0, 3), (0.13 * n, 0.08, 1), (0.26 * n, 0.03, 1), (0.49 * n, 0.01, 1)):
        b = BinSpec(k_min * kf, dk * kf, nb)
        m, s, w, k = shell_modes(n, geo.box_len, b)
        assert 50 < len(m) < 40_000
        amps = _point_sums(pos - np.array(geo.box_min), wts, pos - np.array(geo.observer), m * kf, ell, False)
        for d in (2, 4):
            amps.setdefault(d, np.zeros(len(m), complex))
        ref = _finish(amps, s, w, k, b, norm, False, max(ell, 4))
        with ys.Plan(n, geo.box_min, geo.box_len, geo.observer, assign="ngp", compensate=False, ell_max=ell, k_min=b.k_min,
                     dk=b.dk, n_bins=b.n_bins, stream=torch.cuda.current_stream().cuda_stream) as plan:
            plan.assign(dgal, dran)
            res = plan.measure()
        assert np.array_equal(res.n_modes, ref.n_modes)
        raw = ref.sum0 / ref.n_modes / ref.norm.I
        for l in range(0, ell + 1, 2):
            err = np.abs(getattr(res, f"p{l}") - getattr(ref, f"p{l}")) / raw
            print(n, ell, k_min / n, l, err / COEF[l])
            assert np.all(err <= COEF[l] * 2.5e-6), (l, k_min, err.max() / COEF[l])
