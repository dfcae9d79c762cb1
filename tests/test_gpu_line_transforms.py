"""The y,z stage's line transforms and source fields against the FP64 oracle: every
radix split (N = 16 R2 E2 or 12 R2 E2), every l_max, and observers where the source
fields' scaling matters (on a node, just off one, next to a mesh plane, far away; boxes
in very small and very large units).

Tolerance: |P_l^gpu - P_l^oracle| <= c_l e P_raw in every shell, with P_raw the monopole
before shot-noise subtraction, e = 2e-6 (the relative rounding of a mode after three
float32 transforms of up to 3 log2 N = 24 butterfly levels at 2^-24 each, with head-room
of about 1.4) and c_l the sum of the absolute coefficients of the Legendre combination:
1 + 1 (shot noise), 2.5 (3 + 1), 9/8 (35 + 30 + 3), 13/16 (231 + 315 + 105 + 5).
"""
import numpy as np
import pytest

import oracle
import synth
from oracle.binning import BinSpec

torch = pytest.importorskip("torch")
ys = pytest.importorskip("paper_1505_05341_gb300")

pytestmark = pytest.mark.gpu

E = 2e-6
COEF = {0: 2.0, 2: 10.0, 4: 76.5, 6: 533.0}


def check(n, ell, kind, interlace, side, center, observer, seed):
    gal, ran, geo = synth.poisson_cube(3000, 15000, side=side, center=center, seed=seed)
    geo = type(geo)(geo.box_min, geo.box_len, tuple(observer))
    kf = 2 * np.pi / side
    bins = BinSpec(0.0, 2.0 * kf, n // 4)
    ref = oracle.fft_multipoles(gal, ran, geo, n, bins, assign=kind, interlace=interlace, ell_max=ell)
    dev = lambda c: tuple(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (c.x, c.y, c.z, c.w, c.nbar))  # noqa: E731
    with ys.Plan(n, geo.box_min, geo.box_len, geo.observer, assign=kind, interlace=interlace, ell_max=ell,
                 dk=bins.dk, n_bins=bins.n_bins, stream=torch.cuda.current_stream().cuda_stream) as plan:
        plan.assign(dev(gal), dev(ran))
        res = plan.measure()
    assert np.array_equal(res.n_modes, ref.n_modes)
    has = ref.n_modes > 0
    raw = ref.sum0[has] / ref.n_modes[has] / ref.norm.I
    for l in range(0, ell + 1, 2):
        err = np.abs(getattr(res, f"p{l}")[has] - getattr(ref, f"p{l}")[has]) / raw
        assert np.all(err <= COEF[l] * E), (l, err.max() / COEF[l])


@pytest.mark.parametrize("ell", [0, 2, 4, 6])
@pytest.mark.parametrize("n", [16, 32, 64, 96, 128, 192, 256])
def test_radix_splits(n, ell):
    check(n, ell, "cic", n == 96, 400.0, (300.0, -120.0, 45.0), (0.0, 0.0, 0.0), n + ell)


@pytest.mark.parametrize("ell", [4, 6])
@pytest.mark.parametrize("side,center,offset", [
    (320.0, (0.0, 0.0, 0.0), (0.0, 0.0, 0.0)),          # on a node of mesh 1
    (320.0, (0.0, 0.0, 0.0), (5.0, 5.0, 5.0)),          # on a node of mesh 2
    (320.0, (0.0, 0.0, 0.0), (1e-3, -2e-3, 5e-4)),      # 1e-4 cells off a node
    (320.0, (0.0, 0.0, 0.0), (1e-9, 37.0, -81.0)),      # next to a mesh plane
    (320.0, (0.0, 0.0, 0.0), (0.0, 0.0, 33.3)),         # on a row of nodes
    (320.0, (0.0, 0.0, 0.0), (1e7, 2e7, -3e7)),         # far away
    (0.7, (0.1, 0.2, 0.3), (0.0, 0.0, 0.0)),            # rounding decides whether a node is hit
    (1e-5, (0.0, 0.0, 0.0), (1e-6, 0.0, 0.0)),          # tiny units
    (3e8, (1e8, 0.0, 0.0), (0.0, 0.0, 0.0)),            # huge units
])
def test_observers_and_units(side, center, offset, ell):
    check(32, ell, "tsc", True, side, center, [c + o for c, o in zip(center, offset)] if side != 3e8 else offset, 5)
