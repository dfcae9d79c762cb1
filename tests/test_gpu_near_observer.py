"""Only a node at r = 0 goes without a line-of-sight weight: with a heavy particle on the
node next to the observer, however near, its direction counts.

Particles sit on nodes (NGP), the heavy one on the node at the origin, the observer a given
vector away from it; the multipoles are compared with the FP64 oracle's galaxy sum, which
equals the mesh estimate there.  Tolerance: that of the line-transform tests, c_l e P_raw
with e = 2e-6 and c_l the sum of the Legendre combination's absolute coefficients.  Dropping
the heavy node's direction moves P_2 by O(P_raw) (asserted on the oracle itself).
"""
import numpy as np
import pytest

import oracle
from oracle.binning import BinSpec
from synth.catalogs import Catalog, Geometry

torch = pytest.importorskip("torch")
ys = pytest.importorskip("paper_1505_05341_gb300")

COEF = {0: 2.0, 2: 10.0, 4: 76.5, 6: 533.0}
SIDE = 384.0  # whole node positions for every mesh below


def case(n, observer, seed):
    """Particles on the nodes of an n^3 mesh with a node at the origin, one of weight 60 there."""
    rng = np.random.default_rng(seed)
    h = SIDE / n

    def cat(m, first=None):
        p = (rng.integers(0, n, (m, 3)) - n // 2) * h
        w = rng.uniform(0.5, 1.5, m).astype(np.float32)
        if first:
            p[0], w[0] = 0.0, first
        return Catalog(*(p[:, i].astype(np.float32) for i in range(3)), w, np.full(m, m / SIDE ** 3, np.float32))

    return cat(200, 60.0), cat(600), Geometry((-SIDE / 2,) * 3, SIDE, tuple(observer))


OFFSETS = [(0.0, 0.0, 0.0), (1e-8, -2e-8, 5e-9), (0.0, 3e-9, 0.0), (-4e-13, 0.0, 1e-13), (0.0, 0.0, 2e-17), (1e-18, 1e-18, -1e-18)]


def bins(n):
    return BinSpec(0.0, 4 * np.pi / SIDE, 4)


def test_the_heavy_node_counts():
    gal, ran, geo = case(32, OFFSETS[1], 1)
    near, far = (oracle.sum_gal(gal, ran, Geometry(geo.box_min, geo.box_len, o), 16, bins(16)) for o in (OFFSETS[1], OFFSETS[0]))
    raw = near.sum0 / near.n_modes / near.norm.I
    assert np.all(np.abs(near.p2 - far.p2)[near.n_modes > 0] > 1e-2 * raw[near.n_modes > 0])


@pytest.mark.gpu
@pytest.mark.parametrize("n,ell", [(16, 2), (32, 4), (32, 6), (96, 4), (128, 6)])
@pytest.mark.parametrize("observer", OFFSETS)
def test_directions_next_to_the_observer(n, ell, observer):
    gal, ran, geo = case(n, observer, n + ell)
    b = bins(n)
    ref = oracle.sum_gal(gal, ran, geo, 16, b, ell_max=ell)
    dev = lambda c: tuple(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (c.x, c.y, c.z, c.w, c.nbar))  # noqa: E731
    with ys.Plan(n, geo.box_min, geo.box_len, geo.observer, assign="ngp", compensate=False, ell_max=ell, dk=b.dk,
                 n_bins=b.n_bins, stream=torch.cuda.current_stream().cuda_stream) as plan:
        plan.assign(dev(gal), dev(ran))
        res = plan.measure()
    has = ref.n_modes > 0
    has[-1] = False  # the last shell reaches the 16^3 lattice's Nyquist frequency
    assert np.array_equal(res.n_modes[has], ref.n_modes[has])
    raw = ref.sum0[has] / ref.n_modes[has] / ref.norm.I
    for l in range(0, ell + 1, 2):
        err = np.abs(getattr(res, f"p{l}")[has] - getattr(ref, f"p{l}")[has]) / raw
        assert np.all(err <= COEF[l] * 2e-6), (l, err.max() / COEF[l])
