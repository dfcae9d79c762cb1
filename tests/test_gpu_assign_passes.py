"""The assignment's passes where their rules switch: one particle, catalogues around the
counting pass's two CTA sizes, tiles shared by clusters of 8, 4, 2 and 1 CTAs, the
aggregated binning (up to 4096 tiles) and the one with a cursor atomic per record, the
two-part scan (more than 1024 tiles), and either catalogue empty.

Node by node against the FP64 oracle deposit with the mesh tests' bar, 2e-6 A +
1e-6 max(A) (A the deposit of |w|).  The catalogue sums have their bars in the parity tests.
"""
import numpy as np
import pytest

import synth
from oracle.assignment import assign_mesh
from synth.catalogs import Catalog

torch = pytest.importorskip("torch")
ys = pytest.importorskip("paper_1505_05341_gb300")

pytestmark = pytest.mark.gpu


def _dev(cat, n):
    return tuple(torch.from_numpy(np.ascontiguousarray(a[:n])).cuda() for a in (cat.x, cat.y, cat.z, cat.w, cat.nbar))


@pytest.mark.parametrize("n,kind,interlace,n_gal,n_ran", [
    (16, "tsc", False, 40_000, 80_001),     # one tile, a cluster of 8
    (32, "cic", True, 1, 1),                # one particle each
    (32, "tsc", True, 0, 2_047),            # no galaxies
    (64, "ngp", False, 70_000, 0),          # no randoms
    (64, "cic", False, 20_011, 160_003),    # just above one particle per thread of the large counting CTAs
    (96, "tsc", True, 300_001, 299_999),    # 216 tiles, a cluster of 4
    (128, "cic", True, 400_000, 1_000_003),  # 512 tiles, a cluster of 2
    (256, "tsc", False, 3_000, 20_000),     # 4096 tiles, aggregated binning
    (384, "tsc", True, 3_000, 20_000),      # 13824 tiles, one cursor atomic per record
])
def test_passes(n, kind, interlace, n_gal, n_ran):
    gal, ran, geo = synth.poisson_cube(max(n_gal, 1), max(n_ran, 1), side=500.0, seed=n + 3)
    rng = np.random.default_rng(n)
    gal.w[:] = rng.integers(1, 9, gal.w.size) / 4.0
    ran.w[:] = rng.integers(1, 9, ran.w.size) / 4.0
    alpha = 0.25
    with ys.Plan(n, geo.box_min, geo.box_len, geo.observer, assign=kind, interlace=interlace, dk=0.05, n_bins=4,
                 alpha=alpha, stream=torch.cuda.current_stream().cuda_stream) as plan:
        plan.assign(_dev(gal, n_gal), _dev(ran, n_ran))
        got = plan.mesh()
        res = plan.measure()
    assert res.alpha == alpha and (n_ran == 0 or res.norm_I > 0)
    cut = lambda c, m: Catalog(c.x[:m], c.y[:m], c.z[:m], c.w[:m], c.nbar[:m])  # noqa: E731
    g, r = cut(gal, n_gal), cut(ran, n_ran)
    for j, shift in enumerate([False, True] if interlace else [False]):
        ref = assign_mesh(g, r, alpha, geo.box_min, geo.box_len, n, kind, interlaced=shift)
        bound = assign_mesh(g, r, -alpha, geo.box_min, geo.box_len, n, kind, interlaced=shift)
        err = np.abs(got[j] - ref) / (2e-6 * bound + 1e-6 * bound.max())
        assert err.max() <= 1.0, (j, err.max())
