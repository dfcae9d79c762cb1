"""The sorted assignment with every scatter-tile shape the autotuner may choose, node by node
against the FP64 oracle deposit: tiles that do not fit twice in shared memory (float sums, by
clusters of CTAs where tiles are few), binning codes with other tile counts, and meshes past
256^3 whose larger tiles bring them back to the aggregated binning without codes.

Bar as in the mesh tests: 2e-6 A + 1e-6 max(A), A the deposit of |w|.
"""
import numpy as np
import pytest

import synth
from oracle.assignment import assign_mesh

torch = pytest.importorskip("torch")
ys = pytest.importorskip("paper_1505_05341_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,kind,interlace,tile", [
    (64, "tsc", True, (32, 16, 32)),     # 16 tiles, float sums, clusters of 8
    (96, "cic", True, (32, 16, 32)),     # 54 tiles, float sums, clusters
    (64, "cic", False, (32, 16, 32)),    # fixed point in clusters
    (32, "tsc", True, (8, 8, 32)),       # one tile along z
    (128, "tsc", True, (8, 16, 32)),     # 512 tiles
    (128, "ngp", False, (8, 8, 32)),     # 1024 tiles
    (256, "cic", False, (8, 16, 32)),    # 4096 tiles: the last with codes
    (256, "tsc", False, (8, 8, 32)),     # 8192 tiles: one cursor atomic per record
    (256, "cic", True, (32, 16, 32)),    # 1024 tiles, float sums
    (384, "cic", False, (32, 16, 32)),   # 3456 tiles, aggregated, located twice
])
def test_tile_shapes(n, kind, interlace, tile):
    lib = ys.load_library()
    gal, ran, geo = synth.poisson_cube(30_011, 120_007, side=500.0, seed=n + tile[0])
    rng = np.random.default_rng(n)
    gal.w[:] = rng.uniform(0.2, 2.0, gal.w.size)
    ran.w[:] = rng.uniform(0.2, 2.0, ran.w.size)
    dev = lambda c: tuple(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (c.x, c.y, c.z, c.w, c.nbar))  # noqa: E731
    with ys.Plan(n, geo.box_min, geo.box_len, geo.observer, assign=kind, interlace=interlace, dk=0.05, n_bins=4, alpha=0.25,
                 max_particles=gal.n + ran.n, stream=torch.cuda.current_stream().cuda_stream) as plan:
        lib._ZN2ys9set_tilesERNS_4PlanEiii(plan._h, *tile)  # ys::set_tiles, as the autotuner calls it
        plan.assign(dev(gal), dev(ran))
        got = plan.mesh()
        plan.measure()
    for j, shift in enumerate([False, True] if interlace else [False]):
        ref = assign_mesh(gal, ran, 0.25, geo.box_min, geo.box_len, n, kind, interlaced=shift)
        bound = assign_mesh(gal, ran, -0.25, geo.box_min, geo.box_len, n, kind, interlaced=shift)
        err = np.abs(got[j] - ref) / (2e-6 * bound + 1e-6 * bound.max())
        assert err.max() <= 1.0, (j, err.max())
