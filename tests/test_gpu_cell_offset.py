"""Sub-cell offsets carry no common stretch: 1 / H is used beyond its float rounding.

Particles of unit weight sit on nodes in y and z and at random places between two nodes in
x (CIC), each alone in its pair of nodes, so a node holds the offset d itself.  The mean of
d_gpu / d over M particles must be 1 to within 5 standard errors of the float roundings of
one offset (at most 2^-24 relative for d >= 1/2, uniform, so 2^-24 / sqrt(3 M)); with a
rounded 1 / H it is off by that rounding, 4.7e-8 for these sides.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
ys = pytest.importorskip("paper_1505_05341_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("direct", [False, True])
@pytest.mark.parametrize("n,side", [(64, 500.0), (32, 1000.0)])
def test_offsets_are_not_stretched(n, side, direct):
    h = side / n
    rng = np.random.default_rng(n)
    ix, iy, iz = np.meshgrid(np.arange(0, n, 2), np.arange(0, n, 1), np.arange(0, n, 1), indexing="ij")
    x = (h * (ix.ravel() + 0.5 + 0.499 * rng.random(ix.size))).astype(np.float32)
    y, z = (np.float32(h) * a.ravel().astype(np.float32) for a in (iy, iz))
    d = x.astype(np.float64) / h - ix.ravel()
    one = np.ones(x.size, np.float32)
    dev = lambda *c: tuple(torch.from_numpy(a).cuda() for a in c)  # noqa: E731
    with ys.Plan(n, (0.0,) * 3, side, assign="cic", dk=0.05, n_bins=4, alpha=1.0, max_particles=x.size,
                 stream=torch.cuda.current_stream().cuda_stream) as plan:
        plan.set_direct_assign(direct)
        plan.assign(dev(x, y, z, one, one), dev(*(np.zeros(0, np.float32),) * 5))
        mesh = np.asarray(plan.mesh(), dtype=np.float64).reshape(n, n, n)
    got = mesh[ix.ravel() + 1, iy.ravel(), iz.ravel()]
    assert abs(np.mean(got / d) - 1.0) <= 5 * 2.0 ** -24 / np.sqrt(3 * x.size)
