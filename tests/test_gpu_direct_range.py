"""The galaxy sum's multipoles do not depend on the weights' unit: weights times 2^100 give
the same P_l (both A_0 A_l^* and I scale by 2^200; every float operation scales exactly, so
only the order of the FP64 additions differs: 1e-12 of the raw monopole times the Legendre
coefficients).  m^6 of the 64^3 lattice is up to 2^30, past the float range with them.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
ys = pytest.importorskip("paper_1505_05341_gb300")

pytestmark = pytest.mark.gpu

COEF = {0: 2.0, 2: 10.0, 4: 76.5, 6: 533.0}


@pytest.mark.parametrize("ell", [0, 2, 4, 6])
def test_unit_of_the_weights(ell):
    rng = np.random.default_rng(ell)
    pos = (50.0 + 300.0 * rng.random((3, 900))).astype(np.float32)
    w = rng.uniform(0.5, 1.5, 900).astype(np.float32)

    def run(scale):
        cat = lambda s: tuple(torch.from_numpy(np.ascontiguousarray(a[s])).cuda()  # noqa: E731
                              for a in (*pos, w * np.float32(scale), np.full(900, 1e-4, np.float32)))
        return ys.sum_gal(64, (50.0,) * 3, 300.0, cat(slice(0, 200)), cat(slice(200, 900)), ell_max=ell, dk=0.05, wedges=True)

    (a, wa), (b, wb) = run(1.0), run(2.0 ** 100)
    raw = np.abs(a.p0 + a.shot_noise)
    has = a.n_modes > 0
    for l in range(0, ell + 1, 2):
        x, y = getattr(a, f"p{l}")[has], getattr(b, f"p{l}")[has]
        assert np.all(np.abs(x - y) <= 1e-12 * COEF[l] * raw[has]), l
    for x, y in zip(wa, wb):
        assert np.all(np.abs(x[has] - y[has]) <= 1e-12 * 4 * raw[has])
