"""alpha, I and S / I against exactly rounded sums, for the counting pass and the direct
assignment's sums, over their CTA sizes.

Tolerance 1e-12: a thread adds at most eight particles here; each addition's error (2^-24 of
the sum) is collected in float, so a sum is off by at most 8 x 8 x 2^-48 = 2.3e-13 of itself,
the meeting of the threads (2^-53 and less per addition) adds less, and a result combines
up to four sums.  Sums whose every term is rounded to float miss it (4e-11 and more).
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
ys = pytest.importorskip("paper_1505_05341_gb300")

pytestmark = pytest.mark.gpu


def run(n_gal, n_ran, direct, scale, seed):
    rng = np.random.default_rng(seed)
    cats = []
    for n in (n_gal, n_ran):
        p = (100.0 + 499.0 * rng.random((3, n))).astype(np.float32)
        nbar = (1e-3 * rng.random(n) + 1e-5).astype(np.float32)
        w = (np.float32(scale) / (1.0 + 1e4 * nbar)).astype(np.float32)
        cats.append((p[0], p[1], p[2], w, nbar))
    dev = [tuple(torch.from_numpy(a).cuda() for a in c) for c in cats]
    with ys.Plan(32, (100.0,) * 3, 500.0, dk=0.05, max_particles=n_gal + n_ran,
                 stream=torch.cuda.current_stream().cuda_stream) as plan:
        plan.set_direct_assign(direct)
        plan.assign(*dev)
        res = plan.measure()
    (wg, _), (wr, nb) = [(c[3].astype(np.float64), c[4].astype(np.float64)) for c in cats]
    alpha = math.fsum(wg) / math.fsum(wr)
    norm = alpha * math.fsum(wr * wr * nb)
    shot = math.fsum(wg * wg) + alpha ** 2 * math.fsum(wr * wr)
    for got, want in ((res.alpha, alpha), (res.norm_I, norm), (res.shot_noise, shot / norm)):
        assert abs(got / want - 1.0) <= 1e-12, (got, want)


@pytest.mark.parametrize("direct", [False, True])
@pytest.mark.parametrize("n_gal,n_ran", [(1, 1), (33, 1000), (5_003, 40_001), (20_011, 160_003), (300_007, 1_200_011)])
def test_weighted_sums(n_gal, n_ran, direct):
    run(n_gal, n_ran, direct, 1.0, n_gal)


@pytest.mark.parametrize("direct", [False, True])
def test_sums_beyond_float(direct):
    """w^2 up to 1e38: every thread's sums are floats, those of a warp are not."""
    run(2_000, 9_000, direct, 1e19, 3)
