"""Rows past the end of the last tile leave no trace in the gradient: weights for which the
given rows stay finite but an all-zero row overflows in the second hidden layer.

Only the first input feeds the first layer, W1[o] x_0 + b1[o] with b1 = -W1 = 3e38: zero for
the rows given (x_0 = 1; W2's gradient is then exactly zero), 3e38 for x = 0.  Every value of
the given rows is small, so the gradient test's bars apply: each layer within 1e-3 of its
largest gradient.
"""
import numpy as np
import pytest

from oracle import mlp as ref

torch = pytest.importorskip("torch")
ys = pytest.importorskip("paper_1505_05341_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 63, 64, 65, 190])
def test_rows_past_the_end(rows):
    p = ref.init_params(5).astype(np.float32)
    big = ref.bf16_round(np.full(1, 3e38)).astype(np.float32)[0]
    w1 = np.zeros((64, 5), np.float32)
    w1[:, 0] = -big
    p[:320], p[320:384] = w1.ravel(), big
    p[384:384 + 64 * 64] *= 16.0
    rng = np.random.default_rng(rows)
    X = rng.standard_normal((rows, 5)).astype(np.float32)
    X[:, 0] = 1.0
    T = rng.standard_normal((rows, 3)).astype(np.float32)
    net = ys.Mlp(p)
    g = torch.empty(ys.MLP_PARAMS, dtype=torch.float32, device="cuda")
    sse = torch.zeros(1, dtype=torch.float64, device="cuda")
    net.gradient(torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda(), d_grad=g, d_sse=sse)
    got = g.cpu().numpy().astype(np.float64)
    loss, want = ref.loss_and_grad(ref.bf16_round(p), X.astype(np.float64), T.astype(np.float64))
    assert np.all(np.isfinite(want)) and np.all(np.isfinite(got))
    assert abs(sse.item() / (3 * rows) - loss) <= 1e-5 * loss
    at = 0
    for fan_in, fan_out in ref.LAYERS:
        for size in (fan_in * fan_out, fan_out):
            a, b = got[at:at + size], want[at:at + size]
            assert np.abs(a - b).max() <= 1e-3 * np.abs(b).max(), at
            at += size
    net.close()
