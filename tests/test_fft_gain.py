"""Gain of the line transforms (csrc/fft.cuh) with their twiddles and constants as rounded
to float.  Rounding to nearest leaves the moduli of the few constants of a radix-16 butterfly
short, all the same way, which scales every mode and biases P_0; errors of the additions
average out, this one does not.

The transforms are rebuilt here in FP64 with the header's float constants and float tables;
the gain of output k is the mean of Re(M_kn / W_kn) - 1 over the inputs.  Its mean over k must
be no further from zero than 1.15 times that of a transform of radix-8 (radix-4 and 3) stages
whose constants are the nearest floats (P_0 moves by two to four of these gains, and the
window's float roundings by as much as the 15 %); with two radix-16 stages of nearest floats
it is 1.3 to 1.4 times.
"""
import os
import re

import numpy as np
import pytest

HEADER = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1505_05341_gb300", "csrc", "fft.cuh")
f32 = lambda v: np.float64(np.float32(v))  # noqa: E731


def constants():
    """The header's floats: of a line with one radix-16 stage, and of one with two."""
    text = open(HEADER).read()
    k = {n: f32(re.search(r"\b%s = ([0-9.]+)f" % n, text).group(1)) for n in ("h", "s1", "s3")}
    up, near = re.search(r"c1 = LONG \? ([0-9.]+)f : ([0-9.]+)f", text).groups()
    return {**k, "c1": f32(near)}, {**k, "c1": f32(up)}


ONE, TWO = constants()
NEAR = {"h": f32(0.5 ** 0.5), "c1": f32(np.cos(np.pi / 8)), "s1": f32(np.sin(np.pi / 8)), "s3": f32(0.75 ** 0.5)}


def root(turn):
    turn = np.asarray(turn, dtype=np.float64)
    return f32(np.cos(2 * np.pi * turn)) - 1j * f32(np.sin(2 * np.pi * turn))


def d4(v):
    a, b, c, d = v
    return [a + b + c + d, a - c - 1j * (b - d), a + c - b - d, a - c + 1j * (b - d)]


def dft(r, v, k):
    if r == 1:
        return v
    if r == 2:
        return [v[0] + v[1], v[0] - v[1]]
    if r == 3:
        s, d = v[1] + v[2], v[1] - v[2]
        return [v[0] + s, v[0] - 0.5 * s - 1j * k["s3"] * d, v[0] - 0.5 * s + 1j * k["s3"] * d]
    if r == 4:
        return d4(v)
    if r == 8:
        e, o = d4(v[0::2]), d4(v[1::2])
        o = [o[0], k["h"] * (1 - 1j) * o[1], -1j * o[2], -k["h"] * (1 + 1j) * o[3]]
        return [e[i] + o[i] for i in range(4)] + [e[i] - o[i] for i in range(4)]
    out = [None] * r
    if r == 12:  # prime-factor mapping
        t = [dft(3, [v[(3 * b) % 12], v[(4 + 3 * b) % 12], v[(8 + 3 * b) % 12]], k) for b in range(4)]
        for i in range(3):
            for q, x in enumerate(d4([t[b][i] for b in range(4)])):
                out[(4 * i + 9 * q) % 12] = x
        return out
    c, s, h = k["c1"], k["s1"], k["h"]
    w = {1: c - 1j * s, 2: h * (1 - 1j), 3: s - 1j * c, 4: -1j, 6: -h * (1 + 1j), 9: -c + 1j * s}
    t = [d4([v[b], v[4 + b], v[8 + b], v[12 + b]]) for b in range(4)]
    for i in range(4):
        for q, x in enumerate(d4([t[b][i] * (w[b * i] if b * i else 1) for b in range(4)])):
            out[i + 4 * q] = x
    return out


def line(x, n):
    """LineFft<n>: radix R1 over stride n / R1, R2, then E2."""
    p2 = n & (n - 1) == 0
    r1, big = (16, 256) if p2 else (12, 192)
    e2 = max(1, n // big)
    r2, tpl = n // (r1 * e2), n // r1
    K = TWO if r2 == 16 else ONE
    t = np.arange(tpl)
    v = dft(r1, [x[tpl * r:tpl * (r + 1)] for r in range(r1)], K)
    v = [v[k] * (root(t * k / n) if k else np.ones(tpl))[:, None] for k in range(r1)]
    out = np.empty_like(x)
    for k1 in range(r1):
        b = [[y * (root(e * q / (r2 * e2)) if e * q else 1) for q, y in enumerate(dft(r2, [v[k1][e + e2 * s] for s in range(r2)], K))]
             for e in range(e2)]
        for q in range(r2):
            for h, y in enumerate(dft(e2, [b[e][q] for e in range(e2)], K)):
                out[k1 + r1 * q + (n // e2) * h] = y
    return out


def stages(x, radices):
    """Stockham autosort stages with the nearest floats."""
    n, ns = x.shape[0], 1
    for r in radices:
        y, j = np.empty_like(x), np.arange(n // r)
        k = j % ns
        v = dft(r, [x[j + q * (n // r)] * (root(q * k / (ns * r)) if ns > 1 and q else np.ones(n // r))[:, None] for q in range(r)], NEAR)
        for q in range(r):
            y[(j // ns) * ns * r + k + q * ns] = v[q]
        x, ns = y, ns * r
    return x


def plain_radices(n):
    p2 = n & (n - 1) == 0
    m, big, out = (n, 8, []) if p2 else (n // 3, 4, [])
    while m >= big:
        out.append(big)
        m //= big
    return out + ([m] if m > 1 else []) + ([] if p2 else [3])


def mean_gain(m):
    n = m.shape[0]
    w = np.exp(-2j * np.pi * (np.outer(np.arange(n), np.arange(n)) % n) / n)
    assert np.abs(m - w).max() < 1e-6
    return ((m * w.conj()).real - 1.0).mean()


@pytest.mark.parametrize("n", [16, 32, 64, 96, 128, 192, 256, 384, 512, 768, 1024])
def test_mean_gain(n):
    eye = np.eye(n, dtype=complex)
    assert abs(mean_gain(line(eye, n))) <= 1.15 * abs(mean_gain(stages(eye, plain_radices(n))))


def test_constants_within_an_ulp():
    for k, true in (("h", 0.5 ** 0.5), ("c1", np.cos(np.pi / 8)), ("s1", np.sin(np.pi / 8)), ("s3", 0.75 ** 0.5)):
        assert all(abs(c[k] - true) < np.spacing(np.float32(true)) for c in (ONE, TWO)), k
