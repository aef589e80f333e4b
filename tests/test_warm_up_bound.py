"""The warm-up of cascades with coincident poles, checked as mathematics on the
CPU against FP64 impulse responses: with r the largest pole radius, A = prod_k
B_k r^-2 (B_k = |b0| + |b1| + |b2|) and the pole pairs far from the axis counted
as one factor of 1 / sin(angle) r^n instead of two, the tail's energy from the
first n on where A' C(n + m - 1, m - 1) r^n / sqrt(1 - ratio^2) is below 2^-21
||h||_2 is below that too; and the norm of 32 points across the nearest poles'
peaks is one from below."""
import math

import numpy as np
import pytest

import oracle
from synth import filters

N = 1 << 15


def _impulse(sos):
    x = np.zeros(N)
    x[0] = 1.0
    return oracle.sosfilt(x, sos[None], K=np.array([len(sos)], dtype=np.int32),
                          lengths=np.array([N]))[0]


def _rows(sos):
    return sos[:, [0, 1, 2, 4, 5]] / sos[:, 3:4]


def _warm_up(rows, P, norm):
    r, loga, m = 0.0, 0.0, 0
    for b0, b1, b2, a1, a2 in rows:
        p = np.roots([1.0, a1, a2])
        r = max(r, np.abs(p).max())
        loga += math.log(abs(b0) + abs(b1) + abs(b2))
        csc = math.sqrt(a2) / abs(p[0].imag) if p[0].imag else math.inf
        if csc * 2 * len(rows) < P:
            loga, m = loga + math.log(csc), m + 1
        else:
            m += 2
    loga -= 2 * len(rows) * math.log(r) + math.lgamma(m)
    n = np.arange(1, N, dtype=np.float64)
    ratio = r * (n + m) / (n + 1)
    with np.errstate(invalid="ignore", divide="ignore"):
        t = (loga + n * math.log(r) + sum(np.log(n + i) for i in range(1, m))
             - 0.5 * np.log(1 - ratio ** 2))
    ok = (ratio < 1) & (t <= math.log(2.0 ** -21 * norm))
    return int(n[np.argmax(ok)])


def _peak_norm(rows):
    p = [q for row in rows for q in np.roots([1.0, row[3], row[4]])]
    d = 1 - np.abs(p)
    best = 0.0
    for q in p:
        if q.imag < 0 or 1 - abs(q) > 4 * d.min():
            continue
        w = np.angle(q) + (1 - abs(q)) * (0.125 * (np.arange(32) + 0.5) - 2)
        w = w[(w >= 0) & (w <= math.pi)]
        z = np.exp(-1j * w)
        h = np.ones_like(z)
        for b0, b1, b2, a1, a2 in rows:
            h = h * (b0 + b1 * z + b2 * z * z) / (1 + a1 * z + a2 * z * z)
        best = max(best, math.sqrt((np.abs(h) ** 2).sum() * 0.125 * (1 - abs(q)) / math.pi))
    return best


def _cascades():
    out = [np.concatenate([filters.butter_lowpass2_closed_form(wn)] * K)
           for wn in (0.003, 0.01, 0.05) for K in (2, 3, 4, 8)]
    for seed in range(6):
        s = filters.random_sections(9100 + seed, 2, 0.9, 0.99)
        out += [np.concatenate([s[:1]] * 4), np.concatenate([s, s]), np.concatenate([s, s, s])]
    return out


@pytest.mark.parametrize("idx", range(30))
def test_tail_below_the_bound(idx):
    sos = _cascades()[idx]
    h = _impulse(sos)
    norm = np.sqrt((h ** 2).sum())
    low = _peak_norm(_rows(sos))
    assert low <= norm * (1 + 1e-3)
    # at P = 0 every section counts twice; with P large, all complex pairs once
    for P in (0, 200, 1 << 30):
        n = _warm_up(_rows(sos), P, max(low, 1e-3 * norm))
        assert n > 1 and np.sqrt((h[n:] ** 2).sum()) <= 2.0 ** -21 * norm, (P, n)
