"""The error bound of the FP32 filter (csrc/kl_filter.cuh), restated in numpy:
the offset that the FP32 operations give is within E = eps R (64 + 32 |g| R) +
c0 of the FP64 one, R any bound on the offset.  FP32 multiply-adds are formed
in FP64 and rounded once."""
import numpy as np
import pytest

import klsynth
import oracle

F = np.float32
EPS = 2.0 ** -24


def fma(a, b, c):
    return F(np.float64(a) * np.float64(b) + np.float64(c))


@pytest.mark.parametrize("group", [klsynth.GASKET, klsynth.NEAR_CUSP, klsynth.FUCHSIAN,
                                   klsynth.Group(2.7 - 0.03j, 2.1 + 0.05j)])
@pytest.mark.parametrize("p,sx", [(3, 4096 / 3.0), (7, 8192 / 4.0), (11, 1024 / 3.0)])
def test_offset_error_is_below_the_bound(group, p, sx):
    rng = np.random.default_rng(p)
    g, seeds = oracle.group(group.ta, group.tb)
    g = np.asarray(g, dtype=np.float64).reshape(4, 2, 2, 2)
    g = g[..., 0] + 1j * g[..., 1]
    worst = 0.0
    for _ in range(60):
        word = [int(rng.integers(4))]
        while len(word) < p + 8:
            w = int(rng.integers(4))
            if w != (word[-1] + 2) % 4:
                word.append(w)
        P = np.eye(2, dtype=complex)
        for w in word[:p]:
            P = P @ g[w]
        # suffix points starting with the word's next letter, of several depths
        v = []
        for depth in range(1, 9):
            s = np.asarray(seeds, dtype=np.float64).reshape(4, 2)
            z = complex(*s[word[p + depth - 1]])
            for w in reversed(word[p:p + depth]):
                M = g[w]
                z = (M[0, 0] * z + M[0, 1]) / (M[1, 0] * z + M[1, 1])
            v.append(z)
        v = np.array(v)
        beta = -(P[0, 0] * P[1, 1] - P[0, 1] * P[1, 0]) / P[1, 0] ** 2
        gamma = P[1, 1] / P[1, 0]
        off = 1.0 / ((v + gamma) / (sx * beta))
        true = np.stack([off.real, -off.imag], 1)
        b1, b2 = F((sx * beta).real), F((sx * beta).imag)
        q = F(1.0 / np.float64(fma(b1, b1, F(b2 * b2))))
        k1, k2 = F(b1 * q), F(-b2 * q)
        gr, gi = F(gamma.real), F(gamma.imag)
        g1, g2 = fma(k1, gr, -F(k2 * gi)), fma(k1, gi, F(k2 * gr))
        vr, vi = v.real.astype(F), v.imag.astype(F)
        wr = fma(k1, vr, fma(-k2, vi, g1))
        wi = fma(k2, vr, fma(k1, vi, g2))
        r = F(1.0 / np.float64(fma(wr, wr, (wi * wi).astype(F))))
        r = F(r * (1.0 + 2.0 ** -23))                     # the reciprocal seed's error
        got = np.stack([F(wr * r), F(wi * r)], 1).astype(np.float64)
        R = np.abs(got).sum(1)
        E = EPS * R * (64 + 32 * (abs(g1) + abs(g2)) * R) + 4 * EPS * 2
        worst = max(worst, float((np.abs(got - true).max(1) / E).max()))
    assert 0.0 < worst < 1.0, worst
