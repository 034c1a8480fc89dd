"""The error bound of the FP32 evaluation of FP64 words (csrc/kl_common.cuh,
near_words64), restated in numpy: the local pixel coordinates that the FP32
operations give are within E = eps R (64 + 8 q) + c0 of the FP64 ones, also far
outside the window, near the pole and for gamma and v that nearly cancel.  FP32
multiply-adds are formed in FP64 and rounded once."""
import numpy as np
import pytest

import klsynth
import oracle

F = np.float32
EPS = F(2.0 ** -24)


def fma(a, b, c):
    return F(np.float64(a) * np.float64(b) + np.float64(c))


@pytest.mark.parametrize("group", [klsynth.GASKET, klsynth.NEAR_CUSP, klsynth.FUCHSIAN])
@pytest.mark.parametrize("p,sx,sy", [(3, 4096 / 3.0, 4096 / 3.0), (8, 2048 / 0.02, 2048 / 0.02),
                                     (7, 65536 / 3.0, 7 / 3.0), (11, 1024 / 3.0, 512 / 3.0)])
def test_local_coordinates_are_within_the_bound(group, p, sx, sy):
    rng = np.random.default_rng(p)
    g, _ = oracle.group(group.ta, group.tb)
    g = np.asarray(g, dtype=np.float64).reshape(4, 2, 2, 2)
    g = g[..., 0] + 1j * g[..., 1]
    worst, used = 0.0, 0
    for _ in range(80):
        word = [int(rng.integers(4))]
        while len(word) < p:
            w = int(rng.integers(4))
            if w != (word[-1] + 2) % 4:
                word.append(w)
        P = np.eye(2, dtype=complex)
        for w in word:
            P = P @ g[w]
        beta = -(P[0, 0] * P[1, 1] - P[0, 1] * P[1, 0]) / P[1, 0] ** 2
        gamma = P[1, 1] / P[1, 0]
        # points anywhere, and close to the pole -gamma
        v = rng.normal(size=300) + 1j * rng.normal(size=300)
        v[::3] = -gamma + v[::3] * 10.0 ** rng.uniform(-7, 0, size=100)
        frac = rng.random(2)  # alpha's local coordinates
        off = beta / (v + gamma)
        true = np.stack([sx * off.real + frac[0], -sy * off.imag + frac[1]], 1)
        c1, c2 = F((sx * beta).real), F((sx * beta).imag)
        c3, c4 = F((-sy * beta).imag), F((sy * beta).real)
        gr, gi, ax, ay = F(gamma.real), F(gamma.imag), F(frac[0]), F(frac[1])
        vr, vi = v.real.astype(F), v.imag.astype(F)
        wr, wi = F(vr + gr), F(vi + gi)
        m = fma(wr, wr, F(wi * wi))
        rw = F(F(1.0 / np.sqrt(m.astype(np.float64))) * F(1.0 + 2.0 ** -22))  # the root's error
        r = F(rw * rw)
        # sx Re(beta conj(w)) / |w|^2 and -sy Im(beta conj(w)) / |w|^2
        X = F(fma(c1, wr, F(c2 * wi)) * r)
        Y = F(fma(c3, wr, F(c4 * wi)) * r)
        nrm = F(np.sqrt(float(c1) ** 2 + float(c2) ** 2 + float(c3) ** 2 + float(c4) ** 2))
        q = F(F(8) * EPS * F(np.abs(gr) + np.abs(gi) + np.abs(vr) + np.abs(vi)) * rw)
        c0 = F(4) * EPS * F(2 + np.abs(ax) + np.abs(ay))
        E = fma(F(nrm * rw), F(q + F(64) * EPS), c0)
        got = np.stack([F(X + ax), F(Y + ay)], 1).astype(np.float64)
        ok = (m > F(1e-30)) & (m < F(1e30)) & (q < F(0.25))
        used += int(ok.sum())
        worst = max(worst, float((np.abs(got - true).max(1) / E)[ok].max()))
    assert used > 10000 and 0.0 < worst < 1.0, (used, worst)
