"""The FP32 leaf test of the scan (csrc/kl_fsa.cu, fsa_leaf32), restated in
numpy: a leaf that it settles lies in that pixel in FP64, whatever the scale of
the generator's matrix (a Moebius map does not depend on it) and of the point.
FP32 multiply-adds are formed in FP64 and rounded once."""
import numpy as np
import pytest

import klsynth
import oracle

F = np.float32
EPS = F(2.0 ** -24)
TINY = F(2.0 ** -76)
UNSETTLED = -2
W, H = 400, 300
X0, X1, Y0, Y1 = -1.51, 1.5, -1.2, 1.313  # (0 inside a pixel)


def fma(a, b, c):
    return F(np.float64(a) * np.float64(b) + np.float64(c))


def leaf32(M, z):
    """Pixels of the points z under the matrix M = (p, q, r, s)."""
    v = np.array([[m.real, m.imag] for m in M]).astype(F)
    n1 = np.abs(v).sum(axis=1, dtype=F)
    np_, nq, nr_, ns = n1[0], F(n1[1] + TINY), n1[2], F(n1[3] + TINY)
    zr, zi = z.real.astype(F), z.imag.astype(F)

    def row(a, b):
        return (fma(v[a, 0], zr, fma(-v[a, 1], zi, v[b, 0])),
                fma(v[a, 0], zi, fma(v[a, 1], zr, v[b, 1])))
    nr, ni = row(0, 1)
    dr, di = row(2, 3)
    m = fma(dr, dr, F(di * di))
    flushed = np.where(m < F(2.0 ** -126), 0.0, m.astype(np.float64))
    rd = F(F(1.0 / np.sqrt(flushed)) * F(1.0 + 2.0 ** -23))      # the root's own error
    rc = F(rd * rd)
    wr, wi = F(fma(nr, dr, F(ni * di)) * rc), F(fma(ni, dr, -F(nr * di)) * rc)
    az, aw = F(np.abs(zr) + np.abs(zi)), F(np.abs(wr) + np.abs(wi))
    A, B = fma(np_, az, nq), fma(nr_, az, ns)
    x0, y1 = F(X0), F(Y1)
    sx, sy = F(W / (X1 - X0)), F(H / (Y1 - Y0))
    u, w = F(F(wr - x0) * sx), F(F(y1 - wi) * sy)
    e = fma(F(F(12) * EPS * rd), fma(aw, B, A), F(F(20) * EPS * aw))
    eu = F(fma(F(5) * EPS, np.abs(x0), e) * sx)
    ew = F(fma(F(5) * EPS, np.abs(y1), e) * sy)
    ok = ((m > F(1e-30)) & (m < F(1e30)) & (az < F(1e15)) &
          (F(F(12) * EPS * B) * rd < F(0.25)) & (eu < F(0.25)) & (ew < F(0.25)))
    out = (u < -eu) | (u > F(W) + eu) | (w < -ew) | (w > F(H) + ew)
    c0, c1 = np.floor(F(u - eu)), np.floor(F(u + eu))
    r0, r1 = np.floor(F(w - ew)), np.floor(F(w + ew))
    one = (c0 == c1) & (r0 == r1) & (c0 >= 0) & (r0 >= 0) & (c0 < W) & (r0 < H)
    inside = np.where(ok & one, r0 * W + c0, 0).astype(np.int64)
    return np.where(ok & out, -1, np.where(ok & one, inside, UNSETTLED))


@pytest.mark.parametrize("power", [-130, -100, -70, -64, -50, -40, 0, 40, 55, 60, 62, 63, 64, 65,
                                   66, 80, 120, 127])
def test_a_settled_leaf_is_in_its_pixel(power):
    rng = np.random.default_rng(power + 200)
    g, _ = oracle.group(klsynth.NEAR_CUSP.ta, klsynth.NEAR_CUSP.tb)
    g = np.asarray(g, dtype=np.float64).reshape(4, 4, 2)
    maps = list(g[..., 0] + 1j * g[..., 1])
    maps += list(rng.normal(size=(4, 4)) + 1j * rng.normal(size=(4, 4)))
    settled = total = 0
    for M in maps:
        # points near 0, ordinary, far, and near the pole -s / r
        z = rng.normal(size=4000) + 1j * rng.normal(size=4000)
        z *= 10.0 ** rng.choice([-18, -3, 0, 0, 0, 3, 16], size=4000)
        z[::8] = -M[3] / M[2] + 1e-3 * z[::8]
        S = M * 2.0 ** power
        with np.errstate(all="ignore"):
            pix = leaf32(S, z)
            w = (M[0] * z + M[1]) / (M[2] * z + M[3])
        u, v = (w.real - X0) * (W / (X1 - X0)), (Y1 - w.imag) * (H / (Y1 - Y0))
        inside = (u >= 0) & (u < W) & (v >= 0) & (v < H)
        want = np.where(inside, np.floor(v) * W + np.floor(u), -1).astype(np.int64)
        clear = (np.abs(u - np.round(u)) > 1e-9) & (np.abs(v - np.round(v)) > 1e-9)
        use = (pix != UNSETTLED) & clear
        assert np.array_equal(pix[use], want[use])
        settled += int(use.sum())
        total += z.size
    if -40 <= power <= 40:
        assert settled > 0.5 * total
