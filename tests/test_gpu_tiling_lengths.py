"""A tiling render is the sum of the renders of its lengths, value for value:
lengths that share prefix tables go together in one launch (10 .. 17 of the
default plans), others are renders of their own, the short ones are walked as
trees; the sizes are the edges of those ranges."""
import pytest

import klsynth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kl():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device for a gpu-marked test")
    from paper_1709_08018_gb300 import build
    build.build()
    import paper_1709_08018_gb300 as kl
    return kl


@pytest.mark.parametrize("prec", ["fp64", "mixed", "df64"])
@pytest.mark.parametrize("d,fields", [(9, {}), (10, {}), (11, {"block_threads": 64}),
                                      (14, {"prefix_len": 6}), (17, {"block_threads": 256}),
                                      (18, {})])
def test_tiling_is_the_sum_of_its_lengths(kl, d, fields, prec):
    import torch
    prec = {"fp64": kl.FP64, "mixed": kl.MIXED, "df64": kl.DF64}[prec]
    g = klsynth.NEAR_CUSP

    def one(depth, **more):
        p = kl.params_init(g.ta, g.tb, depth, 801, 333, (-1.7, 1.6, -1.2, 1.3), prec, **more)
        image, counters = kl.render(p)
        return image.to(torch.int64), counters[:3].clone()

    image, words = one(d, mode=kl.TILING, **fields)
    want, count = one(9, mode=kl.TILING)
    for k in range(10, d + 1):
        i, c = one(k, **(fields if k == d else {}))
        want, count = want + i, count + c
    assert torch.equal(image, want)
    assert torch.equal(words, count)
    assert int(words[0] + words[1]) == 2 * (3 ** d - 1)


@pytest.mark.parametrize("d", range(1, 10))
def test_short_lengths_are_the_words_evaluated_one_by_one(kl, d):
    """FP64 words in plain numpy, one by one; a word within 1e-6 pixel of an
    edge (FP64 rounding is far below that) may fall to either side."""
    import numpy as np
    p = kl.params_init(2.3 + 0.02j, 2.7 - 0.03j, d, 301, 217, (-1.3, 1.4, -1.1, 1.2), kl.FP64,
                       mode=kl.TILING)
    image, counters = kl.render(p)
    g = np.array(list(p.gens)).reshape(4, 4, 2)
    M = g[..., 0] + 1j * g[..., 1]
    s = np.array(list(p.seeds)).reshape(4, 2)
    sx, sy = p.width / (p.x1 - p.x0), p.height / (p.y1 - p.y0)
    z = [np.array([complex(*s[x])]) for x in range(4)]
    want, near, total = np.zeros((p.height, p.width), dtype=np.int64), 0, 0
    for k in range(1, d + 1):
        right = z if k == 1 else [np.concatenate([z[y] for y in range(4) if y != (x + 2) % 4])
                                  for x in range(4)]
        z = [(M[x, 0] * right[x] + M[x, 1]) / (M[x, 2] * right[x] + M[x, 3]) for x in range(4)]
        w = np.concatenate(z)
        u, v = (w.real - p.x0) * sx, (p.y1 - w.imag) * sy
        near += int(((np.abs(u - np.round(u)) < 1e-6) | (np.abs(v - np.round(v)) < 1e-6)).sum())
        ok = (u >= 0) & (u < p.width) & (v >= 0) & (v < p.height)
        np.add.at(want, (v[ok].astype(int), u[ok].astype(int)), 1)
        total += w.size
    assert int(counters[0] + counters[1]) == total == 2 * (3 ** d - 1)
    assert int(np.abs(image.cpu().numpy().astype(np.int64) - want).sum()) <= 2 * near
