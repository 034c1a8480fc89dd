"""Renders whose prefixes the FP32 filter does not serve (views and pixels out of
its range): the exact map alone, one prefix to a lane.  The image is the one that
kl_eval_words gives, word for word, as for filtered renders."""
import pytest

import klsynth
from test_gpu_filter import check, kl  # noqa: F401

pytestmark = pytest.mark.gpu

N = klsynth.NEAR_CUSP


def params(kl, prec, d, half, plen=0, W=300, H=260, flat=1.0):  # noqa: F811
    """A view of half width `half` (height: over `flat`) a little off the fixed
    point of a."""
    p = kl.params_init(N.ta, N.tb, d, W, H, (-1.0, 1.0, -1.0, 1.0),
                       {"fp64": kl.FP64, "df64": kl.DF64, "mixed": kl.MIXED}[prec],
                       prefix_len=plen)
    a = [complex(p.gens[2 * k], p.gens[2 * k + 1]) for k in range(4)]
    z = 0.3 + 0.1j
    for _ in range(300):
        z = (a[0] * z + a[1]) / (a[2] * z + a[3])
    z += half * (0.0123 + 0.0171j)
    p.x0, p.x1 = z.real - half, z.real + half
    p.y0, p.y1 = z.imag - half / flat, z.imag + half / flat
    return p


@pytest.mark.parametrize("prec", ["fp64", "df64"])
@pytest.mark.parametrize("d,half,plen,flat", [
    (11, 1e15, 0, 1.0),    # all words in one pixel
    (11, 1e-13, 0, 1.0),   # pixels far smaller than the words' rounding
    (12, 1e15, 3, 1.0),    # nine prefixes of a letter: the warp's lanes share them
    (13, 1e15, 4, 1.0),    # 27 prefixes of a letter: a lane each, five lanes idle
    (11, 1.3, 4, 3e7),     # pixels far wider than high
    (12, 1e-6, 5, 1.0),    # in range, nothing certified: full queues
    (12, 2000.0, 0, 1.0),  # the limit set well inside one pixel, in range
    (12, 60.0, 0, 1.0),    # in a few pixels
    (8, 1e-13, 0, 1.0),    # one word to a prefix and letter
    (9, 1e-13, 7, 1.0),    # three
])
def test_exact_map_alone(kl, prec, d, half, plen, flat):  # noqa: F811
    check(kl, params(kl, prec, d, half, plen, flat=flat))


@pytest.mark.parametrize("prec", ["fp64", "df64", "mixed"])
@pytest.mark.parametrize("half", [1e15, 1e-13])
def test_tiling_out_of_range(kl, prec, half):  # noqa: F811
    import torch

    def one(d, mode):
        p = params(kl, prec, d, half)
        p.mode = mode
        image, counters = kl.render(p)
        return image.to(torch.int64), counters[:2].clone()

    image, words = one(12, kl.TILING)
    want, count = one(9, kl.TILING)
    for d in (10, 11, 12):
        i, c = one(d, kl.LIMIT_SET)
        want, count = want + i, count + c
    assert torch.equal(image, want) and torch.equal(words, count)
