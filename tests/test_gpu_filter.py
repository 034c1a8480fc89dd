"""The certified FP32 filter of the FP64 and double-float renders: the image is
bit for bit the one that the exact per-word map gives.  kl_eval_words returns
that map's pixel coordinates for every word; binning them is the expected image
(no tolerance)."""
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


G, N = klsynth.GASKET, klsynth.NEAR_CUSP
B = klsynth.draw_groups(klsynth.BATCH_SEED, 8)[7][0]
FULL = (-1.5, 1.5, -1.5, 1.5)
CASES = [
    (G, 2, 0, 64, 64, FULL),                            # one prefix letter, one suffix point
    (G, 10, 0, 1024, 1024, FULL),                       # one point per first letter
    (N, 11, 8, 333, 1000, (-2.0, 2.0, -2.0, 2.0)),      # pixels three times as wide as high
    (B, 12, 4, 5000, 7, (-1.5, 1.5, -1.5, 1.5)),        # very flat pixels
    (G, 12, 1, 8192, 8192, FULL),                       # large offsets: queues overflow
    (N, 13, 5, 512, 512, (0.9, 0.9002, 0.1, 0.1002)),   # a window far smaller than a prefix's piece
    (N, 11, 0, 256, 256, (1e4, 1e4 + 1.0, 0.0, 1.0)),   # nothing in the window, far alpha
    (B, 13, 0, 1, 1, FULL),                             # one pixel
]


@pytest.mark.parametrize("prec", ["fp64", "df64"])
@pytest.mark.parametrize("group,d,plen,W,H,window", CASES)
def test_image_is_the_exact_maps(kl, group, d, plen, W, H, window, prec):
    check(kl, kl.params_init(group.ta, group.tb, d, W, H, window,
                             {"fp64": kl.FP64, "df64": kl.DF64}[prec], prefix_len=plen))


@pytest.mark.parametrize("prec", ["fp64", "df64"])
def test_prefixes_without_a_pole(kl, prec):
    """Maskit's b(z) = z + 2: the prefixes b^p and B^p have no pole form."""
    gens, seeds = kl.maskit(-0.097 + 1.838j)
    check(kl, kl.params_group(gens, seeds, 11, 700, 500, (-1.0, 3.0, -0.08, 1.92),
                              {"fp64": kl.FP64, "df64": kl.DF64}[prec], prefix_len=3))


def check(kl, p):
    """kl_eval_words returns a double-float coordinate as the FP64 sum of its two
    parts, which loses a low part below 2^-53 of the high one: where that sum is
    a whole number, the word may lie just below it (Maskit's words on the real
    axis do), in the pixel before.  Such words are placed by their number only."""
    import torch
    n = kl.word_count(p.depth)
    uv = kl.eval_words(p, torch.arange(n, device="cuda"))
    image, counters = kl.render(p)
    image = image.reshape(-1).to(torch.int64)

    def binned(words, du=0, dv=0):
        u, v = torch.floor(words[:, 0]) - du, torch.floor(words[:, 1]) - dv
        ok = (u >= 0) & (u < p.width) & (v >= 0) & (v < p.height)
        at = v[ok].to(torch.int64) * p.width + u[ok].to(torch.int64)
        return torch.bincount(at, minlength=p.width * p.height)

    whole = (uv == torch.floor(uv)).any(dim=1)
    if p.precision != kl.DF64:
        whole[:] = False
    rest = image - binned(uv[~whole])
    may = sum(binned(uv[whole], du, dv) for du in (0, 1) for dv in (0, 1))
    assert bool((rest >= 0).all()) and bool((rest <= may).all())
    assert int(rest.sum()) <= int(whole.sum())
    assert int(counters[0]) == int(image.sum()) and int(counters[0] + counters[1]) == n
