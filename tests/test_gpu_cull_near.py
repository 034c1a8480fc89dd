"""Culled renders of FP64 prefixes test blocks and words in FP32 with an error
bound first: the image and the counts are those of the per-word render of the
same split, value for value (FP64, and mixed with every prefix near-parabolic)."""
import pytest

import klsynth

pytestmark = pytest.mark.gpu

N, G = klsynth.NEAR_CUSP, klsynth.GASKET
B = klsynth.draw_groups(klsynth.BATCH_SEED, 8)[7][0]
CASES = [
    (G, 4, 2, 64, 64, (-1.5, 1.5, -1.5, 1.5)),            # blocks of fewer than 9 points
    (N, 13, 4, 512, 512, (-2.0, 2.0, -2.0, 2.0)),         # large blocks
    (B, 14, 7, 5000, 7, (-1.5, 1.5, -1.5, 1.5)),          # very flat pixels
    (B, 14, 7, 7, 5000, (-1.5, 1.5, -1.5, 1.5)),          # very tall pixels
    (N, 13, 5, 512, 512, (0.9, 0.9002, 0.1, 0.1002)),     # a window far smaller than a block
    (G, 15, 6, 8192, 8192, (-1.5, 1.5, -1.5, 1.5)),       # most words of a block apart
    (N, 12, 3, 256, 256, (1e4, 1e4 + 1.0, 0.0, 1.0)),     # nothing in the window
    (B, 13, 5, 1, 1, (-1.5, 1.5, -1.5, 1.5)),             # one pixel
]


@pytest.fixture(scope="module")
def kl():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device for a gpu-marked test")
    from paper_1709_08018_gb300 import build
    build.build()
    import paper_1709_08018_gb300 as kl
    return kl


def both(kl, make):
    import torch
    (a, ca), (b, cb) = (kl.render(make(cull)) for cull in (0, 1))
    assert torch.equal(a, b)
    assert torch.equal(ca[:3], cb[:3])


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("group,d,plen,W,H,window", CASES)
def test_culled_is_the_per_word_render(kl, group, d, plen, W, H, window, prec):
    fields = {"parabolic_tol": 1e6} if prec == "mixed" else {}
    both(kl, lambda cull: kl.params_init(group.ta, group.tb, d, W, H, window,
                                         {"fp64": kl.FP64, "mixed": kl.MIXED}[prec],
                                         prefix_len=plen, cull=cull, **fields))


def test_prefixes_without_a_pole(kl):
    gens, seeds = kl.maskit(-0.097 + 1.838j)
    both(kl, lambda cull: kl.params_group(gens, seeds, 12, 700, 500, (-1.0, 3.0, -0.08, 1.92),
                                          kl.FP64, prefix_len=4, cull=cull))
