"""Words of a mixed render's FP64 prefixes are placed in FP32 where an error
bound settles their pixel: with every prefix near-parabolic the image is the FP64
render's of the same split, value for value, single and batched."""
import pytest

import klsynth

pytestmark = pytest.mark.gpu

N, G = klsynth.NEAR_CUSP, klsynth.GASKET
B = klsynth.draw_groups(klsynth.BATCH_SEED, 8)[7][0]
CASES = [
    (G, 2, 1, 64, 64, (-1.5, 1.5, -1.5, 1.5)),            # one suffix point per letter
    (N, 13, 4, 512, 512, (-2.0, 2.0, -2.0, 2.0)),         # several chunks of suffix points
    (B, 12, 6, 5000, 7, (-1.5, 1.5, -1.5, 1.5)),          # very flat pixels
    (B, 12, 6, 7, 5000, (-1.5, 1.5, -1.5, 1.5)),          # very tall pixels
    (N, 13, 5, 512, 512, (0.9, 0.9002, 0.1, 0.1002)),     # large offsets: few words settled
    (G, 13, 6, 8192, 8192, (-1.5, 1.5, -1.5, 1.5)),
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


@pytest.mark.parametrize("group,d,plen,W,H,window", CASES)
def test_near_parabolic_words_are_the_fp64_renders(kl, group, d, plen, W, H, window):
    import torch

    def make(prec):
        return kl.params_init(group.ta, group.tb, d, W, H, window, prec, prefix_len=plen,
                              parabolic_tol=1e6)

    want, cw = kl.render(make(kl.FP64))
    image, c = kl.render(make(kl.MIXED))
    assert torch.equal(image, want)
    assert torch.equal(c[:2], cw[:2]) and int(c[2]) == kl.word_count(d)
    batch = kl.Batch([make(kl.MIXED)] * 2)
    images, counters = batch.render()
    for g in range(2):
        assert torch.equal(images[g], want)
        assert torch.equal(counters[g, :3], c[:3])
