"""Work items at the ends of their range: the longest words in the smallest
chunks of suffix points, every word drawn or dropped once."""
import pytest

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
def test_longest_words_in_the_smallest_chunks(kl, prec):
    """24 letters, one pair of points to a chunk: 5.9e9 items of 32 prefixes
    would overflow the 32-bit item count."""
    p = kl.params_init(2.1 + 0.01j, 2.3, 24, 64, 64, (-1.5, 1.5, -1.5, 1.5),
                       {"fp64": kl.FP64, "mixed": kl.MIXED, "df64": kl.DF64}[prec],
                       chunk_pairs=1)
    image, counters = kl.render(p)
    assert int(counters[0]) + int(counters[1]) == kl.word_count(24)
    assert int(image.long().bitwise_and(0xFFFFFFFF).sum()) % 2 ** 32 == int(counters[0]) % 2 ** 32


def test_batch_of_long_words_in_the_smallest_chunks(kl):
    """Four FP64 groups of 22 letters, one pair of points to a chunk: 2.6e9
    items of 32 prefixes, 6.5e8 with chunks four times as long."""
    make = lambda side: kl.params_init(2.1 + 0.01j, 2.3, 22, side, side, (-1.5, 1.5, -1.5, 1.5),
                                       kl.FP64, chunk_pairs=1)
    images, counters = kl.Batch([make(64)] * 4).render()
    want, count = kl.render(make(64))
    for g in range(4):
        assert int(counters[g, 0]) + int(counters[g, 1]) == kl.word_count(22)
        assert int(images[g].long().sum()) == int(counters[g, 0])
    assert bool((images[1:] == images[0]).all())
    # the batch splits the words at other letters: words on a pixel's edge may
    # lie on either side of it
    assert abs(int(counters[0, 0]) - int(count[0])) <= 1000
    assert int((images[0] - want).abs().sum()) <= 1e-6 * kl.word_count(22)


def test_longest_words_on_the_fp64_path(kl):
    """24 letters, mixed, every prefix far from the window (FP64 words): 5.9e9
    fallback units of 64 points would overflow the 32-bit unit count."""
    p = kl.params_init(2.1 + 0.01j, 2.3, 24, 64, 64, (1e9, 1e9 + 1.0, 0.0, 1.0), kl.MIXED)
    image, counters = kl.render(p)
    assert int(counters[2]) == int(counters[1]) == kl.word_count(24)
    assert int(counters[0]) == 0 and not bool(image.any())
