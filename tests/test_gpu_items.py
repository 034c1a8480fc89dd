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
