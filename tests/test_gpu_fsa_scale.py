"""The scan of generators scaled by a power of two: the same maps, and the same
FP64 words bit for bit, so the image is the unscaled one's value for value."""
import pytest

import klsynth
from conftest import golden_table
from test_gpu_fsa import kl  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("power", [-120, -100, -70, -64, -50, -30, 30, 60, 62, 63, 64, 65, 66, 100])
def test_scaled_generators_give_the_same_image(kl, power):  # noqa: F811
    import torch
    table = golden_table("t11_indexed_cayley.txt")
    p = kl.params_init(klsynth.NEAR_CUSP.ta, klsynth.NEAR_CUSP.tb, 9, 400, 300,
                       (-1.51, 1.5, -1.2, 1.313), kl.FP64)
    f = kl.fsa_from_params(table, p)
    want, count = kl.render_fsa(f, p)
    for k in range(32):
        f.gens[k] = f.gens[k] * 2.0 ** power
    image, counters = kl.render_fsa(f, p)
    assert torch.equal(image, want)
    assert torch.equal(counters[:3], count[:3])
