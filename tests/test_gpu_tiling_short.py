"""The short words of a tiling render have the same FP64 value, bit for bit,
wherever they are evaluated: from their seed, as a walk's first or second letter,
or as strings of the scan.  The image of every depth up to 9 is the sum of the
scans of its lengths, also where words lie on pixel edges (symmetric views)."""
import pytest

import klsynth
from conftest import golden_table
from test_gpu_fsa import kl  # noqa: F401

pytestmark = pytest.mark.gpu

GROUPS = [klsynth.GASKET, klsynth.NEAR_CUSP, klsynth.FUCHSIAN]


@pytest.mark.parametrize("group", GROUPS + ["maskit"])
@pytest.mark.parametrize("window,W,H", [((-1.5, 1.5, -1.5, 1.5), 1024, 1024),
                                        ((-2.0, 2.0, -2.0, 2.0), 4096, 4096),
                                        ((-1.0, 3.0, -0.08, 1.92), 700, 500)])
def test_short_lengths_are_the_scans(kl, group, window, W, H):  # noqa: F811
    import torch
    table = golden_table("t11_indexed_cayley.txt")

    def make(d, mode, accumulate=0):
        if group == "maskit":
            p = kl.params_group(*kl.maskit(-0.097 + 1.838j), d, W, H, window, kl.FP64)
        else:
            p = kl.params_init(group.ta, group.tb, d, W, H, window, kl.FP64)
        p.mode, p.accumulate = mode, accumulate
        return p

    image = torch.empty((H, W), dtype=torch.int32, device="cuda")
    counters = torch.zeros(kl.KL_N_COUNTERS, dtype=torch.int64, device="cuda")
    for d in range(1, 10):
        p = make(d, kl.LIMIT_SET, int(d > 1))
        kl.render_fsa(kl.fsa_from_params(table, p), p, image, counters)
        tiling, words = kl.render(make(d, kl.TILING))
        assert torch.equal(tiling, image), d
        assert torch.equal(words[:2], counters[:2])
