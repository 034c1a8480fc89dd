"""The tree walk of the scan (kl_render_fsa) where its subtrees are uneven:
states with no, one and many symbols, words shorter and longer than the walked
subtree, against the oracle's scan render."""
import pytest

from test_gpu_fsa import kl, run  # noqa: F401

pytestmark = pytest.mark.gpu

# state 1 is a dead end, state 2 leads everywhere, state 3 only to itself
TABLE = [[0, 1, 2, 3], [0, 0, 0, 0], [0, 1, 2, 3], [0, 0, 0, 3]]
GENS = [[[1.2, 0.3j], [0.2, (1 + 0.06j) / 1.2]], [[0.9, 0.4], [-0.5j, (1 - 0.2j) / 0.9]],
        [[1.0, 0.25 + 0.5j], [0.0, 1.0]]]
SEEDS = [0.31 + 0.17j, -0.43 + 0.29j, 0.12 - 0.61j]


@pytest.mark.parametrize("d", [1, 3, 4, 5, 6, 11])
def test_uneven_subtrees(kl, d):  # noqa: F811
    run(kl, TABLE, GENS, SEEDS, d, (-4.1, 3.9, -3.7, 4.3), 257, 199)
