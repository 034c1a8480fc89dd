"""The scan's subtrees are as high as the number of roots allows: words and
alphabets on either side of the heights, against the oracle's scan render."""
import cmath

import pytest

from test_gpu_fsa import kl, run  # noqa: F401

pytestmark = pytest.mark.gpu


# every string kept: heights 0, 0, 1, 2 with nine letters, 0 .. 4 with three;
# uneven: state 1 is a dead end and state m leads only to itself (heights 1, 2, 3)
@pytest.mark.parametrize("m,d,uneven", [(9, 2, 0), (9, 5, 0), (9, 6, 0), (9, 7, 0), (3, 8, 0),
                                        (3, 10, 0), (3, 11, 0), (3, 12, 0), (3, 13, 0),
                                        (9, 6, 1), (9, 7, 1), (6, 10, 1)])
def test_heights(kl, m, d, uneven):  # noqa: F811
    table = [list(range(m + 1)) for _ in range(m + 1)]
    if uneven:
        table[1] = [0] * (m + 1)
        table[m] = [0] * m + [m]
    turn = [cmath.exp(2j * cmath.pi * k / m) for k in range(m)]
    # contractions of the disk |z| < 3, poles at |z| = 10
    gens = [[[0.35 * turn[k] ** 2, 1.3 * turn[k]], [0.1 * turn[-k], 1.0]] for k in range(m)]
    seeds = [0.3 * t + 0.1 for t in turn]
    run(kl, table, gens, seeds, d, (-2.1, 1.9, -1.7, 2.3), 257, 199)
