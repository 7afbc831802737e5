"""Co-location sums of at most 32 iterations (entries of one word) and of one
more (entries of four), at the edges of the pair tiles, for one-bit to
sixteen-bit owners and every determinant width: equal to the oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,words,ranks,nu", [
    (2, 1, 1, 0), (31, 2, 2, 0), (33, 3, 3, 3), (64, 4, 300, 1), (65, 5, 32, 5), (97, 6, 65535, 2), (129, 3, 7, 63),
    (40, 2, 5, 64),
])
@pytest.mark.parametrize("checks", [[1], [7, 31], [1, 2, 30, 32], [32, 33]])
def test_short_runs(n, words, ranks, nu, checks):
    import paper_1807_03749_gb300 as ccmc

    rng = np.random.default_rng(n + 7 * words)
    dets = rng.integers(0, 1 << 63, size=(n, words), dtype=np.uint64)
    g1, g2 = ccmc.colocation(dets, ranks, nu, checks)
    o1, o2 = oracle.colocation(dets, ranks, nu, checks)
    assert np.array_equal(g1, o1) and np.array_equal(g2, o2)
