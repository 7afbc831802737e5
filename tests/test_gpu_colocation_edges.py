"""Co-location sums at the edges of the pair tiles (32 x 64 excitors), of the
128-iteration groups and of the 1024-iteration owner chunks, for one-bit to
sixteen-bit owners and every determinant width: equal to the oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,words,ranks,nu,checks", [
    (2, 1, 1, 0, [1]),
    (31, 2, 2, 0, [1, 31, 32, 33, 64, 127]),
    (33, 3, 3, 3, [127, 128, 129]),
    (64, 4, 300, 1, [5, 128, 256, 300]),
    (65, 5, 32, 5, [1023, 1024, 1025, 1100]),
    (97, 6, 65535, 2, [128, 1024]),
    (129, 3, 7, 63, [40, 200]),
    (40, 2, 5, 64, [3, 130, 131, 132, 133]),
])
def test_colocation_edges(n, words, ranks, nu, checks):
    import paper_1807_03749_gb300 as ccmc

    rng = np.random.default_rng(n + 7 * words)
    dets = rng.integers(0, 1 << 63, size=(n, words), dtype=np.uint64)
    g1, g2 = ccmc.colocation(dets, ranks, nu, checks)
    o1, o2 = oracle.colocation(dets, ranks, nu, checks)
    assert np.array_equal(g1, o1) and np.array_equal(g2, o2)
