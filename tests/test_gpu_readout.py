"""Reading configurations: long readouts take 64 sites per thread, short ones
one, from 2^18 sites on.  A population read at once, in pieces on both sides of
that size and as the oracle draws it are the same bytes, in every layout."""
import numpy as np
import pytest

import oracle
import paper_1704_01888_gb300 as pa

pytestmark = pytest.mark.gpu
SITES = 1 << 18


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_01888_gb300 import build

    build.build()
    oracle.build()


@pytest.mark.parametrize("q", [2, 3, 10, 20, 40, 128])
@pytest.mark.parametrize("L", [8, 16, 32, 64, 192, 256, 18, 48, 100])
def test_readouts_agree_on_both_sides_of_the_threshold(L, q):
    N = L * L
    edge = -(-SITES // N)  # the smallest count that is a long readout
    R = edge + 5
    with pa.Population(pa.PAParams(q=q, L=L, R=R, seed=12)) as pop:
        whole = pop.spins()
        assert np.array_equal(whole, oracle.init_random(q, L, 0, R, 12).reshape(R, L, L))
        for begin, count in ((0, edge), (3, edge), (0, edge - 1), (4, edge - 1), (R - 1, 1), (1, 0)):
            assert np.array_equal(pop.spins(begin, count), whole[begin:begin + count]), (begin, count)
