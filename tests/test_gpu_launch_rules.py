"""Launch shapes of which the caller gives one number, and groups handed out
from the counter over more than three rounds, whose last half round goes out in
half groups."""
import numpy as np
import pytest

import paper_1704_01888_gb300 as pa

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_01888_gb300 import build

    build.build()


def _shape(q, L, R, launch):
    with pa.Population(pa.PAParams(q=q, L=L, R=R, seed=1)) as pop:
        pop.set_launch(*launch)
        return pop.launch_shape()


def test_threads_alone_fill_their_warps_and_passes():
    """At least a warp of site words to a block; whole passes of 512 threads."""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for threads in (256, 512):
        assert _shape(6, 32, 1000, (0, threads))[:2] == (2, threads)  # 16 words per colour
        assert _shape(2, 8, 1000, (0, threads))[:2] == (32, threads)  # one word per colour
        # ten replicas of 64 words would be a pass and a quarter
        assert _shape(10, 64, 40 * sms, (0, threads))[:2] == (8, threads)
    assert _shape(20, 256, 100, (0, 512))[0] == 1


@pytest.mark.parametrize("q,L,rpb,threads", [(10, 32, 6, 32), (3, 16, 20, 32), (2, 8, 40, 32), (20, 48, 5, 64),
                                             (5, 100, 4, 416), (6, 64, 8, 128)])
def test_half_groups_give_the_same_population(q, L, rpb, threads):
    """Sizes that divide into neither the groups nor the halves."""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    betas = np.array([0.0, 0.5, 1.0])

    def run(R, launch):
        with pa.Population(pa.PAParams(q=q, L=L, R=R, seed=2)) as pop:
            pop.set_launch(*launch)
            shape = pop.launch_shape()
            obs, _ = pop.run(betas, 1)
            return shape, [(o["R"], o["sumE"], o["sumE2"], o["sumMt"]) for o in obs], pop.energies(), pop.spins()

    blocks = _shape(q, L, 1000000 // (L * L // 64), (rpb, threads))[2]  # as many as fit the GPU
    assert blocks % sms == 0
    R = 3 * blocks * rpb + blocks * rpb // 3 + 1
    shape, obs, E, spins = run(R, (rpb, threads))
    assert shape == (rpb, threads, blocks) and 3 * blocks * rpb < min(o[0] for o in obs) and R < 16 * blocks * rpb
    other = run(R, (max(1, rpb // 2), 2 * threads))
    assert obs == other[1] and np.array_equal(E, other[2]) and np.array_equal(spins, other[3])


@pytest.mark.parametrize("L,R", [(8, 1), (8, 100000), (16, 1000), (32, 10000), (48, 50000), (64, 1), (64, 151),
                                 (64, 153), (64, 1000), (64, 20000), (64, 100000), (96, 3000), (100, 5003),
                                 (100, 30000), (128, 1000), (192, 3000), (256, 600)])
def test_automatic_shape_is_an_even_share(L, R):
    """A block's replicas are the share of a round of all the blocks that an SM
    holds, for the population with the spread of its copy numbers."""
    import math

    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with pa.Population(pa.PAParams(q=8, L=L, R=R, seed=1)) as pop:
        rpb, threads, blocks = pop.launch_shape()
    planned = R + 2 * math.ceil(math.sqrt(R))
    slots = -(-blocks // sms) * sms
    rounds = -(-planned // (slots * rpb))
    assert rpb == -(-planned // (slots * rounds))
    assert blocks == min(slots, -(-planned // rpb))
    assert threads % 32 == 0 and 32 <= threads <= 1024


@pytest.mark.parametrize("lattices,shape", [((16, 64), (32768, 256)), ((40,), (32768, 256)), ((96, 100), (131072, 1024)),
                                            ((18, 66), (131072, 1024)), ((256,), (65536, 512))])
def test_batch_shape_follows_the_words_that_threads_find(lattices, shape):
    """Few and many of 256 threads without a site word; the runs are lone runs."""
    betas = np.array([0.0, 0.5, 1.0])
    runs = [(pa.PAParams(q=q, L=L, R=300, seed=4, stream=m), betas, 2)
            for m, (q, L) in enumerate((q, L) for L in lattices for q in (3, 10))]
    with pa.Batch(runs) as b:
        assert b.launch_shape()[:2] == shape
        b.run()
        for m, (p, _, _) in enumerate(runs):
            with pa.Population(p) as pop:
                obs, _ = pop.run(betas, 2)
                E, Mt = b.measurements(m)
                assert b.observables(m)[1:] == obs
                assert np.array_equal(E, pop.energies()) and np.array_equal(Mt, pop.occupations())
