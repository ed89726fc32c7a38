"""The automatic launch shapes and the two sweep kernels they choose between:
small populations run the latency kernel in even shares, larger ones the
throughput kernel.  Every row geometry and plane count gives the bits of the
throughput kernel in a 1024-thread block, at lattices with more and with fewer
site words than a block has threads."""
import numpy as np
import pytest

import paper_1704_01888_gb300 as pa

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_01888_gb300 import build

    build.build()


def _trajectory(q, L, R, launch, fam=False):
    with pa.Population(pa.PAParams(q=q, L=L, R=R, seed=9, track_families=fam)) as pop:
        if launch:
            pop.set_launch(*launch)
        obs, _ = pop.run(np.array([0.0, 0.4, 0.9, 1.3, 1.8]), 2)
        return ([(o["R"], o["sumE"], o["sumE2"], o["sumMt"], o["n_families"]) for o in obs], pop.spins(),
                pop.occupations(), pop.launch_shape())


@pytest.mark.parametrize("q", [2, 3, 8, 10, 20, 40, 128])
@pytest.mark.parametrize("L,R", [(8, 333), (16, 153), (32, 500), (48, 161), (64, 305), (18, 200), (66, 77), (100, 153),
                                 (128, 40), (256, 5)])
def test_latency_and_throughput_kernels_agree(q, L, R):
    ref = _trajectory(q, L, R, None, fam=True)
    for launch in ((3, 1024) if L < 256 else (1, 1024), (1, 32), (2, 416)):
        if launch[0] * L * L * 7 // 8 > 200000:
            continue
        got = _trajectory(q, L, R, launch, fam=True)
        assert got[0] == ref[0], launch
        assert np.array_equal(got[1], ref[1]) and np.array_equal(got[2], ref[2]), launch


@pytest.mark.parametrize("L,R", [(16, 1), (64, 151), (64, 153), (64, 1000), (32, 10000), (100, 5003), (128, 10000)])
def test_automatic_shape_spreads_the_population(L, R):
    """No block of the automatic shape takes more than an even share of a
    round, and no SM more than one block above the others'."""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with pa.Population(pa.PAParams(q=8, L=L, R=R, seed=1)) as pop:
        rpb, threads, blocks = pop.launch_shape()
    assert threads % 32 == 0 and 32 <= threads <= 1024 and rpb >= 1
    if rpb * blocks >= R:  # one round
        assert (rpb - 1) * ((blocks + sms - 1) // sms) * sms < R + 3 * R ** 0.5 + sms * 8
