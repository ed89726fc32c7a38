"""A resampling step whose new population exceeds the capacity, at capacities
on both sides of every change of the scatter's launch: one cluster with one
and with two chunks of replicas to a block (2048, 4096), blocks of 128 and of
256 replicas.  The step is refused as a whole: nothing is written to the parent
map or behind it, and the population, its histogram and its sums stay."""
import numpy as np
import pytest

import oracle
import paper_1704_01888_gb300 as pa

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_01888_gb300 import build

    build.build()
    oracle.build()


@pytest.mark.parametrize("mode", [pa.RESAMPLE_NEAREST_INT, pa.RESAMPLE_POISSON])
@pytest.mark.parametrize("cap", [2048, 2049, 3000, 4095, 4096, 4097, 131073])
def test_refused_step_writes_no_parents(cap, mode):
    import torch

    R, L, guard = cap, 32, 4096
    E = np.random.default_rng(cap).integers(-1500, -900, size=R).astype(np.int32)
    E_dev = torch.tensor(E, device="cuda")
    lnq = torch.zeros(1, dtype=torch.float64, device="cuda")
    size = torch.zeros(1, dtype=torch.int32, device="cuda")
    parent = torch.full((cap + guard,), -7, dtype=torch.int32, device="cuda")
    s = torch.cuda.current_stream().cuda_stream

    def call(R_target, step):
        size.fill_(99)
        lnq.fill_(99.0)
        pa.resample_noalloc(E_dev.data_ptr(), R, L, 0.01, R_target, mode, step, 11, parent.data_ptr(), cap,
                            lnq.data_ptr(), size.data_ptr(), s)
        return size.item()

    for step in range(1, 101):
        assert call(2 * R, step) == -pa.PA_ERR_CAPACITY and lnq.item() == 0.0
    assert bool((parent == -7).all())
    # the working memory serves the next call: a step that fits
    r, ref, R_new, _ = oracle.copy_numbers(E, 0.01, R // 2, mode, 200, 11)
    assert call(R // 2, 200) == R_new and lnq.item() == pytest.approx(ref, rel=1e-12, abs=1e-12)
    assert np.array_equal(parent[:R_new].cpu().numpy(), oracle.parents(r))
    assert bool((parent[cap:] == -7).all())


@pytest.mark.parametrize("R", [2049, 3000, 4096, 4500])
def test_refused_step_keeps_the_population(R):
    """R_cap = R: about every second step is refused (which ones, the oracle
    says); the population then goes on where it stood."""
    with pa.Population(pa.PAParams(q=4, L=8, R=R, seed=8, R_cap=R, track_families=True)) as pop:
        E, refused, beta = pop.energies(), 0, 0.0
        for step in range(1, 41):
            r, ref, R_new, _ = oracle.copy_numbers(E, 0.02, R, pa.RESAMPLE_NEAREST_INT, step, 8)
            if R_new <= R:
                lnq, got = pop.resample(0.02, step, sync=True)
                assert got == R_new and lnq == pytest.approx(ref, rel=1e-12, abs=1e-12)
                assert np.array_equal(pop.parents(R_new), oracle.parents(r))
                beta += 0.02
                pop.sweep(beta, 1, step)
                E = pop.energies()
                continue
            refused += 1
            before, hist = pop.observables(with_hist=True)
            spins, fam = pop.spins(), pop.ancestors()
            with pytest.raises(pa.PAError) as e:
                pop.resample(0.02, step, sync=True)
            assert e.value.status == pa.PA_ERR_CAPACITY
            after, hist2 = pop.observables(with_hist=True)
            assert after == before and np.array_equal(hist, hist2) and hist2.sum() == E.size
            assert np.array_equal(pop.spins(), spins) and np.array_equal(pop.ancestors(), fam)
            assert np.array_equal(pop.energies(), E)
        assert 5 <= refused <= 39


def test_refused_run_of_a_batch_leaves_the_others():
    """One run of a batch outgrows its capacity; the others give what they
    give without it."""
    betas = np.linspace(0.0, 1.2, 13)
    good = [(pa.PAParams(q=5, L=16, R=1500, seed=3, stream=m), betas, 2) for m in (0, 1)]
    tight = (pa.PAParams(q=6, L=16, R=3000, R_cap=3000, seed=3, stream=7), betas, 2)
    with pa.Batch(good) as b:
        b.run()
        ref = [(b.observables(m), b.measurements(m)) for m in (0, 1)]
    with pa.Batch([good[0], tight, good[1]]) as b:
        with pytest.raises(pa.PAError) as e:
            b.run()
        assert e.value.status == pa.PA_ERR_CAPACITY
        assert [b.status(m) for m in range(3)] == [0, pa.PA_ERR_CAPACITY, 0]
        for m, (obs, meas) in zip((0, 2), ref):
            assert b.observables(m) == obs
            assert all(np.array_equal(x, y) for x, y in zip(b.measurements(m), meas))
