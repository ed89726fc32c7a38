"""Resampling at the edges of its kernels' shares -- blocks of 128 and 256
replicas, the cluster's slices of the energy bins, weights over hundreds of
binades, energies wider than a block's histogram -- against the oracle: copy
numbers (as the parent map) and sizes equal, ln Q within 1e-12 (S is the same
double on both sides; only the logarithm differs)."""
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


@pytest.mark.parametrize("R,dbeta", [(700, 0.4), (5003, 0.05), (5003, 0.4), (5003, 2.0), (20000, 1.2)])
def test_poisson_tables_give_the_oracles_copy_numbers(R, dbeta):
    """pa_resample draws full Poisson pieces (mean 64) from a table: copy
    numbers from one to thousands."""
    cap = 2 * R + 2000
    with pa.Population(pa.PAParams(q=5, L=16, R=R, seed=4, resample_mode=pa.RESAMPLE_POISSON, R_cap=cap)) as pop:
        E = pop.energies()
        lnq, R_new = pop.resample(dbeta, 1, sync=True)
        r, ref_lnq, ref_R, rho = oracle.copy_numbers(E, dbeta, R, pa.RESAMPLE_POISSON, 1, 4)
        assert R_new == ref_R and lnq == pytest.approx(ref_lnq, rel=1e-12, abs=1e-12)
        assert np.array_equal(pop.parents(R_new), oracle.parents(r))
    assert dbeta < 2.0 or rho.max() > 200.0


@pytest.mark.parametrize("R,cap", [(1, 8), (127, 1500), (128, 1500), (129, 1500), (2047, 5000), (2049, 5000),
                                   (5003, 131072), (5003, 131073), (150000, 200000)])
@pytest.mark.parametrize("L,lo,hi,dbeta", [(64, -4300, -4200, 0.01), (64, -8192, 0, -0.01), (256, -131072, 0, 1e-4),
                                           (256, -90000, -20000, 0.01), (256, -131072, -131072, 0.3), (8, -128, 0, 0.05)])
@pytest.mark.parametrize("mode", [pa.RESAMPLE_NEAREST_INT, pa.RESAMPLE_POISSON])
def test_copy_numbers_and_lnq_match_the_oracle(R, cap, L, lo, hi, dbeta, mode):
    import torch

    rng = np.random.default_rng(R + L)
    E = rng.integers(lo, hi + 1, size=R).astype(np.int32)
    r, lnq, R_new, _ = oracle.copy_numbers(E, dbeta, R, mode, 3, 11)
    E_dev = torch.tensor(E, device="cuda")
    parent = torch.full((cap,), -1, dtype=torch.int32, device="cuda")
    lnq_dev = torch.zeros(1, dtype=torch.float64, device="cuda")
    size = torch.zeros(1, dtype=torch.int32, device="cuda")
    pa.resample_noalloc(E_dev.data_ptr(), R, L, dbeta, R, mode, 3, 11, parent.data_ptr(), cap, lnq_dev.data_ptr(),
                        size.data_ptr(), torch.cuda.current_stream().cuda_stream)
    if R_new == 0 or R_new > cap:
        assert size.item() == -pa.PA_ERR_CAPACITY
        return
    assert size.item() == R_new
    assert np.array_equal(parent[:R_new].cpu().numpy(), oracle.parents(r))
    assert lnq_dev.item() == pytest.approx(lnq, rel=1e-12, abs=1e-12)
