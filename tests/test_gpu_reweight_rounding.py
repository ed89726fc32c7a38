"""Rounding of the reweighting kernels: no more of it than sums in one block and
a division per gradient would have."""
import numpy as np
import pytest

import paper_1704_01888_gb300 as pa  # noqa: F401

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_01888_gb300 import build

    build.build()


def _grad_O(E, dbeta, g):
    import torch
    from paper_1704_01888_gb300 import autograd as ag

    O = torch.zeros(E.size, dtype=torch.float64, device="cuda", requires_grad=True)
    d = torch.tensor(dbeta, dtype=torch.float64, device="cuda")
    ag.reweighted_mean(O, d, torch.tensor(E, device="cuda")).backward(torch.tensor(g, dtype=torch.float64, device="cuda"))
    return O.grad.cpu().numpy()


def test_gradient_is_one_division_and_one_product():
    """n replicas at the lowest energy have w = 1; the others' weights, below
    2^-60 in all, vanish in S = n.  With n = 1024 the division by S only moves
    the exponent, so that run shows the kernel's own w; with n = 1000 and a g
    the gradient is the rounded quotient times g, rounded."""
    dbeta, far = 0.01, np.arange(4600, 6600, dtype=np.int32)  # exp(-46) .. exp(-66)
    e = np.concatenate([np.zeros(1024, dtype=np.int32), far]) - 7000
    w = _grad_O(e, dbeta, 1.0)[1024:] * 1024.0
    assert np.all(w > 0) and w.sum() < 2.0 ** -54 and np.allclose(w, np.exp(-dbeta * far), rtol=1e-14)
    got = _grad_O(np.concatenate([e[:1000], e[1024:]]), dbeta, 0.3)
    assert np.array_equal(got[1000:], 0.3 * (w / 1000.0)) and np.all(got[:1000] == 0.3 * (1.0 / 1000.0))


def _tree(v):
    v = np.concatenate([v, np.zeros(32 - len(v))])
    for o in (16, 8, 4, 2, 1):
        v = v + np.concatenate([v[o:], np.zeros(o)])
    return v[0]


def _one_block(t):
    """1024 threads, each a strided share, then warp trees."""
    pad = np.zeros(-(-len(t) // 1024) * 1024)
    pad[:len(t)] = t
    a = np.zeros(1024)
    for row in pad.reshape(-1, 1024):
        a = a + row
    return _tree(np.array([_tree(a[32 * i:32 * i + 32]) for i in range(32)]))


def test_sums_over_the_cluster_round_no_more_than_in_one_block():
    """Root mean squares over 160 populations of the relative errors of S,
    <O> and cov(O, E), against those of the same sums in one block and the
    differences taken directly.  Both root mean squares scatter by
    1 / sqrt(2 * 160) = 5.6 %, their quotient by 8 %: two of these are allowed."""
    import torch
    from paper_1704_01888_gb300 import autograd as ag

    lib, one = [], []
    for seed in range(160):
        rng = np.random.default_rng(seed)
        R, L = int(np.exp(rng.uniform(np.log(20000), np.log(200000)))), int(rng.choice([32, 64, 128]))
        dbeta = float(rng.uniform(0.001, 0.01))
        E = np.clip(np.round(rng.normal(size=R) * 0.8 * L - 1.2 * L * L), -2 * L * L, 0).astype(np.int32)
        O = 0.5 + 0.1 * rng.normal(size=R)
        out = ag.reweight_forward(torch.tensor(E, device="cuda"), torch.tensor(dbeta, dtype=torch.float64, device="cuda"),
                                  torch.tensor(O, device="cuda")).cpu().numpy()
        e = (E - E.min()).astype(np.float64)
        wl = np.exp(-LD(dbeta) * e.astype(LD))
        S, mO, m1 = wl.sum(), (wl * O).sum() / wl.sum(), (wl * e).sum() / wl.sum()
        cov = (wl * (O - mO) * (e - m1)).sum() / S
        scale = mO * m1  # the covariance is a difference of terms of this size
        w = np.exp(-dbeta * e)
        s = [_one_block(x) for x in (w, w * e, w * O, w * O * e)]
        lib.append([(out[6] - S) / S, (out[3] - mO) / mO, (out[4] - cov) / scale])
        one.append([(s[0] - S) / S, (s[2] / s[0] - mO) / mO, (s[3] / s[0] - (s[2] / s[0]) * (s[1] / s[0]) - cov) / scale])
    lib, one = (np.sqrt((np.array(x, dtype=LD) ** 2).mean(axis=0)) for x in (lib, one))
    assert np.all(lib <= 1.16 * one), (lib, one)


@pytest.mark.parametrize("R,big", [(300, 1e304), (30000, 1e302)])
def test_covariance_of_observables_beyond_the_doubles(R, big):
    """sum w O e above the largest double: infinite, as SOe / S - <O> <e> is; an
    infinite or undefined O leaves no number."""
    import torch
    from paper_1704_01888_gb300 import autograd as ag

    E = np.random.default_rng(R).integers(-9000, -4000, size=R).astype(np.int32)
    E[0] = -9000
    d = torch.tensor(1e-5, dtype=torch.float64, device="cuda")

    def cov(O):
        out = ag.reweight_forward(torch.tensor(E, device="cuda"), d, torch.tensor(O, device="cuda")).cpu().numpy()
        return out[3], out[4]

    mean, c = cov(np.full(R, big))
    assert mean == pytest.approx(big, rel=1e-14) and c == np.inf
    mean, c = cov(np.full(R, -big))
    assert mean == pytest.approx(-big, rel=1e-14) and c == -np.inf
    for bad in (np.inf, np.nan):
        O = np.ones(R)
        O[R // 2] = bad
        mean, c = cov(O)
        assert (mean == bad or np.isnan(bad) and np.isnan(mean)) and np.isnan(c)
