"""The reweighting sums and the Newton step as one cluster of blocks: sizes at
the edges of the blocks' shares, energies within and beyond the histogram
table, and histograms wider than the blocks keep.

Tolerances: w = exp(-dbeta e) carries the rounding of dbeta e, at most
2^-53 |dbeta e| <= 45 x 1.1e-16 = 5e-15 relative for the spreads used here,
CUDA's exp 1 ulp, and each sum of positive terms a few roundings more: 2e-14
relative covers S and the moments about E_ref.  A central moment is a
difference of such moments and is off by at most 2e-14 of the terms it is the
difference of.
"""
import math
import struct

import numpy as np
import pytest

import oracle
import paper_1704_01888_gb300 as pa

pytestmark = pytest.mark.gpu
REL = 2e-14


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_01888_gb300 import build

    build.build()
    oracle.build()


@pytest.mark.parametrize("R", [1, 2, 31, 513, 1024, 1025, 2049, 16385, 40000])
@pytest.mark.parametrize("spread,dbeta", [(0, 0.01), (40, 0.05), (40, -0.05), (4095, 0.01), (4096, -0.01), (30000, 0.0015)])
def test_forward_against_sums_in_64_bits(R, spread, dbeta):
    import torch
    from paper_1704_01888_gb300 import autograd as ag

    rng = np.random.default_rng(R + spread)
    E = (-70000 + rng.integers(-spread, spread + 1, size=R)).astype(np.int32)
    if R > 2:
        E[:2] = -70000 - spread, -70000 + spread  # 2 spread + 1 bins: 8191 fit the table, 8193 do not
    O = rng.normal(0.5, 0.1, size=R)
    d = torch.tensor(dbeta, dtype=torch.float64, device="cuda")
    out = ag.reweight_forward(torch.tensor(E, device="cuda"), d, torch.tensor(O, device="cuda")).cpu().numpy()
    alone = ag.reweight_forward(torch.tensor(E, device="cuda"), d).cpu().numpy()
    assert np.array_equal(alone[[0, 1, 2, 5, 6, 7]], out[[0, 1, 2, 5, 6, 7]]) and alone[3] == alone[4] == 0.0
    ref = int(E.min() if dbeta >= 0 else E.max())
    e = E.astype(np.float64) - ref
    w = np.exp(-dbeta * e)
    S = math.fsum(w)
    m1, m2, m3 = (math.fsum(w * e ** k) / S for k in (1, 2, 3))
    mO, mOe = math.fsum(w * O) / S, math.fsum(w * O * e) / S
    assert out[5] == ref and out[6] == pytest.approx(S, rel=REL)
    assert out[0] == pytest.approx(-dbeta * ref + math.log(S / R), rel=REL)
    assert out[1] == pytest.approx(ref + m1, abs=REL * abs(m1) + 1e-16 * abs(ref))
    assert abs(out[2] - (m2 - m1 * m1)) <= 2 * REL * (m2 + m1 * m1)
    absO = math.fsum(w * abs(O)) / S
    assert out[3] == pytest.approx(mO, abs=REL * absO)
    assert abs(out[4] - (mOe - mO * m1)) <= 2 * REL * (math.fsum(w * abs(O * e)) / S + absO * abs(m1))
    assert abs(out[7] - (m3 - 3 * m1 * m2 + 2 * m1 ** 3)) <= 4 * REL * (abs(m3) + 3 * abs(m1) * m2 + 2 * abs(m1) ** 3)


def _fnv1a(data: bytes) -> int:
    h = 1469598103934665603
    for b in data:
        h = ((h ^ b) * 1099511628211) & 0xFFFFFFFFFFFFFFFF
    return h


@pytest.mark.parametrize("ground", [0, 2])
def test_newton_step_over_a_wide_histogram(tmp_path, ground):
    """Random replicas of 256 x 256 beside ground states: 65536 bins between
    them, more than the blocks keep in shared memory (ground = 0: a narrow
    histogram).  The population is placed through a checkpoint."""
    L, R, N = 256, 6, 256 * 256
    path = str(tmp_path / "pop.ckpt")
    with pa.Population(pa.PAParams(q=2, L=L, R=R, seed=5)) as pop:
        pop.save(path)
        E = pop.energies().copy()
    raw = open(path, "rb").read()[:-8]
    at = len(raw) - 4 * (2 * R + 2 * N + 1) - R * N  # header bytes
    spins = np.frombuffer(raw[at:at + R * N], dtype=np.uint8).reshape(R, N).copy()
    spins[:ground] = 0
    E[:ground] = -2 * N
    Mt = np.array([np.bincount(s, minlength=2).max() for s in spins], dtype=np.int32)
    hist = np.bincount(E + 2 * N, minlength=2 * N + 1).astype(np.int32)
    body = raw[:at] + spins.tobytes() + E.astype(np.int32).tobytes() + Mt.tobytes() + hist.tobytes()
    with open(path, "wb") as f:
        f.write(body + struct.pack("<Q", _fnv1a(body)))
    with pa.Population.load(path) as pop:
        for target, cap in ((0.85, 0.05), (0.5, 0.01), (0.9, 1e-5)):
            assert pop.next_dbeta(target, cap) == oracle.newton_dbeta(E, target, cap)
