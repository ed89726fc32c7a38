"""A block of the sweep that gives up its wait for the bulk copies: the call
reports PA_ERR_TIMEOUT, the context (of a batch, every run of the launch) has
failed, and the GPU serves the next context.  The checked build counts the
wait of the groups that PA_CHECKED_GIVE_UP names by their first slot (plus one)
as run out; the copies themselves arrive, so nothing hangs or faults."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import os
import numpy as np
import oracle
import paper_1704_01888_gb300 as pa

oracle.build()
betas = np.linspace(0.0, 0.8, 5)


def status(call):
    try:
        call()
    except pa.PAError as e:
        return e.status
    return 0


def runs():
    return [(pa.PAParams(q=q, L=L, R=3000, seed=6, stream=m), betas, 2)
            for m, (q, L) in enumerate(((5, 32), (10, 64), (20, 32), (3, 48)))]


def expect(whole):
    out = oracle.run(5, 32, 3000, 6, 2, betas, want_state=False)
    assert [o["sumE"] for o in whole] == list(out["sumE"]), (whole, out["sumE"])


for slot in (0, 1000, 2000):
    os.environ.pop("PA_CHECKED_GIVE_UP", None)
    with pa.Population(runs()[0][0]) as pop:
        pop.set_launch(2, 1024)  # the throughput kernel, on every SM
        pop.run(betas[:3], 2)
        os.environ["PA_CHECKED_GIVE_UP"] = str(slot + 1)
        pop.resample(0.1)
        pop.sweep(0.3, 2)
        assert status(pop.observables) == pa.PA_ERR_TIMEOUT
        assert status(pop.energies) == pa.PA_ERR_TIMEOUT
        assert status(lambda: pop.resample(0.1)) == pa.PA_ERR_STATE
    os.environ.pop("PA_CHECKED_GIVE_UP")
    with pa.Population(runs()[0][0]) as pop:
        pop.run(betas, 2)
        expect(pop.history(5))
for graph in (False, True):
    with pa.Batch(runs()) as b:
        os.environ["PA_CHECKED_GIVE_UP"] = "1"  # a group of every run starts at slot 0
        assert status(lambda: b.run(use_graph=graph)) == pa.PA_ERR_TIMEOUT
        assert [b.status(m) for m in range(4)] == [pa.PA_ERR_TIMEOUT] * 4
    os.environ.pop("PA_CHECKED_GIVE_UP")
with pa.Batch(runs()) as b:
    b.run()
    expect(b.observables(0))
print("ok")
"""


def test_a_block_that_gives_up_fails_its_runs_alone():
    from paper_1704_01888_gb300 import build

    env = dict(os.environ, PA_LIBRARY=build.build(checked=True), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
