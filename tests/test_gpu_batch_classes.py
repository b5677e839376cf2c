"""Every size class of an ensemble, alone and together, under the persistent and the grid schedule: the
block of the persistent launch is that of the widest item present, its items' tiles are wider than the
grid schedule's in the FP32 classes of 96^3 and 128^3, and a tile's width changes no bit."""
import numpy as np
import pytest

from paper_2603_08892_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ns,prec", [([16], 0), ([48, 16], 0), ([128, 48], 0), ([96], 0), ([96, 32, 64, 128], 0),
                                     ([96, 16, 48], 1), ([32], 1)])
@pytest.mark.parametrize("ct,steps", [(1.0, 3), (0.6, 1)])
def test_schedules_give_identical_results(ns, Ns, prec, ct, steps):
    us = [inputs.random_solenoidal(N, 300 + N, kcut=N / 2, energy_total=1.0) for N in Ns]
    out = []
    for sched in ((0, 0), (1, 0), (4, 1)):
        with ns.Batch(Ns, [0.01] * len(Ns), [ct * N / 2 for N in Ns], seeds=list(range(len(Ns))), precision=prec) as b:
            b.set_schedule(*sched)
            for i, u in enumerate(us):
                b.set_velocity(i, u)
            b.step([0.004] * len(Ns), steps)
            out.append([b.get_state(i) for i in range(len(Ns))])
    for o in out[1:]:
        for a, c in zip(out[0], o):
            assert np.array_equal(a, c)
