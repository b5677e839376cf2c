"""The exact scheme (two fields per pencil tile) in FP32 on the grids whose energy sums are grouped
through shared memory (N = 24, 48), with and without those sums.

Two passes over the same tiles of shared memory follow each other there; the results must not depend
on how the warps of a block interleave: every run gives the same bits, the recorded one too, and they
are the FP64 oracle's within the FP32 bound of the parity tests (2e-5 a step).
"""
import math

import numpy as np
import pytest

from oracle import diagnostics as dg
from oracle import schemes as sc
from oracle import spectral as osp
from paper_2603_08892_gb300 import inputs

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("N", [24, 48])
def test_exact_scheme_fp32(ns, N):
    nu, kmax, dt, steps = 0.01, 2 * math.sqrt(2) / 3 * N / 2, 0.005, 4
    u = inputs.random_solenoidal(N, 7, kcut=N / 3, energy_total=1.0)
    prob = sc.Problem(N, nu, kmax)
    S0 = osp.set_velocity(u, kmax)
    ref = sc.run(S0, dt, steps, prob, sc.SCHEME_PS_EXACT)[0]
    with ns.Solver(N, nu, kmax, scheme=ns.RK2_PS_EXACT, precision=ns.FP32) as s:
        def run(go):
            s.set_velocity(u)
            s.set_time(0.0, 0)
            out = go()
            return s.get_state(), out

        first, _ = run(lambda: s.step(dt, steps))
        assert rel(first, ref) < 2e-5 * steps
        for _ in range(20):
            assert np.array_equal(run(lambda: s.step(dt, steps))[0], first)
        got, (E, eps) = run(lambda: s.step_diag(dt, steps))
        assert np.array_equal(got, first)
        assert abs(E[-1] / dg.energy(ref) - 1) < 1e-4 and abs(eps[-1] / dg.dissipation(ref, nu) - 1) < 1e-4

        got, _ = run(lambda: s.step_cfl(0.3, 1.0, steps))
        want, t, _ = sc.run_cfl(S0, 0.3, 1.0, steps, prob, sc.SCHEME_PS_EXACT)
        assert rel(got, want) < 2e-5 * steps and abs(s.time()[0] / t - 1) < 1e-6
        assert np.array_equal(run(lambda: s.step_cfl(0.3, 1.0, steps))[0], got)
