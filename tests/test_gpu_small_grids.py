"""Single small grids: the instances that load the state first and give the x rows more threads
(N <= 64), and the FP64 radix-4 plans (N = 16 .. 96), against the FP64 oracle.  Bounds: those of the
parity tests, 2e-5 (FP32) and 1e-12 (FP64) a step."""
import math

import numpy as np
import pytest

from oracle import forcing as fo
from oracle import schemes as sc
from oracle import spectral as osp
from paper_2603_08892_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme", [sc.SCHEME_RK2, sc.SCHEME_RK4, sc.SCHEME_PS_EXACT, sc.SCHEME_PS_APPROX,
                                    sc.SCHEME_PS_RANDOM])
@pytest.mark.parametrize("N,prec", [(8, 1), (12, 0), (16, 1), (24, 0), (48, 0), (64, 0), (48, 1), (64, 1), (96, 1)])
def test_steps_match_oracle(ns, N, prec, scheme):
    code = {sc.SCHEME_RK2: ns.RK2, sc.SCHEME_RK4: ns.RK4, sc.SCHEME_PS_EXACT: ns.RK2_PS_EXACT,
            sc.SCHEME_PS_APPROX: ns.RK2_PS_APPROX, sc.SCHEME_PS_RANDOM: ns.RK2_PS_RANDOM}[scheme]
    nu, kmax, dt, steps = 0.01, 0.9 * N / 2, 0.004, 2
    u = inputs.random_solenoidal(N, N + 1, kcut=N / 2, energy_total=1.0)
    forced = N >= 16 and scheme in (sc.SCHEME_RK4, sc.SCHEME_PS_RANDOM)
    f = fo.Forcing(N, 2.0, 3.0, 0.5, 0.5, seed=4) if forced else None
    da = [0.3 * 2 * math.pi / N] * 3
    ref, _ = sc.run(osp.set_velocity(u, kmax), dt, steps, sc.Problem(N, nu, kmax), scheme, shifts=[da] * steps, forcing=f)
    with ns.Solver(N, nu, kmax, scheme=code, precision=prec) as s:
        if forced:
            s.set_forcing(2.0, 3.0, 0.5, 0.5, seed=4)
        s.set_velocity(u)
        s.set_shifts([da] * steps)
        s.step(dt, steps)
        got = s.get_state()
        s.set_velocity(u)
        s.set_shifts([da] * steps)
        E, eps = s.step_diag(dt, steps)
        assert np.array_equal(s.get_state(), got) or prec
        e, d = s.energy()
    tol = (1e-12 if prec else 2e-5) * steps
    assert np.linalg.norm(got - ref) < tol * np.linalg.norm(ref)
    assert abs(E[-1] / e - 1) < (1e-12 if prec else 1e-5) and abs(eps[-1] / d - 1) < (1e-12 if prec else 1e-5)
