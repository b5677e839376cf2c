"""The kernels for sizes without compile-time instances, where their stages and tiles change shape.

Odd half lengths (18, 54, 162), tiles of 9 and 12 columns, blocks of one to sixteen rows with the
groups of the forward x rows on halves, the physical fields in and out (c2r, r2c), a nonlinear term
and two steps of the exact scheme (two inputs and two outputs of the pencil) against the FP64 oracle.
The tolerances are those of the parity tests: 1e-12 (FP64) and 2e-5 (FP32) per evaluation or step.
"""
import math

import numpy as np
import pytest

from oracle import nonlinear as onl
from oracle import schemes as sc
from oracle import spectral as osp
from paper_2603_08892_gb300 import inputs

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("prec", [1, 0])
@pytest.mark.parametrize("N", [18, 36, 54, 108, 162])
def test_runtime_size(ns, N, prec):
    tol = 1e-12 if prec else 2e-5
    kmax = N / 2
    u = inputs.random_solenoidal(N, N, kcut=kmax, energy_total=1.0)
    S = osp.set_velocity(u, kmax)
    dx = 2 * math.pi / N
    delta = [0.2 * dx, 0.9 * dx, 0.4 * dx]
    with ns.Solver(N, 0.01, kmax, scheme=2, precision=prec) as s:
        s.set_velocity(u)
        assert rel(s.get_state(), S) < tol
        assert rel(s.get_velocity(), osp.inverse(S)) < tol
        assert rel(s.nonlinear(delta, S), onl.nonlinear(S, delta, kmax)) < tol
        if N <= 108:
            s.set_state(S)
            s.step(0.1 / N, 2)
            ref, _ = sc.run(S, 0.1 / N, 2, sc.Problem(N, 0.01, kmax), sc.SCHEME_PS_EXACT)
            assert rel(s.get_state(), ref) < 2 * tol
