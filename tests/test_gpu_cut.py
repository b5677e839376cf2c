"""States with modes outside the truncation, and states written through the device address.

The compile-time kernels leave out the columns (kx, ky) outside the truncation when the state
vanishes there.  A state that does not (ns_set_state truncates nothing, and a caller may write
through ns_device_state) takes the full passes: one step equals the FP64 oracle's on the same
state, for every scheme, truncation kind and C_t, at sizes with both kinds of last stage (24, 48:
radix 3; 32: radix 4) and with the forcing block reaching beyond the truncation.  The tolerance is
the parity tests': u = 1.1e-16 times log2 N^3 stages times the cancellation of the projection,
below 1e-12.
"""
import math

import numpy as np
import pytest

from oracle import forcing as fo
from oracle import schemes as sc
from oracle import spectral as sp
from paper_2603_08892_gb300 import inputs

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _full_state(N, seed):
    """Solenoidal state with energy in every stored mode (Nyquist rows aside)."""
    return sp.project(sp.forward(inputs.random_solenoidal(N, seed, kcut=2 * N, energy_total=1.0)))


@pytest.mark.parametrize("N,code,kind,ct,forced", [
    (24, 4, 0, 0.6, False), (32, 4, 0, 0.7, False), (48, 3, 1, 0.5, False), (32, 0, 1, 0.6, False),
    (24, 1, 0, 0.5, False), (32, 2, 2, 0.9, False), (64, 4, 2, 0.97, False), (24, 4, 0, 0.3, True),
    (32, 0, 0, 0.25, True), (96, 4, 0, 2 / 3, False)])
@pytest.mark.parametrize("inside", [False, True])
def test_step_from_untruncated_state(ns, N, code, kind, ct, forced, inside):
    kmax, nu, dt = ct * N / 2, 0.01, 0.01
    S = _full_state(N, N + code)
    if inside:
        S = S * sp.truncation_mask(N, kmax, kind)
    da = [0.3 * 2 * math.pi / N, 0.6 * 2 * math.pi / N, 0.1 * 2 * math.pi / N]
    f = fo.Forcing(N, 2.0, 3.0, 0.5, 0.5, seed=3) if forced else None
    prob = sc.Problem(N, nu, kmax, kind)
    ref, t = S, 0.0
    for _ in range(2):
        ref, t = sc.run(ref, dt, 1, prob, code, shifts=[da], forcing=f, t0=t)
    with ns.Solver(N, nu, kmax, scheme=code, truncation=kind, precision=ns.FP64) as s:
        if forced:
            s.set_forcing(2.0, 3.0, 0.5, 0.5, seed=3)
        s.set_state(S)
        s.set_shifts([da, da])
        s.step(dt, 2)
        assert rel(s.get_state(), ref) < 1e-12
        # and once more after the state was read (the next pass starts from the state again)
        E, eps = s.step_diag(dt, 1)
        assert np.isfinite(E[0]) and np.isfinite(eps[0])


@pytest.mark.parametrize("N", [32, 48])
def test_state_written_through_the_device_address(ns, N):
    import torch

    kmax, nu, dt = 0.6 * N / 2, 0.01, 0.01
    S = _full_state(N, 5)
    with ns.Solver(N, nu, kmax, precision=ns.FP64, seed=1) as a, \
            ns.Solver(N, nu, kmax, precision=ns.FP64, seed=1) as b:
        a.set_velocity(inputs.taylor_green(N))  # truncated
        a.step(dt, 1)
        ptr, _, _ = a.device_state()

        class Own:
            __cuda_array_interface__ = {"shape": (3, N, N, N // 2), "typestr": "<c16", "data": (ptr, False), "version": 3}

        view = torch.as_tensor(Own(), device="cuda")
        torch.cuda.synchronize()
        view.copy_(torch.from_numpy(S))
        torch.cuda.synchronize()
        b.set_state(S)
        for s in (a, b):
            s.set_time(0.0, 7)  # another step: its first input is formed from the state
            s.step(dt, 2)
        assert np.array_equal(a.get_state(), b.get_state())
        # back to a truncated state, by the address again
        T = S * sp.truncation_mask(N, kmax)
        view.copy_(torch.from_numpy(T))
        torch.cuda.synchronize()
        b.set_state(T)
        for s in (a, b):
            s.set_time(0.0, 11)
            s.step(dt, 3)
        assert np.array_equal(a.get_state(), b.get_state())


def test_ensemble_members_with_untruncated_states(ns):
    Ns, nu, dt = [32, 48], 0.01, 0.01
    kmaxs = [0.6 * n / 2 for n in Ns]
    with ns.Batch(Ns, [nu] * 2, kmaxs, seeds=[1, 2], precision=ns.FP64) as b:
        refs = []
        for i, n in enumerate(Ns):
            S = _full_state(n, 9 + i) if i == 0 else _full_state(n, 9 + i) * sp.truncation_mask(n, kmaxs[i])
            from paper_2603_08892_gb300 import binding as raw
            h = raw._batch_member(b._h, i)
            c = np.ascontiguousarray(S)
            assert raw._set_state(h, c.ctypes.data_as(raw._dp)) == 0
            refs.append(sc.run(S, dt, 2, sc.Problem(n, nu, kmaxs[i]), sc.SCHEME_PS_RANDOM, seed=1 + i)[0])
        b.step([dt] * 2, 2)
        for i in range(2):
            assert rel(b.get_state(i), refs[i]) < 1e-12
