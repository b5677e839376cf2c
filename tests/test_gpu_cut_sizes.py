"""Column skipping where it is used (from 5 MB of state on), FP32 as well as FP64.

The state is looked at only where something may have written it, once per look; and steps of states
with modes outside the truncation, among them states written through the device address between two
calls (the next call's first evaluation then reads fields formed from the old state, under the old
state's flag), agree with the run-time kernels, which leave no column out: within the parity bounds
of the two (FP32 2e-5 a step, FP64 1e-12).  Recorded energies are those of the resulting state.
"""
import numpy as np
import pytest

from oracle import spectral as sp
from paper_2603_08892_gb300 import inputs

pytestmark = pytest.mark.gpu

MODES = {"default": {}, "tiles": {"NS_TILE_VARIANT": "11"},
         "pipeline": {"NS_SLAB_PIPE": "1", "NS_PIPE_RING": "16"},
         "two_streams": {"NS_SLAB_STREAMS": "2", "NS_SLAB_PLANES": "24"}}


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def view(s, N, prec):
    import torch

    ptr, _, _ = s.device_state()

    class Own:
        __cuda_array_interface__ = {"shape": (3, N, N, N // 2), "typestr": "<c16" if prec else "<c8",
                                    "data": (ptr, False), "version": 3}

    return torch.as_tensor(Own(), device="cuda")


@pytest.mark.parametrize("N,expected", [(128, (0, 0, 0, 0, 0, 1, 0, 1, 1)), (64, (0,) * 9), (72, (0,) * 9)])
def test_looks_at_the_state(ns, monkeypatch, N, expected):
    from torch.profiler import ProfilerActivity, profile

    import torch

    monkeypatch.setenv("NS_AUTOTUNE", "0")
    kmax, dt = N / 3, 1e-3
    u = inputs.taylor_green(N)
    with ns.Solver(N, 0.01, kmax, precision=ns.FP32, seed=1) as s:
        S = sp.set_velocity(u, kmax)
        before = [lambda: s.set_velocity(u), s.get_velocity, lambda: s.nonlinear([0.1, 0.2, 0.3]),
                  lambda: s.set_shifts([[0.1] * 3] * 2), s.energy_flux, lambda: s.set_state(S), s.energy, s.device_state,
                  lambda: None]
        s.set_velocity(u)
        torch.zeros(1, device="cuda")
        with profile(activities=[ProfilerActivity.CUDA]):  # (the first use of the profiler starts it)
            s.step(dt, 1)
            torch.cuda.synchronize()
        got = []
        for f in before:
            f()
            with profile(activities=[ProfilerActivity.CUDA]) as p:
                s.step(dt, 2)
                s.energy()
                torch.cuda.synchronize()
            names = [e.name for e in p.events()]
            assert any("k_energy" in n for n in names)  # (the library's kernels are recorded)
            got.append(sum("k_cut" in n for n in names))
    assert tuple(got) == expected


@pytest.mark.parametrize("N,prec,scheme,kind,ct,mode", [
    (128, 0, 1, 1, 2 / 3, "default"), (128, 0, 2, 0, 0.8, "default"), (96, 1, 4, 0, 2 / 3, "default"),
    (96, 1, 2, 1, 0.6, "default")] + [(128, 0, 4, 0, 2 / 3, m) for m in MODES])
def test_states_written_between_calls(ns, monkeypatch, N, prec, scheme, kind, ct, mode):
    import torch

    kmax, nu, dt = ct * N / 2, 0.01, 0.002
    full = sp.project(sp.forward(inputs.random_solenoidal(N, 5, kcut=2 * N, energy_total=1.0)))
    cut = sp.project(sp.forward(inputs.random_solenoidal(N, 6, kcut=N / 3, energy_total=1.0))) * sp.truncation_mask(N, kmax, kind)
    monkeypatch.setenv("NS_AUTOTUNE", "0")
    monkeypatch.setenv("NS_SLAB_CLUSTER", "0")
    for k, v in MODES[mode].items():
        monkeypatch.setenv(k, v)
    dev = torch.complex128 if prec else torch.complex64

    def go(generic):
        if generic:
            monkeypatch.setenv("NS_GENERIC_KERNELS", "1")
        else:
            monkeypatch.delenv("NS_GENERIC_KERNELS", raising=False)
        out = []
        with ns.Solver(N, nu, kmax, scheme=scheme, truncation=kind, precision=prec, seed=2) as s:
            s.set_state(full)
            for S, steps in ((None, 1), (cut, 1), (full, 2), (cut, 3), (None, 1)):
                if S is not None:  # written behind the library's back: the step counter goes on
                    view(s, N, prec).copy_(torch.from_numpy(S).to(dev))
                    torch.cuda.synchronize()
                E, eps = s.step_diag(dt, steps)
                e, d = s.energy()
                assert abs(E[-1] / e - 1) < 1e-5 and abs(eps[-1] / d - 1) < 1e-5
                out.append((s.get_state(), steps))
        return out

    for (a, n), (b, _) in zip(go(False), go(True)):
        assert rel(a, b) < (1e-12 if prec else 2e-5) * n
