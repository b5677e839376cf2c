"""The work that users of this library have it do, as cases that can be timed and checked.

A case is one call, or the few calls that belong together, through the public entry points:
the time stepper of every scheme at the sizes of the paper's workloads and of the tests, the
batched ensemble, the adjoint through torch.autograd, the diagnostics, and the whole path from
a host field and back.  Inputs are made on the GPU from a seed: Taylor-Green fields with a
small solenoidal perturbation, or random solenoidal fields with a developed spectrum.

`exact` gives what a pass returns in 64 bits, from plain torch operations on complex128 half
spectra [3, kz, ky, kx] (kx = 0 .. N/2 - 1), following the equations of the paper.
"""
import ctypes
import math

import torch

from paper_2603_08892_gb300 import autograd
from paper_2603_08892_gb300 import binding as ns

SCHEMES = {"rk2": ns.RK2, "rk4": ns.RK4, "exact": ns.RK2_PS_EXACT, "approx": ns.RK2_PS_APPROX,
           "random": ns.RK2_PS_RANDOM}
TRUNC = {"spherical": ns.TRUNC_SPHERICAL, "cubic": ns.TRUNC_CUBIC, "noalias": ns.TRUNC_NO_DOUBLE_ALIAS}
PREC = {"fp32": ns.FP32, "fp64": ns.FP64}
EVALS = {"rk2": 2, "rk4": 4, "exact": 4, "approx": 2, "random": 2}


def _step(name, N, scheme, prec, steps, kmax, trunc="spherical", flow="tgv", forced=False, how="step"):
    case = {"kind": "step", "how": how, "N": N, "scheme": scheme, "prec": prec, "steps": steps,
            "kmax": kmax, "trunc": trunc, "flow": flow, "forced": forced}
    return dict(case, name=name) if name else case


def listed():
    return [
        # the smallest workload of the paper's kind: a 32^3 Taylor-Green run in FP64 with the exact
        # scheme, energy and dissipation recorded after every step
        _step("tgv32_exact_fp64_diag", 32, "exact", "fp64", 20, 2 * math.sqrt(2) / 3 * 16, how="diag"),
        # one nonlinear term on the caller's own device buffers, inside a loop that must not allocate
        {"name": "nonlinear48_noalloc", "kind": "noalloc", "N": 48, "kmax": 24.0, "trunc": "spherical"},
        # the flagship: Rogallo's random phase shifts at 256^3, spherical truncation at C_t = 1
        _step("tgv256_random_fp32", 256, "random", "fp32", 4, 128.0),
        # its baseline at the same kmax: RK4 with the 2/3 truncation
        _step("tgv384_rk4_fp32", 384, "rk4", "fp32", 2, 128.0),
        # forced isotropic turbulence, the largest workload that runs the phase-shifted scheme
        _step("hit512_split_fp32", 512, "random", "fp32", 2, 256.0, flow="hit", forced=True),
        # the accuracy study at kmax = 108: a grid that is no power of two, no double aliases
        _step("tgv216_random_noalias_fp32", 216, "random", "fp32", 4, 108.0, trunc="noalias"),
        # a production run with the adaptive time step, on the cubic truncation
        _step("hit192_cfl_approx_cubic_fp32", 192, "approx", "fp32", 8, 80.0, trunc="cubic", flow="hit", how="cfl"),
        # double precision at a size where it is used for verification, plain RK2
        _step("hit128_rk2_fp64", 128, "rk2", "fp64", 4, 2.0 / 3 * 64, flow="hit"),
        # an ensemble of uneven members advanced together
        {"name": "ensemble64_fp32", "kind": "batch", "sizes": "32,64,96,128", "each": 16, "prec": "fp32",
         "scheme": "random", "steps": 10},
        # the gradient of a loss of u(T) with respect to u(0), through the steps of a forced flow
        {"name": "adjoint64_forced_fp32", "kind": "vjp", "N": 64, "prec": "fp32", "steps": 20, "ckpt": 10,
         "kmax": 32.0, "forced": True},
        # what is looked at between stretches of a run: energy, spectra, flux of the exact term
        {"name": "diagnostics256_fp32", "kind": "flux", "N": 256, "prec": "fp32", "kmax": 128.0, "shifts": 2},
        # from a field in host memory through ten steps to a field in host memory
        {"name": "host_to_host256_fp32", "kind": "e2e", "N": 256, "prec": "fp32", "scheme": "random",
         "steps": 10, "kmax": 128.0},
    ]


# grid sizes N = 2^a 3^b that the library takes, up to what a drawn case may cost
SIZES = [24, 32, 36, 48, 54, 64, 72, 96, 108, 128, 144, 162, 192, 216, 256, 288, 324, 384]


def _log_size(rng, lo, hi, sizes=SIZES):
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(sizes, key=lambda n: abs(math.log(n / x)))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "batch", "vjp", "flux", "e2e", "noalloc"])
    if kind == "noalloc":
        N = rng.choice([24, 32, 36, 48, 54, 64])
        return {"kind": kind, "N": N, "kmax": round(N / 2 * rng.uniform(0.6, 1.0), 3),
                "trunc": rng.choice(sorted(TRUNC))}
    if kind == "batch":
        sizes = rng.sample([16, 32, 48, 64, 96, 128], rng.randint(1, 4))
        return {"kind": kind, "sizes": ",".join(str(n) for n in sorted(sizes)), "each": rng.randint(1, 16),
                "prec": "fp64" if rng.random() < 0.2 and max(sizes) <= 64 else "fp32",
                "scheme": rng.choice(["random", "approx"]), "steps": rng.randint(2, 10)}
    prec = "fp64" if rng.random() < 0.3 else "fp32"
    if kind == "vjp":
        N = _log_size(rng, 24, 96 if prec == "fp32" else 48)
        return {"kind": kind, "N": N, "prec": prec, "steps": rng.randint(2, 20), "ckpt": rng.randint(2, 10),
                "kmax": round(N / 2 * rng.uniform(0.8, 1.0), 3), "forced": rng.random() < 0.5}
    N = _log_size(rng, 24, 384 if prec == "fp32" else 128)
    kmax = round(N / 2 * rng.choice([2.0 / 3, 2 * math.sqrt(2) / 3, 1.0, rng.uniform(0.6, 1.0)]), 3)
    if kind == "flux":
        return {"kind": kind, "N": N, "prec": prec, "kmax": kmax, "shifts": rng.randint(0, 3)}
    scheme = rng.choice(sorted(SCHEMES))
    steps = rng.randint(1, 3) if N > 200 else rng.randint(2, 8)
    if kind == "e2e":
        return {"kind": kind, "N": min(N, 256), "prec": prec, "scheme": scheme, "steps": steps,
                "kmax": min(kmax, min(N, 256) / 2)}
    return _step(None, N, scheme, prec, steps, kmax, trunc=rng.choice(sorted(TRUNC)),
                 flow=rng.choice(["tgv", "hit"]), forced=rng.random() < 0.3,
                 how=rng.choice(["step", "step", "diag", "cfl"]))


# ---- inputs -----------------------------------------------------------------------------
def _wave(N, device="cuda"):
    k = torch.fft.fftfreq(N, 1.0 / N, device=device, dtype=torch.float64)
    return k[:, None, None], k[None, :, None], k[None, None, : N // 2].abs()


def _solenoidal(N, seed, flow):
    """A random solenoidal field float64 [3, N, N, N] on the GPU, rms 1 per component for a
    developed spectrum ("hit"), or band-limited to |k| <= 4 for a perturbation."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    kz, ky, kx = _wave(N)
    k2 = kz * kz + ky * ky + kx * kx
    S = torch.empty((3, N, N, N // 2), dtype=torch.complex128, device="cuda")
    for c in range(3):
        a = torch.randn((N, N, N), generator=g, device="cuda", dtype=torch.float64)
        S[c] = torch.fft.rfftn(a)[..., : N // 2]
    kd = (kx * S[0] + ky * S[1] + kz * S[2]) / k2.clamp(min=1.0)
    for c, q in enumerate((kx, ky, kz)):
        S[c] -= q * kd
    if flow == "hit":  # E(k) ~ k^4 up to k = 4, k^(-5/3) beyond, a dissipation range near N / 3
        amp = torch.sqrt(k2 / (k2 + 16.0) ** (17.0 / 6)) * torch.exp(-2.0 * torch.sqrt(k2) / (N / 2))
    else:
        amp = (k2 <= 16.0).double()
    amp = amp * (k2 < (N // 2) ** 2) * (k2 > 0)
    u = torch.stack([_inv(S[c] * amp) for c in range(3)])
    return u / torch.sqrt((u * u).mean())


def _field(N, seed, flow):
    if flow == "hit":
        return _solenoidal(N, seed, "hit")
    x = torch.arange(N, device="cuda", dtype=torch.float64) * (2 * math.pi / N)
    cz, cy, cx = torch.cos(x)[:, None, None], torch.cos(x)[None, :, None], torch.cos(x)[None, None, :]
    sy, sx = torch.sin(x)[None, :, None], torch.sin(x)[None, None, :]
    u = torch.stack([sx * cy * cz, -cx * sy * cz, torch.zeros((N, N, N), device="cuda", dtype=torch.float64)])
    return u + 0.01 * 0.5 * _solenoidal(N, seed, "low")


def _nu(case, flow):
    return 1.0 / 1600 if flow == "tgv" else float(case["kmax"]) ** (-4.0 / 3)


def _dt(N, flow):
    # well inside the stability range of RK2 at the grid scale, whatever the truncation, so that a
    # run goes on for as long as it is asked to
    return (0.1 if flow == "tgv" else 0.01) * 2 * math.pi / N


class _Own:
    """A device buffer of the library as a torch tensor, without a copy; it keeps the solver or
    batch that owns the buffer."""

    def __init__(self, ptr, shape, prec, owner):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<c8" if prec == "fp32" else "<c16",
                                         "data": (ptr, False), "version": 3}


def _view(ptr, N, prec, owner):
    return torch.as_tensor(_Own(ptr, (3, N, N, N // 2), prec, owner), device="cuda")


def _solver(case, flow, seed):
    s = ns.Solver(case["N"], _nu(case, flow), case["kmax"], scheme=SCHEMES[case.get("scheme", "random")],
                  truncation=TRUNC[case.get("trunc", "spherical")], precision=PREC[case["prec"]], seed=int(seed))
    if case.get("forced"):
        s.set_forcing(2.0, 3.0, 1.0, 0.5, seed=int(seed))
    return s


def _members(case):
    return [int(n) for n in case["sizes"].split(",") for _ in range(case["each"])]


def _member_view(batch, i, N, prec):
    lib = ctypes.CDLL(ns.LIB_PATH)
    lib.ns_batch_member.restype = ctypes.c_void_p
    lib.ns_batch_member.argtypes = [ctypes.c_void_p, ctypes.c_int]
    lib.ns_device_state.argtypes = [ctypes.c_void_p, ctypes.POINTER(ctypes.c_void_p), ctypes.c_void_p, ctypes.c_void_p]
    p = ctypes.c_void_p()
    lib.ns_device_state(lib.ns_batch_member(batch._h, i), ctypes.byref(p), None, None)
    return _view(p.value, N, prec, batch)


def _shifts(case):
    h = math.pi / case["N"]
    return [[0.0, 0.0, 0.0], [h, h, h], [0.5 * h, 1.5 * h, 0.25 * h]][: case["shifts"]]


def _delta(case, seed):
    dx = 2 * math.pi / case["N"]
    return [dx * _uniform(seed, i) for i in range(3)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        sizes = _members(case)
        b = ns.Batch(sizes, [1.0 / 1600] * len(sizes), [n / 2 for n in sizes],
                     seeds=[1000 * int(seed) + i for i in range(len(sizes))], scheme=SCHEMES[case["scheme"]],
                     precision=PREC[case["prec"]])
        for i, n in enumerate(sizes):
            b.set_velocity(i, _field(n, 1000 * seed + i, "tgv").cpu().numpy())
        return {"kind": kind, "batch": b, "steps": case["steps"], "dts": [_dt(n, "tgv") for n in sizes],
                "views": [_member_view(b, i, n, case["prec"]) for i, n in enumerate(sizes)]}
    N = case["N"]
    if kind == "noalloc":
        S = _project(_fwd(_field(N, seed, "hit")), N, case["kmax"], case["trunc"]).to(torch.complex64).contiguous()
        torch.cuda.synchronize()
        return {"kind": kind, "case": case, "S": S, "out": torch.empty_like(S), "delta": _delta(case, seed)}
    if kind == "vjp":
        u = _field(N, seed, "hit").to(torch.float32 if case["prec"] == "fp32" else torch.float64)
        return {"kind": kind, "case": case, "solver": _solver(case, "hit", seed), "u0": u.requires_grad_(True),
                "target": torch.roll(u.detach(), 1, 1), "dt": _dt(N, "hit")}
    flow = case.get("flow", "hit" if kind == "flux" else "tgv")
    s = _solver(case, flow, seed)
    host = _field(N, seed, flow).cpu()
    st = {"kind": kind, "case": case, "solver": s, "dt": _dt(N, flow)}
    if kind == "e2e":
        st["u"] = host.pin_memory().numpy()
        st["out"] = torch.empty((3, N, N, N), dtype=torch.float64).pin_memory().numpy()
    else:
        s.set_velocity(host.numpy())
        st["view"] = _view(s.device_state()[0], N, case["prec"], s)
    return st


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["batch"].step(state["dts"], state["steps"])
        return state["views"]
    case = state["case"]
    if kind == "noalloc":
        ns.nonlinear_noalloc(state["S"].data_ptr(), state["out"].data_ptr(), case["N"], case["kmax"],
                             state["delta"], truncation=TRUNC[case["trunc"]])
        return state["out"]
    s, dt = state["solver"], state["dt"]
    if kind == "vjp":
        uT = autograd.Trajectory.apply(state["u0"], s, case["steps"], dt, case["ckpt"])
        loss = 0.5 * (uT - state["target"]).square().mean()
        (grad,) = torch.autograd.grad(loss, state["u0"])
        return {"loss": loss.detach(), "uT": uT.detach(), "grad": grad}
    if kind == "flux":
        flux, cum = s.energy_flux(shifts=_shifts(case))
        E, eps = s.energy()
        return {"E": E, "eps": eps, "shell": s.spectrum(ns.SPEC_SHELL), "x": s.spectrum(ns.SPEC_X),
                "flux": flux, "cum": cum}
    if kind == "e2e":
        s.set_velocity(state["u"])
        E, eps = s.step_diag(dt, case["steps"])
        return {"E": E, "eps": eps, "u": s.get_velocity(out=state["out"])}
    if case["how"] == "diag":
        E, eps = s.step_diag(dt, case["steps"])
        return {"E": E, "eps": eps, "state": state["view"]}
    if case["how"] == "cfl":
        s.step_cfl(0.4, 1.0, case["steps"])
        return {"t": s.time()[0], "state": state["view"]}
    s.step(dt, case["steps"])
    return state["view"]


def _work(N, prec, scheme, steps):
    """Each evaluation of the nonlinear term needs the whole state and gives a whole one: the
    state (three half-spectrum fields) is read and written once per evaluation; nine real 3D
    transforms and about 60 operations per grid point."""
    ev = EVALS[scheme] * steps
    C = N ** 3 * (4.0 if prec == "fp32" else 8.0)
    return {"bytes": 6 * C * ev, "flops": (9 * 2.5 * 3 * math.log2(N) + 60.0) * N ** 3 * ev}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        each = [_work(n, case["prec"], case["scheme"], case["steps"]) for n in _members(case)]
        return {q: sum(w[q] for w in each) for q in ("bytes", "flops")}
    N = case["N"]
    prec = case.get("prec", "fp32")
    if kind == "noalloc":
        w = _work(N, prec, "random", 1)
        return {q: w[q] / 2 for q in w}
    if kind == "vjp":  # the steps, their recomputation, and two linearised evaluations for each
        w = _work(N, prec, "random", case["steps"])
        return {q: 4 * w[q] for q in w}
    if kind == "flux":
        w = _work(N, prec, "random", 1)
        n = max(1, case["shifts"])
        return {q: w[q] / 2 * n for q in w}
    w = _work(N, prec, case["scheme"], case["steps"])
    if kind == "e2e":
        w["bytes"] += 48.0 * N ** 3
    return w


# ---- the same in 64 bits, from plain torch ------------------------------------------------
MASK64 = (1 << 64) - 1


def _uniform(seed, n):
    z = (int(seed) + (int(n) + 1) * 0x9E3779B97F4A7C15) & MASK64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & MASK64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & MASK64
    return ((z ^ (z >> 31)) >> 11) * (1.0 / 9007199254740992.0)


def _fwd(u):
    N = u.shape[-1]
    return torch.fft.rfftn(u, dim=(-3, -2, -1))[..., : N // 2] / float(N) ** 3


def _inv(S):
    N = S.shape[-2]
    full = torch.cat([S, torch.zeros(S.shape[:-1] + (1,), dtype=S.dtype, device=S.device)], dim=-1)
    return torch.fft.irfftn(full, s=(N, N, N), dim=(-3, -2, -1)) * float(N) ** 3


def _below(q):
    m = math.floor(q)
    return m - 1 if m == q else m


def _mask(N, kmax, trunc):
    kz, ky, kx = _wave(N)
    if trunc == "cubic":
        m = _below(float(kmax))
        return (kz.abs() <= m) & (ky.abs() <= m) & (kx <= m)
    m = _below(float(kmax) ** 2)
    keep = kz * kz + ky * ky + kx * kx <= m
    if trunc == "noalias":
        ax, ay, az = (N - q.abs() for q in (kx, ky, kz))
        keep = keep & (ax * ax + ay * ay + kz * kz > 4 * m)
        keep = keep & (ax * ax + az * az + ky * ky > 4 * m) & (ay * ay + az * az + kx * kx > 4 * m)
    return keep


def _project(F, N, kmax, trunc):
    kz, ky, kx = _wave(N)
    k2 = kz * kz + ky * ky + kx * kx
    keep = (_mask(N, kmax, trunc) & (k2 > 0)).double()
    kd = (kx * F[0] + ky * F[1] + kz * F[2]) / k2.clamp(min=1.0)
    return torch.stack([(F[c] - q * kd) * keep for c, q in enumerate((kx, ky, kz))])


class _Ref:
    """The schemes of the paper (Sec. 4.1, 4.2, 6.1) on complex128 half spectra."""

    def __init__(self, N, nu, kmax, trunc="spherical", seed=0, forced=False):
        self.N, self.nu, self.kmax, self.trunc, self.seed, self.forced = N, nu, kmax, trunc, int(seed), forced
        self.pats = {}

    def E(self, tau):
        ez, ey, ex = (torch.exp(-self.nu * k * k * tau) for k in _wave(self.N))
        return ez * ey * ex

    def shift(self, d):
        kz, ky, kx = _wave(self.N)
        return torch.exp(1j * kx * d[0]) * torch.exp(1j * ky * d[1]) * torch.exp(1j * kz * d[2])

    def shifted(self, S, d):
        return S if d is None else S * self.shift(d)

    def nl(self, S, d=None):
        kz, ky, kx = _wave(self.N)
        s = self.shifted(S, d)
        u = [_inv(s[c]) for c in range(3)]
        w = [_inv(1j * (ky * s[2] - kz * s[1])), _inv(1j * (kz * s[0] - kx * s[2])), _inv(1j * (kx * s[1] - ky * s[0]))]
        F = torch.stack([_fwd(u[(c + 1) % 3] * w[(c + 2) % 3] - u[(c + 2) % 3] * w[(c + 1) % 3]) for c in range(3)])
        if d is not None:
            F = F * self.shift(d).conj()
        return _project(F, self.N, self.kmax, self.trunc)

    def _pattern(self, j):
        if j not in self.pats:
            N, K, modes = self.N, 3, []
            for kz in range(-K, K + 1):
                for ky in range(-K, K + 1):
                    for kx in range(0, K + 1):
                        k2 = kx * kx + ky * ky + kz * kz
                        if 4 <= k2 <= 9 and kx < N // 2 and (kx > 0 or kz > 0 or (kz == 0 and ky > 0)):
                            modes.append((kx, ky, kz, k2))
            f = torch.zeros((3, N, N, N // 2), dtype=torch.complex128)
            for m, (kx, ky, kz, k2) in enumerate(modes):
                v = []
                for c in range(3):
                    n = (j * len(modes) + m) * 3 + c
                    r = math.sqrt(-2.0 * math.log(1.0 - _uniform(self.seed, 2 * n)))
                    th = 2.0 * math.pi * _uniform(self.seed, 2 * n + 1)
                    v.append(complex(r * math.cos(th), r * math.sin(th)))
                kd = (kx * v[0] + ky * v[1] + kz * v[2]) / k2
                for c, q in enumerate((kx, ky, kz)):
                    p = v[c] - q * kd
                    f[c, kz, ky, kx] = p
                    if kx == 0:
                        f[c, -kz, -ky, 0] = p.conjugate()
            self.pats[j] = f.cuda()
        return self.pats[j]

    def force(self, S, t, dt):
        if not self.forced:
            return 0.0
        x = t / 0.5
        j = math.floor(x)
        f = (1.0 - (x - j)) * self._pattern(j) + (x - j) * self._pattern(j + 1)
        w = torch.full((self.N // 2,), 2.0, dtype=torch.float64, device="cuda")
        w[0] = 1.0
        b = (w * (S.conj() * f).real).sum()
        c = 0.5 * dt * (w * (f.conj() * f).real).sum()
        r = torch.sqrt(b * b + 4.0 * c)
        return 2.0 / torch.where(b >= 0, b + r, b - r) * f

    def alpha(self, scheme, n):
        if scheme != "random":
            return None
        return [2 * math.pi / self.N * _uniform(self.seed, 3 * n + i) for i in range(3)]

    def step(self, S0, scheme, dt, t, n):
        E1, Eh, h = self.E(dt), self.E(0.5 * dt), math.pi / self.N
        if scheme in ("random", "approx"):
            a = self.alpha(scheme, n)
            b = [(a[i] if a else 0.0) + h for i in range(3)]
            N0 = self.nl(S0, a) + self.force(S0, t, dt)
            S1 = (S0 + dt * N0) * E1
            N1 = self.nl(S1, b) + self.force(S1, t + dt, dt)
            return S0 * E1 + 0.5 * dt * Eh * (N0 + N1)
        if scheme in ("rk2", "exact"):
            nl = self.nl if scheme == "rk2" else (lambda S: 0.5 * (self.nl(S) + self.nl(S, [h, h, h])))
            S1 = (S0 + 0.5 * dt * (nl(S0) + self.force(S0, t, dt))) * Eh
            return S0 * E1 + dt * Eh * (nl(S1) + self.force(S1, t + 0.5 * dt, dt))
        k1 = self.nl(S0) + self.force(S0, t, dt)
        acc, S = S0 * E1 + dt / 6 * E1 * k1, (S0 + 0.5 * dt * k1) * Eh
        k2 = self.nl(S) + self.force(S, t + 0.5 * dt, dt)
        acc, S = acc + dt / 3 * Eh * k2, S0 * Eh + 0.5 * dt * k2
        k3 = self.nl(S) + self.force(S, t + 0.5 * dt, dt)
        acc, S = acc + dt / 3 * Eh * k3, S0 * E1 + dt * Eh * k3
        return acc + dt / 6 * (self.nl(S) + self.force(S, t + dt, dt))

    def run(self, S, scheme, dt, steps, cfl=None):
        t, E, eps = 0.0, [], []
        for n in range(steps):
            if cfl:
                s = self.shifted(S, self.alpha(scheme, n))
                f = sum(float(_inv(s[c]).abs().max()) for c in range(3)) * self.N / (2 * math.pi)
                dt = min(1.0, cfl / f)
            S = self.step(S, scheme, dt, t, n)
            t += dt
            if not S.requires_grad:
                e, d = self.energy(S)
                E.append(e)
                eps.append(d)
        return S, t, torch.tensor(E, dtype=torch.float64), torch.tensor(eps, dtype=torch.float64)

    def modes(self, S):
        w = torch.full((self.N // 2,), 2.0, dtype=torch.float64, device="cuda")
        w[0] = 1.0
        return 0.5 * w * (S.real.square() + S.imag.square()).sum(0)

    def energy(self, S):
        kz, ky, kx = _wave(self.N)
        e = self.modes(S)
        return float(e.sum()), float(2 * self.nu * ((kz * kz + ky * ky + kx * kx) * e).sum())


def _bins(idx, w, nbins):
    idx = idx.expand(w.shape).reshape(-1)
    ok = idx < nbins
    return torch.bincount(idx[ok], weights=w.reshape(-1)[ok], minlength=nbins).cpu()


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for i, n in enumerate(_members(case)):
            r = _Ref(n, 1.0 / 1600, n / 2, seed=1000 * int(seed) + i)
            S = _project(_fwd(_field(n, 1000 * seed + i, "tgv")), n, n / 2, "spherical")
            out.append(r.run(S, case["scheme"], _dt(n, "tgv"), case["steps"])[0])
        return out
    N, kmax, trunc = case["N"], case["kmax"], case.get("trunc", "spherical")
    if kind == "noalloc":
        S = _project(_fwd(_field(N, seed, "hit")), N, kmax, trunc).to(torch.complex64).to(torch.complex128)
        return _Ref(N, 0.0, kmax, trunc).nl(S, _delta(case, seed))
    flow = "hit" if kind in ("vjp", "flux") else case.get("flow", "tgv")
    r = _Ref(N, _nu(case, flow), kmax, trunc, seed, bool(case.get("forced")))
    u, dt = _field(N, seed, flow), _dt(N, flow)
    if kind == "vjp":
        if case["prec"] == "fp32":  # the inputs that run is given
            u = u.float().double()
        u.requires_grad_(True)
        uT = _inv(r.run(_project(_fwd(u), N, kmax, trunc), "random", dt, case["steps"])[0])
        loss = 0.5 * (uT - torch.roll(u.detach(), 1, 1)).square().mean()
        (grad,) = torch.autograd.grad(loss, u)
        return {"loss": loss.detach(), "uT": uT.detach(), "grad": grad}
    S = _project(_fwd(u), N, kmax, trunc)
    del u
    if kind == "flux":
        kz, ky, kx = _wave(N)
        k2 = kz * kz + ky * ky + kx * kx
        shell = torch.floor(torch.sqrt(k2) + 0.5).long()
        nb = int(math.ceil(math.sqrt(3) * N / 2)) + 1
        sh = _shifts(case) or [None]
        NL = sum(r.nl(S, d) for d in sh) / len(sh)
        e = r.modes(S)
        w = torch.full((N // 2,), 2.0, dtype=torch.float64, device="cuda")
        w[0] = 1.0
        T = w * (S.conj() * NL).real.sum(0)
        E, eps = r.energy(S)
        return {"E": E, "eps": eps, "shell": _bins(shell, e, N // 2 + 1), "x": _bins(kx.long(), e, N // 2 + 1),
                "flux": -torch.cumsum(_bins(shell, T, nb), 0),
                "cum": torch.cumsum(_bins(shell, 2 * r.nu * k2 * e, nb), 0)}
    S, t, E, eps = r.run(S, case["scheme"], dt, case["steps"], cfl=0.4 if case.get("how") == "cfl" else None)
    if kind == "e2e":
        return {"E": E, "eps": eps, "u": _inv(S)}
    if case["how"] == "diag":
        return {"E": E, "eps": eps, "state": S}
    return {"t": t, "state": S} if case["how"] == "cfl" else S
