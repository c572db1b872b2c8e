"""The work this library is used for, as measurable cases.

Every case goes through the package's public classes (`TDSE`, `Batch`,
`Server`) the way a program that propagates wavefunctions calls them: states
come in, a block of steps runs, states or observables come back.  Sizes follow
the paper's configurations and the batched / served ones built on them
(hydrogen, length gauge unless said, a sin^2 pulse, the cos^(1/8) absorber over
the last 50 a.u. of the larger boxes).

Time steps: `dt` is the step in a.u.; 0 asks for the largest step at which a
Krylov propagator of the case's dimension converges on its grid
(rho(H) dt = m / 2), or the explicit methods are stable.
"""
import math

import numpy as np
import torch

import paper_1308_1856_gb300 as tdse

C_AU = 137.035999084                  # speed of light in atomic units
INTENSITY_AU = 3.50944506e16          # W/cm^2 of a field of 1 a.u.
HARTREE_NM = 45.5633525               # photon energy (a.u.) times wavelength (nm)
ABSORBER_WIDTH = 50.0
PULSE_AT = 0.37                       # fraction of the pulse at which propagation starts


def listed():
    return [
        # The paper's hydrogen run: a small box, explicit steps.  A user's script advances it in
        # blocks of a few steps between plots, so launch latency is the whole cost.
        dict(name="small_taylor8", kind="steps", N=500, dr=0.2, lmax=4, stencil=3, method="taylor", order=8,
             dt=0.01, steps=20, precision="fp64", gauge="length", absorber=False),
        # The same box with the Krylov propagator at the large step it allows.
        dict(name="small_lanczos12", kind="steps", N=500, dr=0.2, lmax=4, stencil=3, method="lanczos", order=12,
             dt=0.05, steps=10, precision="fp64", gauge="length", absorber=False),
        # One application of the Hamiltonian, for a program with its own integrator.
        dict(name="hpsi_scale", kind="hpsi", N=8000, dr=0.05, lmax=63, stencil=5, precision="fp64", gauge="length"),
        # Strong-field box at the paper's precision, explicit method.
        dict(name="scale_taylor12", kind="steps", N=8000, dr=0.05, lmax=63, stencil=5, method="taylor", order=12,
             dt=4e-6, steps=4, precision="fp64", gauge="length", absorber=True),
        # The same box with the Krylov propagator: the usual production run of one pulse.
        dict(name="scale_lanczos12", kind="steps", N=8000, dr=0.05, lmax=63, stencil=5, method="lanczos", order=12,
             dt=0.0, steps=3, precision="fp64", gauge="length", absorber=True),
        # The same run in mixed precision, as a parameter scan would use it.
        dict(name="scale_lanczos12_mixed", kind="steps", N=8000, dr=0.05, lmax=63, stencil=5, method="lanczos",
             order=12, dt=0.0, steps=6, precision="mixed", gauge="length", absorber=True),
        # A ragged medium box in the velocity gauge (the gauge check of a length-gauge result).
        dict(name="velocity_lanczos16", kind="steps", N=4001, dr=0.1, lmax=31, stencil=5, method="lanczos", order=16,
             dt=0.0, steps=4, precision="fp64", gauge="velocity", absorber=True),
        # An embedded Runge-Kutta pair with its error estimate, 3-point stencil, odd sizes.
        dict(name="dormand_prince", kind="rk", N=3001, dr=0.1, lmax=24, stencil=3, tableau="dormand_prince", dt=0.0,
             steps=4, absorber=True),
        # An intensity / wavelength scan: many uneven instances in one batch, states in from and out to the host.
        dict(name="batch_fp64", kind="batch", count=32, nmin=2000, nmax=16000, dr=0.1, lmin=15, lmax=127, mmin=8,
             mmax=16, dt=0.0, steps=4, precision="fp64"),
        # The same scan in mixed precision.
        dict(name="batch_mixed", kind="batch", count=32, nmin=2000, nmax=16000, dr=0.1, lmin=15, lmax=127, mmin=8,
             mmax=16, dt=0.0, steps=8, precision="mixed"),
        # Harmonic spectra and photoelectron flux for several pulses: observables after every step.
        dict(name="batch_hhg", kind="hhg", count=8, nmin=2000, nmax=8000, dr=0.1, lmin=15, lmax=63, mmin=8, mmax=16,
             dt=0.0, steps=8, angles=45),
        # A service that admits requests of different sizes as they come and returns their observables.
        dict(name="served_fp64", kind="served", count=10, nmin=2000, nmax=8000, dr=0.1, lmin=15, lmax=63, mmin=8,
             mmax=16, dt=0.0, steps=10, batch_steps=5),
    ]


def _log_int(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["small", "scale", "scale", "mid", "rk", "hpsi", "imag", "batch", "batch", "hhg", "served"])
    if kind == "small":
        method, order = rng.choice([("taylor", rng.randint(4, 12)), ("rk4", 4), ("lanczos", rng.randint(4, 16))])
        return dict(kind="steps", N=_log_int(rng, 200, 1600), dr=rng.choice([0.1, 0.2]), lmax=rng.randint(0, 8),
                    stencil=rng.choice([3, 5]), method=method, order=order, dt=0.0, steps=rng.randint(4, 20),
                    precision="fp64", gauge="length", absorber=False)
    if kind == "hpsi":
        return dict(kind="hpsi", N=_log_int(rng, 500, 12000), dr=rng.choice([0.05, 0.1, 0.2]), lmax=rng.randint(4, 63),
                    stencil=rng.choice([3, 5, 5]), precision=rng.choice(["fp64", "fp64", "mixed"]),
                    gauge=rng.choice(["length", "length", "velocity"]))
    if kind in ("scale", "mid"):
        method, order = rng.choice([("taylor", rng.randint(6, 12)), ("rk4", 4), ("lanczos", rng.randint(8, 16)),
                                    ("lanczos", 12)])
        N = _log_int(rng, 4000, 10000) if kind == "scale" else _log_int(rng, 1600, 4000)
        return dict(kind="steps", N=N, dr=rng.choice([0.05, 0.1]),
                    lmax=rng.randint(24, 63) if kind == "scale" else rng.randint(7, 31),
                    stencil=rng.choice([3, 5, 5]), method=method, order=order, dt=0.0, steps=rng.randint(2, 5),
                    precision=rng.choice(["fp64", "fp64", "mixed"]),
                    gauge=rng.choice(["length", "length", "length", "velocity"]), absorber=True)
    if kind == "rk":
        return dict(kind="rk", N=_log_int(rng, 1000, 8000), dr=rng.choice([0.1, 0.2]), lmax=rng.randint(4, 47),
                    stencil=rng.choice([3, 5]), dt=0.0, steps=rng.randint(2, 5), absorber=True,
                    tableau=rng.choice(["euler", "classic", "fehlberg", "cash_karp", "dormand_prince", "merson"]))
    if kind == "imag":
        # ground states by relaxation: few partial waves, many steps
        return dict(kind="imag", N=_log_int(rng, 1000, 8000), dr=rng.choice([0.1, 0.2]), lmax=rng.randint(0, 4),
                    stencil=rng.choice([3, 5]), method="lanczos", order=rng.randint(8, 16), dt=0.0,
                    steps=rng.randint(5, 20))
    if kind == "batch":
        precision = rng.choice(["fp64", "mixed"])
        return dict(kind="batch", count=rng.randint(5, 24), nmin=_log_int(rng, 1000, 4000), nmax=rng.randint(6000, 16000),
                    dr=0.1, lmin=rng.randint(7, 31), lmax=rng.randint(48, 127), mmin=8, mmax=16, dt=0.0,
                    steps=rng.randint(2, 5), precision=precision)
    if kind == "hhg":
        return dict(kind="hhg", count=rng.randint(3, 8), nmin=_log_int(rng, 1000, 2000), nmax=rng.randint(4000, 8000),
                    dr=0.1, lmin=7, lmax=rng.randint(20, 63), mmin=8, mmax=16, dt=0.0, steps=rng.randint(4, 8),
                    angles=rng.randint(9, 90))
    return dict(kind="served", count=rng.randint(4, 10), nmin=_log_int(rng, 1000, 2000), nmax=rng.randint(4000, 8000),
                dr=0.1, lmin=7, lmax=rng.randint(20, 63), mmin=8, mmax=16, dt=0.0, steps=rng.randint(5, 10),
                batch_steps=rng.randint(2, 6))


# ---- inputs ---------------------------------------------------------------------
def _radius(N, dr):
    return torch.arange(1, N + 1, dtype=torch.float64, device="cuda") * dr


def _state(N, dr, lmax, gen, noise=0.0):
    """A wavefunction in the middle of a pulse: bound shapes r^(l+1) e^(-r/a) and an outgoing packet in every
    partial wave, the amplitudes falling with l, normalised to dr sum |f|^2 = 1.  noise: grid-scale noise of that
    relative size, without which an embedded pair's error estimate on a stiff grid is only rounding."""
    r = _radius(N, dr)
    l = torch.arange(lmax + 1, dtype=torch.float64, device="cuda")[:, None]
    amp = torch.pow(torch.tensor(0.75, dtype=torch.float64, device="cuda"), l)
    F = torch.zeros(lmax + 1, N, dtype=torch.complex128, device="cuda")

    def coef():
        return torch.complex(*(torch.randn(lmax + 1, 1, dtype=torch.float64, device="cuda", generator=gen)
                               for _ in range(2)))

    for a in (1.0, 2.0, 4.0):
        shape = torch.exp((l + 1) * torch.log(r / (a * (l + 1))) - r / a + (l + 1))   # maximum one, at r = a (l + 1)
        F += coef() * amp * shape
    R = N * dr
    u = torch.rand(lmax + 1, 2, dtype=torch.float64, device="cuda", generator=gen)
    r0, k = R * (0.1 + 0.5 * u[:, :1]), 0.2 + 1.3 * u[:, 1:]
    width = 0.02 * R + 2.0
    F += 0.2 * coef() * amp * torch.exp(-((r - r0) / width) ** 2) * torch.exp(1j * k * r)
    F /= torch.sqrt(dr * (F.abs() ** 2).sum())
    if noise:
        e = torch.complex(*(torch.randn(lmax + 1, N, dtype=torch.float64, device="cuda", generator=gen)
                            for _ in range(2)))
        F += noise * e / torch.sqrt(dr * (e.abs() ** 2).sum())
    return F.contiguous()


def _noise(case):
    return 0.02 if case["kind"] == "rk" else 0.0


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rho(N, dr, lmax, stencil, E0):
    """Gershgorin bound of the spectral radius of H."""
    lap = (64.0 / 24.0 if stencil == 5 else 2.0) / (dr * dr)
    return lap + lmax * (lmax + 1) / (2.0 * dr * dr) + 1.0 / dr + 2.0 * abs(E0) * N * dr


def _step(case, N, lmax, m, E0, stencil):
    if case["dt"] > 0:
        return case["dt"]
    explicit = case["kind"] == "rk" or case.get("method") in ("taylor", "rk4")
    if explicit:
        lim = 0.8 if case.get("tableau") == "euler" else 2.0
        return lim / _rho(N, case["dr"], lmax, stencil, E0)
    return 0.5 * m / _rho(N, case["dr"], lmax, stencil, E0)


def _pulse(seed):
    rng = np.random.default_rng([17, int(seed)])
    return dict(E0=0.0534 * rng.uniform(0.8, 1.2), omega=0.057, ncycles=4.0, cep=rng.uniform(0.0, 1.0))


def _specs(case, seed):
    """Instances of a scan: the grids belong to the case, the pulses to the seed."""
    grid = np.random.default_rng([case["count"], case["nmin"], case["nmax"], case["lmin"], case["lmax"]])
    rng = np.random.default_rng([29, int(seed)])
    out = []
    for _ in range(case["count"]):
        N = int(grid.integers(case["nmin"], case["nmax"] + 1))
        lmax = int(grid.integers(case["lmin"], case["lmax"] + 1))
        m = int(grid.integers(case["mmin"], case["mmax"] + 1))
        nc = int(grid.integers(2, 7))
        E0 = math.sqrt(math.exp(rng.uniform(math.log(1e13), math.log(5e14))) / INTENSITY_AU)
        omega = HARTREE_NM / rng.uniform(400.0, 1600.0)
        out.append(dict(N=N, dr=case["dr"], lmax=lmax, E0=E0, omega=omega, ncycles=float(nc), cep=rng.uniform(0.0, 1.0),
                        krylov=m, dt=_step(case, N, lmax, m, 0.12, 5), absorber_r=N * case["dr"] - ABSORBER_WIDTH,
                        r_b=0.2 * N * case["dr"]))
    return out


def _pulse_start(p):
    return PULSE_AT * 2.0 * math.pi * p["ncycles"] / p["omega"]


def prepare(case, seed):
    torch.cuda.current_device()
    kind = case["kind"]
    if kind in ("batch", "hhg"):
        specs = _specs(case, seed)
        gen = _gen(seed)
        sizes = [s["N"] * (s["lmax"] + 1) for s in specs]
        host = torch.empty(sum(sizes), dtype=torch.complex128, pin_memory=True)
        off = 0
        for s, G in zip(specs, sizes):
            host[off:off + G].copy_(_state(s["N"], s["dr"], s["lmax"], gen).reshape(-1))
            off += G
        st = dict(case=case, specs=specs, inp=host, batch=tdse.Batch(specs, 5, case.get("precision", "fp64")),
                  out=torch.empty(sum(sizes), dtype=torch.complex128, pin_memory=True))
        if kind == "hhg":
            st["cos"] = np.cos(np.linspace(0.0, math.pi, case["angles"]))
        return st
    if kind == "served":
        specs = _specs(case, seed)
        probe = tdse.Server(1 << 26, 1, 5, "fp64")
        budget = sum(probe.instance_bytes(s) + 65536 for s in specs)
        probe.close()
        return dict(case=case, specs=specs, server=tdse.Server(budget, case["count"], 5, "fp64"))
    N, dr, lmax = case["N"], case["dr"], case["lmax"]
    h = tdse.TDSE(N, dr, lmax, case["stencil"])
    absorb = bool(case.get("absorber"))
    h.set_options(absorber=absorb, absorber_r=max(0.5 * N * dr, N * dr - ABSORBER_WIDTH) if absorb else 0.0,
                  precision=case.get("precision", "fp64"), gauge=case.get("gauge", "length"))
    p = _pulse(seed)
    h.set_pulse(p["E0"], p["omega"], p["ncycles"], p["cep"])
    stream = torch.cuda.Stream()
    h.set_stream(stream.cuda_stream)
    x = _state(N, dr, lmax, _gen(seed), _noise(case))
    return dict(case=case, handle=h, stream=stream, x=x, y=torch.empty_like(x), pulse=p,
                dt=None if kind == "hpsi" else _step(case, N, lmax, case.get("order", 4), p["E0"], case["stencil"]))


# ---- one pass -------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        b = state["batch"]
        for i, s in enumerate(state["specs"]):
            b.set_time(i, _pulse_start(s))
        b.propagate_io(state["inp"].data_ptr(), state["out"].data_ptr(), case["steps"])
        return state["out"]
    if kind == "hhg":
        b = state["batch"]
        b.set_states_ptr(state["inp"].data_ptr())
        for i, s in enumerate(state["specs"]):
            b.set_time(i, _pulse_start(s))
        b.record_dipole(case["steps"])
        b.flux_setup(state["cos"])
        b.propagate(case["steps"])
        b.get_states_ptr(state["out"].data_ptr())
        n = len(state["specs"])
        flux = [b.flux(i) for i in range(n)]
        return dict(states=state["out"], series=np.stack([b.dipole_series(i) for i in range(n)]),
                    flux=np.array([[f["flux"], f["yield"]] for f in flux]),
                    density=np.stack([f["density"] for f in flux]), pad=np.stack([f["pad"] for f in flux]))
    if kind == "served":
        srv, specs = state["server"], state["specs"]
        half = len(specs) // 2
        ids = [srv.submit(s, case["steps"]) for s in specs[:half]]
        srv.step(case["batch_steps"])
        ids += [srv.submit(s, case["steps"]) for s in specs[half:]]     # arrive while the first ones run
        done = set()
        while len(done) < len(ids):
            srv.step(case["batch_steps"])
            done.update(srv.poll())
        out = [srv.observables(i) for i in ids]
        final = [srv.get_state(i) for i in ids]
        for i in ids:
            srv.release(i)
        return dict(states=final, values=np.array([[o["norm"], o["dipole"], o["yield"], o["p_ground"]] for o in out]),
                    l_pop=np.concatenate([o["l_pop"] for o in out]))
    h, stream, x, y = state["handle"], state["stream"], state["x"], state["y"]
    here = torch.cuda.current_stream()
    stream.wait_stream(here)
    value = None
    if kind == "hpsi":
        h.apply_h(h.field(_pulse_start(state["pulse"])), x.data_ptr(), y.data_ptr())
    else:
        h.set_state_device(x.data_ptr())
        h.time = _pulse_start(state["pulse"])
        if kind == "steps":
            h.propagate(case["method"], case["order"], state["dt"], case["steps"])
        elif kind == "rk":
            value = h.propagate_rk(case["tableau"], state["dt"], case["steps"])
        else:
            value = h.propagate_imag(case["method"], case["order"], state["dt"], case["steps"])
        h.get_state_device(y.data_ptr())
    here.wait_stream(stream)
    return y if value is None else [y, value]


# ---- what a pass cannot do without ----------------------------------------------
_H_FLOPS = 23            # 5-point H x per point: diagonal, four radial neighbours, two couplings, complex x
_STAGES = {"euler": 1, "classic": 4, "fehlberg": 6, "cash_karp": 6, "dormand_prince": 7, "merson": 5}


def work(case):
    """Bytes: the state (16 B a point) in and out once, the step count of states for a call that records after
    every step.  Flops: the operator applications of the method and its vector updates."""
    kind = case["kind"]

    def lanczos(G, m):   # H, recurrence and two dot products per iteration; the combination at the end
        return G * (m * (_H_FLOPS + 16) + 8 * m)

    if kind in ("batch", "hhg", "served"):
        specs = _specs(case, 0)
        G = sum(s["N"] * (s["lmax"] + 1) for s in specs)
        flops = sum(lanczos(s["N"] * (s["lmax"] + 1), s["krylov"]) for s in specs) * case["steps"]
        return {"bytes": 32.0 * G, "flops": float(flops)}
    G = case["N"] * (case["lmax"] + 1)
    if kind == "hpsi":
        return {"bytes": 32.0 * G, "flops": float(_H_FLOPS * G)}
    if kind == "rk":
        s = _STAGES[case["tableau"]]
        return {"bytes": 32.0 * G, "flops": float(G * case["steps"] * s * (_H_FLOPS + 4 * s))}
    if case["method"] == "lanczos":
        return {"bytes": 32.0 * G, "flops": float(lanczos(G, case["order"]) * case["steps"])}
    stages = case["order"] if case["method"] == "taylor" else 4
    return {"bytes": 32.0 * G, "flops": float(G * case["steps"] * stages * (_H_FLOPS + 4))}


# ---- the same results from plain torch in 64 bits -------------------------------
class _Model:
    """H(t) and the propagators of the paper on one grid, complex128."""

    def __init__(self, N, dr, lmax, stencil, pulse, gauge="length", absorber_r=None):
        self.N, self.dr, self.lmax, self.stencil, self.pulse, self.gauge = N, dr, lmax, stencil, pulse, gauge
        self.r = _radius(N, dr)
        l = torch.arange(lmax + 1, dtype=torch.float64, device="cuda")[:, None]
        h2 = dr * dr
        self.c = (30 / (24 * h2), -16 / (24 * h2), 1 / (24 * h2)) if stencil == 5 else (1 / h2, -0.5 / h2, 0.0)
        self.diag = self.c[0] + 0.5 * l * (l + 1) / self.r ** 2 - 1.0 / self.r
        k = torch.arange(1, lmax + 1, dtype=torch.float64, device="cuda")[:, None]
        self.l1, self.kappa = k, torch.sqrt(k * k / (4 * k * k - 1))
        self.mask = None
        if absorber_r is not None:
            R = N * dr
            x = torch.clamp(self.r - absorber_r, min=0.0) / (R - absorber_r)
            m = torch.cos(0.5 * math.pi * x) ** 0.125
            self.mask = torch.where(self.r > absorber_r, m, torch.ones_like(m))

    def field(self, t):
        p = self.pulse
        T = 2 * math.pi * p["ncycles"] / p["omega"]
        return p["E0"] * math.sin(math.pi * t / T) ** 2 * math.sin(p["omega"] * t + p["cep"]) if 0 <= t <= T else 0.0

    def a_over_c(self, t):   # -int_0^t E, closed form
        p = self.pulse
        T = 2 * math.pi * p["ncycles"] / p["omega"]
        t = min(max(t, 0.0), T)

        def part(w):
            return (math.cos(p["cep"]) - math.cos(w * t + p["cep"])) / w if w else t * math.sin(p["cep"])

        W = 2 * math.pi / T
        return -p["E0"] * (part(p["omega"]) / 2 - (part(p["omega"] + W) + part(p["omega"] - W)) / 4)

    @staticmethod
    def _shift(x, k):
        y = torch.zeros_like(x)
        if abs(k) < x.shape[1]:
            if k > 0:
                y[:, :-k] = x[:, k:]
            else:
                y[:, -k:] = x[:, :k]
        return y

    def d1(self, x):
        s = self._shift
        if self.stencil == 5:
            return (8 * (s(x, 1) - s(x, -1)) - (s(x, 2) - s(x, -2))) / (12 * self.dr)
        return (s(x, 1) - s(x, -1)) / (2 * self.dr)

    def coupling(self, t):
        return self.a_over_c(t) if self.gauge == "velocity" else self.field(t)

    def h(self, x, e):
        y = self.diag * x + self.c[1] * (self._shift(x, 1) + self._shift(x, -1))
        if self.stencil == 5:
            y += self.c[2] * (self._shift(x, 2) + self._shift(x, -2))
        if self.lmax and e:
            if self.gauge == "velocity":
                d, w = self.d1(x), torch.zeros_like(x)
                w[1:] += self.kappa * (d[:-1] - self.l1 / self.r * x[:-1])
                w[:-1] += self.kappa * (d[1:] + self.l1 / self.r * x[1:])
                y += -1j * e * w
            else:
                er = e * self.r
                y[1:] += self.kappa * er * x[:-1]
                y[:-1] += self.kappa * er * x[1:]
        return y

    def lanczos(self, x, e, m, z):
        """exp(z H) x, z = -i dt or -dtau, in the Krylov space of dimension m."""
        nrm = torch.linalg.vector_norm(x)
        q, al, be = [x / nrm], [], []
        for j in range(m):
            w = self.h(q[j], e)
            if j:
                w -= be[-1] * q[j - 1]
            al.append(torch.vdot(q[j].reshape(-1), w.reshape(-1)).real.item())
            if j + 1 == m:
                break
            w -= al[-1] * q[j]
            b = torch.linalg.vector_norm(w).item()
            if b <= 1e-13 * max(1.0, max(abs(v) for v in al)):
                break
            be.append(b)
            q.append(w / b)
        d, v = np.linalg.eigh(np.diag(al) + np.diag(be[:len(al) - 1], 1) + np.diag(be[:len(al) - 1], -1))
        c = (v * np.exp(z * d)) @ v[0].conj()
        out = torch.zeros_like(x)
        for ck, qk in zip(c, q):
            out += complex(ck) * nrm * qk
        return out

    def step(self, x, method, order, t, dt):
        if method == "lanczos":
            x = self.lanczos(x, self.coupling(t + 0.5 * dt), order, -1j * dt)
        elif method == "taylor":
            e, term, acc = self.coupling(t + 0.5 * dt), x, x.clone()
            for k in range(1, order + 1):
                term = (-1j * dt / k) * self.h(term, e)
                acc += term
            x = acc
        else:
            x, _ = self.rk(x, "classic", t, dt)
        return x if self.mask is None else x * self.mask

    def rk(self, x, name, t, dt):
        a, b, bh = _TABLEAUS[name]
        ks = []
        for row in a:
            g = x.clone()
            for aij, kj in zip(row, ks):
                g += dt * aij * kj
            ks.append(-1j * self.h(g, self.coupling(t + sum(row) * dt)))
        new = x + dt * sum(bi * ki for bi, ki in zip(b, ks))
        delta = dt * sum((bi - hi) * ki for bi, hi, ki in zip(b, bh, ks))
        return new, float(torch.sqrt((delta.abs() ** 2).sum() / x.numel()))

    def moments(self, x, t):
        """{t, <z>, <zdot>, <zddot>} of the length gauge."""
        n = float(self.dr * (x.abs() ** 2).sum())
        f, g, d = x[:-1], x[1:], self.d1(x)[:-1]
        re = (f.conj() * g).real
        z = 2 * float((self.kappa * self.r * re).sum()) * self.dr
        v = 2 * float((self.kappa * (g.conj() * (d - self.l1 / self.r * f)).imag).sum()) * self.dr
        a = -2 * float((self.kappa * re / self.r ** 2).sum()) * self.dr - self.field(t) * n
        return [t, z, v, a]

    def flux(self, x, r_b, cos):
        i = min(self.N, max(1, math.ceil(r_b / self.dr - 0.5))) - 1
        f, d = x[:, i].cpu().numpy(), self.d1(x)[:, i].cpu().numpy()
        P = np.polynomial.legendre.legvander(cos, self.lmax)
        Y = P * np.sqrt((2 * np.arange(self.lmax + 1) + 1) / (4 * math.pi))
        return np.concatenate([[np.sum((f.conj() * d).imag)], ((Y @ f).conj() * (Y @ d)).imag])


# published Butcher tableaus: rows a_ij, the propagated weights, the companion's
_TABLEAUS = {
    "euler": ([[]], [1.0], [1.0]),
    "classic": ([[], [1 / 2], [0, 1 / 2], [0, 0, 1]], [1 / 6, 1 / 3, 1 / 3, 1 / 6], [1 / 6, 1 / 3, 1 / 3, 1 / 6]),
    "fehlberg": ([[], [1 / 4], [3 / 32, 9 / 32], [1932 / 2197, -7200 / 2197, 7296 / 2197],
                  [439 / 216, -8, 3680 / 513, -845 / 4104], [-8 / 27, 2, -3544 / 2565, 1859 / 4104, -11 / 40]],
                 [16 / 135, 0, 6656 / 12825, 28561 / 56430, -9 / 50, 2 / 55],
                 [25 / 216, 0, 1408 / 2565, 2197 / 4104, -1 / 5, 0]),
    "cash_karp": ([[], [1 / 5], [3 / 40, 9 / 40], [3 / 10, -9 / 10, 6 / 5], [-11 / 54, 5 / 2, -70 / 27, 35 / 27],
                   [1631 / 55296, 175 / 512, 575 / 13824, 44275 / 110592, 253 / 4096]],
                  [37 / 378, 0, 250 / 621, 125 / 594, 0, 512 / 1771],
                  [2825 / 27648, 0, 18575 / 48384, 13525 / 55296, 277 / 14336, 1 / 4]),
    "dormand_prince": ([[], [1 / 5], [3 / 40, 9 / 40], [44 / 45, -56 / 15, 32 / 9],
                        [19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729],
                        [9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656],
                        [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84]],
                       [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84, 0],
                       [5179 / 57600, 0, 7571 / 16695, 393 / 640, -92097 / 339200, 187 / 2100, 1 / 40]),
    "merson": ([[], [1 / 3], [1 / 6, 1 / 6], [1 / 8, 0, 3 / 8], [1 / 2, 0, -3 / 2, 2]],
               [1 / 6, 0, 0, 2 / 3, 1 / 6], [1 / 10, 0, 3 / 10, 2 / 5, 1 / 5]),
}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "hhg", "served"):
        specs = _specs(case, seed)
        gen = _gen(seed)
        states, series, flux, dens, pad, values, pops = [], [], [], [], [], [], []
        cos = np.cos(np.linspace(0.0, math.pi, case["angles"])) if kind == "hhg" else None
        for s in specs:
            mod = _Model(s["N"], s["dr"], s["lmax"], 5, s, "length", s["absorber_r"])
            t = 0.0 if kind == "served" else _pulse_start(s)
            if kind == "served":
                x = torch.zeros(s["lmax"] + 1, s["N"], dtype=torch.complex128, device="cuda")
                p = mod.r * torch.exp(-mod.r)
                x[0] = p / torch.sqrt(s["dr"] * (p * p).sum())
                ref = x[0].clone()
            else:
                x = _state(s["N"], s["dr"], s["lmax"], gen)
            now = mod.flux(x, s["r_b"], cos) if kind == "hhg" else None
            total = 0.0
            for n in range(case["steps"]):
                x = mod.step(x, "lanczos", s["krylov"], t + n * s["dt"], s["dt"])
                if kind == "hhg":
                    series.append(mod.moments(x, t + (n + 1) * s["dt"]))
                    new = mod.flux(x, s["r_b"], cos)
                    total, now = total + 0.5 * s["dt"] * (now + new), new
            states.append(x.cpu())
            if kind == "hhg":
                flux.append([now[0], total[0]])
                dens.append(now[1:])
                pad.append(total[1:])
            elif kind == "served":
                pop = s["dr"] * (x.abs() ** 2).sum(dim=1)
                dip = 2 * s["dr"] * float((mod.kappa * mod.r * (x[:-1].conj() * x[1:]).real).sum())
                inside = s["dr"] * float((x[:, mod.r <= s["r_b"]].abs() ** 2).sum())
                over = s["dr"] * torch.vdot(ref, x[0])
                values.append([float(pop.sum()), dip, 1.0 - inside, float(over.abs() ** 2)])
                pops.append(pop.cpu().numpy())
        if kind == "served":
            return dict(states=[x.numpy() for x in states], values=np.array(values), l_pop=np.concatenate(pops))
        flat = torch.cat([x.reshape(-1) for x in states])
        if kind == "batch":
            return flat
        return dict(states=flat, series=np.array(series).reshape(len(specs), case["steps"], 4), flux=np.array(flux),
                    density=np.stack(dens), pad=np.stack(pad))
    N, dr, lmax, stencil = case["N"], case["dr"], case["lmax"], case["stencil"]
    p = _pulse(seed)
    ra = max(0.5 * N * dr, N * dr - ABSORBER_WIDTH) if case.get("absorber") else None
    mod = _Model(N, dr, lmax, stencil, p, case.get("gauge", "length"), ra)
    x = _state(N, dr, lmax, _gen(seed), _noise(case))
    t = _pulse_start(p)
    if kind == "hpsi":
        e = mod.field(t)
        return mod.h(x, e / C_AU if mod.gauge == "velocity" else e)
    dt = _step(case, N, lmax, case.get("order", 4), p["E0"], stencil)
    value = 0.0
    for n in range(case["steps"]):
        if kind == "steps":
            x = mod.step(x, case["method"], case["order"], t + n * dt, dt)
        elif kind == "rk":
            x, s = mod.rk(x, case["tableau"], t + n * dt, dt)
            x = x if mod.mask is None else x * mod.mask
            value += s
        else:
            n0 = float((x.abs() ** 2).sum())
            x = mod.lanczos(x, 0.0, case["order"], -dt)
            n1 = float((x.abs() ** 2).sum())
            value = -math.log(n1 / n0) / (2 * dt)
            x = x / math.sqrt(dr * n1)
    return x if kind == "steps" else [x, value]
