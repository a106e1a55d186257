"""What this solver is timed on: whole calls of its public Python entry points (the binding of the C
ABI), over the sizes, precisions, integrators and models that users run.

Every case is one of four kinds:

* ``evolve``  put a handle at its start radius (the initial condition by ``reset``, or a state in
  flavour motion by ``set_rho`` from device memory, as a resumed run does), ``evolve`` it over a
  given number of radial steps and read the state back (FP64 handles: also the moments; every
  handle: the mean survival probability);
* ``batch``   the same for many uneven instances in one handle (``evolve_batch``);
* ``adjoint`` the objective and its gradients over fixed RK4 steps;
* ``readout`` what a program that writes snapshots asks of a large state that it has just set: the
  density matrices, moments, flux spectra and mean survival probability.

Adaptive integrators run with ``h_max_km`` = ``h0_km`` set well inside their tolerance (a bounded
output cadence), so that a pass is a known number of steps.  States of mixed-precision handles are
returned in FP32, the type that the handle holds them in (the ABI's doubles are those values).
"""
import math

import numpy as np
import torch

from paper_1912_10596_gb300 import xflat

R_KM = 11.0                                  # neutrino-sphere radius
E_MIN, E_MAX = 1.0, 60.0                     # MeV
RTOL = {"fp64": 1e-9, "mixed": 1e-6}         # the configured tolerances of the two precisions
DM21, DM31, TH3 = 7.5e-5, 2.4e-3, (0.59, 0.15, 0.785)
MATTER = dict(rho0_gcc=1e7, r_ref_km=100.0, power=3.0, Ye=0.5)

# CODATA constants of the exact values below
_GF, _HBARC = 1.1663787e-5, 197.3269804
_HC_EV, _HC_GEV = _HBARC * 1e-12, _HBARC * 1e-21          # hbar c in eV km and GeV km
_C, _MU = 299792.458, 1.66053906660e-24
_SQ2GF = math.sqrt(2.0) * _GF * _HC_GEV ** 2
_INT = {"rk4": xflat.RK4, "dp45": xflat.DP45, "lie_rk4": xflat.LIE_RK4, "lie_adaptive": xflat.LIE_ADAPTIVE}


def _evolve(name, nf, ne, nu, prec, integ, steps, matter, r0, phase, start, nphi=0):
    c = {"kind": "evolve", "nf": nf, "ne": ne, "nu": nu, "nphi": nphi, "prec": prec, "integ": integ,
         "steps": steps, "matter": matter, "r0": r0, "phase": phase, "start": start}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest configured problem, FP64 RK4 without matter: a scan over parameters makes
        # thousands of such runs, so the time of a step and of a call count
        _evolve("small_rk4_fp64", 2, 64, 32, "fp64", "rk4", 16, "none", 100.0, 0.3, "flavour"),
        # the same grid with the exact propagators (the paper's kind of update)
        _evolve("small_lie_rk4_fp64", 2, 64, 32, "fp64", "lie_rk4", 8, "none", 100.0, 1.0, "flavour"),
        # a mid-sized production run in mixed precision, odd sizes (no bin count divides anything)
        _evolve("mid_dp45_mixed", 2, 201, 397, "mixed", "dp45", 24, "power_law", 60.0, 0.1, "coherent"),
        # the large multi-angle run (4M beams), mixed precision: the headline workload
        _evolve("large_dp45_mixed", 2, 1000, 2000, "mixed", "dp45", 12, "power_law", 40.0, 0.1, "coherent"),
        # and in FP64, the reference that mixed runs are checked against
        _evolve("large_dp45_fp64", 2, 1000, 2000, "fp64", "dp45", 3, "power_law", 40.0, 0.03, "coherent"),
        # the large run with the adaptive exact propagators, from the neutrino sphere through dense
        # matter (large rotation angles): how the whole range 11 -> 500 km is integrated
        _evolve("large_lie_mixed", 2, 1000, 2000, "mixed", "lie_adaptive", 4, "power_law", 11.0, 100.0, "flavour"),
        # three flavours, FP64, the configured 262,144 beams
        _evolve("three_dp45_fp64", 3, 256, 512, "fp64", "dp45", 8, "power_law", 50.0, 0.03, "coherent"),
        # three flavours with the adaptive exact propagators in mixed precision: how the whole
        # range 11 -> 1000 km is integrated
        _evolve("three_lie_mixed", 3, 256, 512, "mixed", "lie_adaptive", 5, "power_law", 50.0, 0.1, "coherent"),
        # the extended bulb model (azimuthal bins) at the shape of the paper's runs
        _evolve("extended_dp45_mixed", 2, 100, 2000, "mixed", "dp45", 8, "power_law", 40.0, 0.1, "coherent", nphi=10),
        # 64 independent instances of uneven sizes in one handle (about 28M beams: parameter scans)
        {"name": "batch64_dp45_mixed", "kind": "batch", "inst": 64, "sizes": 3, "e_lo": 50, "e_hi": 500, "u_lo": 100,
         "u_hi": 1500, "steps": 8, "matter": "none", "r0": 100.0, "phase": 0.1},
        # the gradient of the survival probability, checkpointed: fits to a measured spectrum
        {"name": "adjoint_rk4_fp64", "kind": "adjoint", "ne": 200, "nu": 400, "steps": 128, "every": 64, "matter": "none",
         "r0": 100.0, "phase": 0.3},
        # a snapshot of the large state
        {"name": "readout_large_fp64", "kind": "readout", "nf": 2, "ne": 1000, "nu": 2000, "matter": "power_law", "r0": 60.0},
    ]


def _log(rng, lo, hi):
    """An odd-or-even whole number, spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _grid(rng, e_lo, e_hi, u_lo, u_hi, most):
    while True:
        ne, nu = _log(rng, e_lo, e_hi), _log(rng, u_lo, u_hi)
        if 2 * ne * nu <= most:
            return ne, nu


def draw(rng):
    what = rng.choice(["fp64", "fp64", "mixed", "mixed", "lie", "three", "three_lie", "extended", "batch", "adjoint",
                       "readout"])
    matter = rng.choice(["none", "power_law"])
    r0 = round(math.exp(rng.uniform(math.log(30.0), math.log(300.0))), 3)
    if what == "fp64":
        integ = rng.choice(["rk4", "dp45", "lie_rk4"])
        ne, nu = _grid(rng, 16, 1000, 8, 2000, 4_000_000 if integ != "lie_rk4" else 200_000)
        steps = max(2, min(16, 12_000_000 // (2 * ne * nu) if integ != "lie_rk4" else 8))
        return _evolve("", 2, ne, nu, "fp64", integ, rng.randint(2, steps), matter, r0,
                       0.03 if integ == "dp45" else 0.3, rng.choice(["flavour", "coherent"]))
    if what == "mixed":
        ne, nu = _grid(rng, 16, 1000, 8, 2000, 4_000_000)
        return _evolve("", 2, ne, nu, "mixed", rng.choice(["dp45", "dp45", "rk4"]), rng.randint(4, 12), matter, r0, 0.1,
                       "coherent")
    if what == "lie":
        ne, nu = _grid(rng, 16, 1000, 8, 2000, 4_000_000)
        return _evolve("", 2, ne, nu, "mixed", rng.choice(["lie_adaptive", "lie_adaptive", "lie_rk4"]), rng.randint(2, 4),
                       matter, r0, 0.1, "coherent")
    if what == "three":
        ne, nu = _grid(rng, 16, 256, 16, 512, 262_144)
        return _evolve("", 3, ne, nu, rng.choice(["fp64", "fp64", "mixed"]), rng.choice(["dp45", "rk4"]), rng.randint(3, 8),
                       matter, r0, 0.03, "coherent")
    if what == "three_lie":
        ne, nu = _grid(rng, 16, 256, 16, 512, 262_144)
        return _evolve("", 3, ne, nu, "mixed", rng.choice(["lie_adaptive", "lie_rk4"]), rng.randint(2, 5), matter, r0, 0.1,
                       "coherent")
    if what == "extended":
        nphi = rng.randint(3, 16)
        ne, nu = _grid(rng, 16, 200, 16, 2000, 4_000_000 // nphi)
        return _evolve("", 2, ne, nu, "mixed", rng.choice(["dp45", "rk4"]), rng.randint(3, 8), matter, r0, 0.1, "coherent",
                       nphi=nphi)
    if what == "batch":
        return {"kind": "batch", "inst": _log(rng, 2, 64), "sizes": rng.randint(1, 10 ** 6), "e_lo": 50, "e_hi": 500,
                "u_lo": 100, "u_hi": 1500, "steps": rng.randint(3, 8), "matter": matter, "r0": r0, "phase": 0.1}
    if what == "adjoint":
        ne, nu = _grid(rng, 16, 200, 16, 400, 160_000)
        # without matter, where flavour moves: behind dense matter the gradient is a difference of equal numbers
        return {"kind": "adjoint", "ne": ne, "nu": nu, "steps": rng.randint(64, 128), "every": rng.choice([16, 31, 64]),
                "matter": "none", "r0": round(rng.uniform(80.0, 160.0), 3), "phase": 0.3}
    nf = rng.choice([2, 3])
    ne, nu = _grid(rng, 16, 1000, 8, 2000, 4_000_000 if nf == 2 else 400_000)
    return {"kind": "readout", "nf": nf, "ne": ne, "nu": nu, "matter": matter, "r0": r0}


# ---- inputs ------------------------------------------------------------------------------------------
class _Problem:
    """One bulb-model problem: spectra, mixing and the step, made from the seed."""

    def __init__(self, nf, ne, nu, nphi, matter, r0, rng):
        self.nf, self.ne, self.nu, self.nphi, self.matter, self.r0 = nf, ne, nu, nphi, matter, r0
        self.E = E_MIN + (np.arange(ne) + 0.5) * (E_MAX - E_MIN) / ne
        self.sign = 1.0 if rng.random() < 0.5 else -1.0                      # hierarchy
        self.theta = (rng.uniform(0.05, 0.2),) if nf == 2 else tuple(t * rng.uniform(0.95, 1.05) for t in TH3)
        self.N = np.zeros((2, nf, ne))
        for s, means in enumerate(((11.0, 25.0), (16.0, 25.0))):
            for f, mean in enumerate(means):
                mean = mean * rng.uniform(0.95, 1.05)
                shape = self.E ** 2 / (np.exp(np.minimum(self.E * 3.99 / mean - 3.0, 700.0)) + 1.0)   # Fermi-Dirac, eta = 3
                lum = 10.0 ** rng.uniform(50.7, 51.3)
                n = lum / (mean * 1.602176634e-6) * shape / shape.sum()
                if f == 0:
                    self.N[s, 0] = n
                else:
                    self.N[s, 1:] = n
        self.omega = self.sign * (2.4e-3 if nf == 2 else DM31) / (2.0 * self.E * 1e6 * _HC_EV)
        self.omega21 = DM21 / (2.0 * self.E * 1e6 * _HC_EV)

    def lam(self, r):
        if self.matter == "none":
            return 0.0
        m = MATTER
        return _SQ2GF * m["Ye"] * m["rho0_gcc"] / _MU * 1e15 * (m["r_ref_km"] / r) ** m["power"]

    def mu(self, r):
        return _SQ2GF / (4.0 * math.pi * _C * r * r)

    def step(self, phase):
        """The step in which the fastest beam's generator turns by `phase`."""
        x = (R_KM / self.r0) ** 2
        c = math.sqrt(1.0 - (1.0 - 0.5 / self.nu) * x)
        nunu = self.mu(self.r0) * np.abs(self.N[:, 0] - self.N[:, 1]).sum() * (1.0 / c - c)
        return phase * c / (self.lam(self.r0) + nunu + np.abs(self.omega).max())

    def config(self, prec, integ, h):
        c = xflat.default_config()
        c.n_flavor, c.n_energy, c.n_angle, c.n_phi = self.nf, self.ne, self.nu, self.nphi
        c.precision = xflat.MIXED if prec == "mixed" else xflat.FP64
        c.integrator = _INT[integ]
        c.R_km, c.E_min_MeV, c.E_max_MeV = R_KM, E_MIN, E_MAX
        c.dm2_eV2[0], c.dm2_eV2[1] = (self.sign * 2.4e-3, 0.0) if self.nf == 2 else (DM21, self.sign * DM31)
        for i, t in enumerate(self.theta):
            c.theta[i] = t
        if self.matter == "power_law":
            c.matter_kind = xflat.MATTER_POWER_LAW
            for k, v in MATTER.items():
                setattr(c, k, v)
        c.rtol = c.atol = RTOL[prec]
        c.h0_km = c.h_max_km = c.fixed_dr_km = h
        return c


def _coherent(nf, nb, prec, seed):
    """Pure states around a common one (every beam takes part in the collective motion), as NATIVE planes."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    z = torch.randn((nf, 2, nb), generator=g, device="cuda", dtype=torch.float64)
    z = z * (0.3 / z.square().sum((0, 1)).sqrt())
    z[:, 0] += torch.tensor([1.0, 0.4, 0.2][:nf], device="cuda", dtype=torch.float64)[:, None]
    z = z / z.square().sum((0, 1)).sqrt()
    a, b = z[:, 0], z[:, 1]

    def pair(i, j):                                                   # psi_i conj(psi_j)
        return a[i] * a[j] + b[i] * b[j], b[i] * a[j] - a[i] * b[j]

    if nf == 2:
        re, im = pair(0, 1)
        y = torch.stack([2 * re, -2 * im, a[0] ** 2 + b[0] ** 2 - a[1] ** 2 - b[1] ** 2])
    else:
        y = torch.stack([pair(0, 0)[0], pair(1, 1)[0], pair(2, 2)[0], *pair(0, 1), *pair(0, 2), *pair(1, 2)])
    return y.float().double() if prec == "mixed" else y


def _problem(case, seed):
    return _Problem(case.get("nf", 2), case["ne"], case["nu"], case.get("nphi", 0), case["matter"], case["r0"],
                    np.random.default_rng(seed))


def _instances(case, seed):
    size, rng = np.random.default_rng(case["sizes"]), np.random.default_rng(seed)
    return [_Problem(2, int(size.integers(case["e_lo"], case["e_hi"] + 1)), int(size.integers(case["u_lo"], case["u_hi"] + 1)),
                     0, case["matter"], case["r0"], rng) for _ in range(case["inst"])]


def _beams(p):
    return 2 * p.ne * p.nu * max(1, p.nphi)


def prepare(case, seed):
    s = {"kind": case["kind"], "r0": case["r0"]}
    if case["kind"] == "batch":
        ps = _instances(case, seed)
        h = min(p.step(case["phase"]) for p in ps)
        s["solver"] = xflat.Solver([p.config("mixed", "dp45", h) for p in ps])
        for i, p in enumerate(ps):
            s["solver"].set_spectra(p.N, inst=i)
        s["r1"] = np.full(len(ps), case["r0"] + (case["steps"] - 0.5) * h)
        s["at"] = np.concatenate([[0], np.cumsum([3 * _beams(p) for p in ps])])
        s["out"] = torch.empty(int(s["at"][-1]), dtype=torch.float64, device="cuda")
        return s
    p = _problem(case, seed)
    nb, nc = _beams(p), 3 if p.nf == 2 else 9
    if case["kind"] == "readout":
        s["solver"] = xflat.Solver(p.config("fp64", "dp45", 1e-4))
        s["solver"].set_spectra(p.N)
        s["y0"] = _coherent(p.nf, nb, "fp64", seed)
        s["out"] = torch.empty((nb, p.nf, p.nf, 2), dtype=torch.float64, device="cuda")
        return s
    h = p.step(case["phase"])
    if case["kind"] == "adjoint":
        s["solver"] = xflat.Solver(p.config("fp64", "rk4", h))
        s["solver"].set_spectra(p.N)
        s.update(r1=case["r0"] + case["steps"] * h, steps=case["steps"], every=case["every"])
        return s
    s["solver"] = xflat.Solver(p.config(case["prec"], case["integ"], h))
    s["solver"].set_spectra(p.N)
    s["y0"] = _coherent(p.nf, nb, case["prec"], seed) if case["start"] == "coherent" else None
    s["r1"] = case["r0"] + (case["steps"] - (0.5 if _adaptive(case) else 0.0)) * h
    s["out"] = torch.empty((nc, nb), dtype=torch.float64, device="cuda")
    s["fp64"] = case["prec"] == "fp64"
    return s


def _adaptive(case):
    return case["integ"] in ("dp45", "lie_adaptive")


# ---- one pass ------------------------------------------------------------------------------------------
def run(state):
    s, r0 = state["solver"], state["r0"]
    if state["kind"] == "adjoint":
        J, dN, dth = s.adjoint(r0, state["r1"], state["steps"], state["every"])
        return {"J": np.float64(J), "dJ_dN": dN, "dJ_dtheta": np.float64(dth)}
    if state["kind"] == "readout":
        s.set_rho(None, r0, layout=xflat.LAYOUT_NATIVE, device_ptr=state["y0"].data_ptr())
        s.get_rho(xflat.LAYOUT_MATRIX, device_ptr=state["out"].data_ptr())
        J0, J1 = s.moments()
        return {"rho": state["out"], "J0": J0, "J1": J1, "flux": s.flux_spectra(),
                "pee": np.float64(s.pee(per_beam=False)[1])}
    if state["kind"] == "batch":
        s.reset(r0)
        s.evolve_batch(state["r1"])
        for i, at in enumerate(state["at"][:-1]):
            s.get_rho(xflat.LAYOUT_NATIVE, inst=i, device_ptr=state["out"].data_ptr() + 8 * int(at))
        return {"rho": state["out"].float()}
    if state["y0"] is None:
        s.reset(r0)
    else:
        s.set_rho(None, r0, layout=xflat.LAYOUT_NATIVE, device_ptr=state["y0"].data_ptr())
    s.evolve(r0, state["r1"])
    s.get_rho(xflat.LAYOUT_NATIVE, device_ptr=state["out"].data_ptr())
    pee = s.pee(per_beam=False)[1]
    if not state["fp64"]:
        return {"rho": state["out"].float(), "pee": np.float32(pee)}
    J0, J1 = s.moments()
    return {"rho": state["out"], "pee": np.float64(pee), "J0": J0, "J1": J1}


# ---- what a pass cannot do without -----------------------------------------------------------------------
def work(case):
    if case["kind"] == "batch":
        nb = sum(_beams(p) for p in _instances(case, 0))
        return {"bytes": nb * 3 * (4 + 4), "flops": nb * case["steps"] * _flops(2, "dp45", 0)}
    nb = 2 * case["ne"] * case["nu"] * max(1, case.get("nphi", 0))
    if case["kind"] == "adjoint":
        # the state and its cotangent once through every step's start state; a forward and a reverse sweep
        return {"bytes": nb * 3 * 8 * case["steps"] * 2, "flops": nb * case["steps"] * 3 * _flops(2, "rk4", 0)}
    nc = 3 if case["nf"] == 2 else 9
    if case["kind"] == "readout":
        return {"bytes": nb * 8 * (nc + 2 * case["nf"] ** 2), "flops": nb * (4 * nc + 6)}
    size = 8 if case["prec"] == "fp64" else 4
    return {"bytes": nb * nc * (8 * (case["start"] == "coherent") + size),
            "flops": nb * case["steps"] * _flops(case["nf"], case["integ"], case["nphi"])}


def _flops(nf, integ, nphi):
    """Operations a beam and step: stage derivatives or propagators, stage states, moments."""
    nc = 3 if nf == 2 else 9
    rhs = 13 if nf == 2 else 116
    exp = rhs + (50 if nf == 2 else 500)
    moments = 2 * nc * (4 if nphi else 2)
    if integ == "dp45":
        return 6 * (rhs + moments) + 2 * 26 * nc + 8 * nc
    if integ == "rk4":
        return 4 * (rhs + moments) + 2 * 7 * nc
    if integ == "lie_rk4":
        return 4 * (rhs + moments) + 5 * exp
    return 11 * (rhs + moments) + 18 * exp


# ---- the same in 64 bits, in plain torch ---------------------------------------------------------------------
class _Exact:
    """Two flavours: Bloch vectors s [3, 2, angles, energies]; three: matrices [2, angles, energies, 3, 3].
    Antineutrinos carry the conjugate, so that every beam obeys d rho/dr = -i [H, rho] / cos theta with the
    vacuum term's sign reversed and a signed weight."""

    def __init__(self, p):
        self.p, self.dev = p, torch.device("cuda" if torch.cuda.is_available() else "cpu")
        t = lambda v: torch.as_tensor(np.asarray(v), dtype=torch.float64, device=self.dev)  # noqa: E731
        m = max(1, p.nphi)
        self.u = t((np.arange(p.nu) + 0.5) / p.nu).repeat_interleave(m)
        self.phi = t(2 * math.pi * (np.arange(m) + 0.5) / m).repeat(p.nu)
        self.du = 1.0 / (p.nu * m)
        self.eta = t([1.0, -1.0])[:, None, None]
        self.N, self.theta = t(p.N), t(p.theta)
        self.om, self.om21 = t(p.omega), t(p.omega21)
        if p.nf == 3:
            c, s = np.cos(p.theta), np.sin(p.theta)
            U = (np.array([[1, 0, 0], [0, c[2], s[2]], [0, -s[2], c[2]]]) @ np.array([[c[1], 0, s[1]], [0, 1, 0], [-s[1], 0, c[1]]])
                 @ np.array([[c[0], s[0], 0], [-s[0], c[0], 0], [0, 0, 1]]))
            M21, M31 = t(np.outer(U[:, 1], U[:, 1])), t(np.outer(U[:, 2], U[:, 2]))
            self.vac = (self.eta[..., None, None] * (self.om21[:, None, None] * M21 + self.om[:, None, None] * M31)).to(torch.complex128)

    def g(self):
        return torch.stack([self.N[0, 0] - self.N[0, 1], -(self.N[1, 0] - self.N[1, 1])])      # [2, ne]

    def start(self, y0):
        n = (2, len(self.u), self.p.ne)
        if self.p.nf == 2:
            if y0 is not None:
                return y0.to(self.dev).reshape(3, *n)
            s = torch.zeros((3, *n), dtype=torch.float64, device=self.dev)
            s[2] = 1.0
            return s
        if y0 is None:
            y0 = torch.zeros((9, 2 * len(self.u) * self.p.ne), dtype=torch.float64, device=self.dev)
            y0[0] = 1.0
        return self.matrix(y0.to(self.dev)).reshape(*n, 3, 3)

    @staticmethod
    def matrix(y):
        o = [torch.complex(y[3], y[4]), torch.complex(y[5], y[6]), torch.complex(y[7], y[8])]
        d = [v.to(torch.complex128) for v in y[:3]]
        rows = [d[0], o[0], o[1], o[0].conj(), d[1], o[2], o[1].conj(), o[2].conj(), d[2]]
        return torch.stack([v.resolve_conj() for v in rows], -1).reshape(-1, 3, 3)

    def native(self, y):
        if self.p.nf == 2:
            return y.reshape(3, -1)
        y = y.reshape(-1, 3, 3)
        o = [y[:, 0, 1], y[:, 0, 2], y[:, 1, 2]]
        return torch.stack([*(y[:, i, i].real for i in range(3)), *(v for z in o for v in (z.real, z.imag))])

    def rows(self, y):
        """sum over species and energies of weight x state, by angle bin: [3, angles] or [angles, 3, 3]."""
        if self.p.nf == 2:
            return self.du * torch.einsum("sk,csjk->cj", self.g(), y)
        return self.du * torch.einsum("sk,sjkab->jab", self.g().to(torch.complex128), y)

    def moments(self, r, y):
        c = torch.sqrt(1.0 - self.u * (R_KM / r) ** 2)
        F = self.rows(y)
        J0, J1 = ((F / c).sum(-1), F.sum(-1)) if self.p.nf == 2 else ((F / c[:, None, None]).sum(0), F.sum(0))
        if self.p.nf == 2:
            out = []
            for J in (J0, J1):
                out.append(0.5 * torch.stack([torch.complex(J[2], 0 * J[2]), torch.complex(J[0], -J[1]),
                                              torch.complex(J[0], J[1]), torch.complex(-J[2], 0 * J[2])]).reshape(2, 2))
            return out
        eye = torch.eye(3, dtype=torch.complex128, device=self.dev)
        return [J - eye * torch.trace(J) / 3 for J in (J0, J1)]

    def gen(self, r, y):
        """H / cos theta of every beam."""
        p, x = self.p, (R_KM / r) ** 2
        c = torch.sqrt(1.0 - self.u * x)
        F, lam, mu = self.rows(y), p.lam(r), p.mu(r)
        if p.nf == 2:
            nn = (F * (1 / c - 1)).sum(-1, keepdim=True) + (1 - c) * F.sum(-1, keepdim=True)
            if p.nphi:
                st = torch.sqrt(self.u * x)
                for f in (torch.cos, torch.sin):
                    nn = nn - st * f(self.phi) * (F * (st / c) * f(self.phi)).sum(-1, keepdim=True)
            nn = mu * nn                                                                    # [3, angles]
            v = self.eta * self.om                                                          # [2, 1, ne]
            K = [v * torch.sin(2 * self.theta[0]) + nn[0][:, None], nn[1][:, None] + 0 * v,
                 -v * torch.cos(2 * self.theta[0]) + lam + nn[2][:, None]]
            return torch.stack(K) / c[:, None]
        J0m1 = (F * (1 / c - 1)[:, None, None]).sum(0)
        H = mu * (J0m1 + (1 - c)[:, None, None] * F.sum(0))
        H = H.clone()
        H[:, 0, 0] += lam
        return (self.vac + H[:, None]) / c[:, None, None, None]

    def rhs(self, r, y):
        K = self.gen(r, y)
        if self.p.nf == 2:
            return torch.linalg.cross(K, y, dim=0)
        return -1j * (K @ y - y @ K)

    def exp(self, Om, y):
        if self.p.nf == 2:
            t = torch.sqrt((Om * Om).sum(0)).clamp_min(1e-300)
            n = Om / t
            cr = torch.linalg.cross(n, y, dim=0)
            return y + torch.sin(t) * cr + 2 * torch.sin(t / 2) ** 2 * torch.linalg.cross(n, cr, dim=0)
        U = torch.linalg.matrix_exp(-1j * Om)
        return U @ y @ U.mH

    def rk4(self, r, y, h):
        k1 = self.rhs(r, y)
        k2 = self.rhs(r + h / 2, y + (h / 2) * k1)
        k3 = self.rhs(r + h / 2, y + (h / 2) * k2)
        k4 = self.rhs(r + h, y + h * k3)
        return y + (h / 6) * (k1 + 2 * k2 + 2 * k3 + k4)

    def dp45(self, r, y, h):
        a = ((1 / 5,), (3 / 40, 9 / 40), (44 / 45, -56 / 15, 32 / 9), (19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729),
             (9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656), (35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84))
        k = [self.rhs(r, y)]
        for c, row in zip((0.2, 0.3, 0.8, 8 / 9, 1.0, 1.0), a):
            Y = y + h * sum(v * q for v, q in zip(row, k))
            if len(k) < 6:
                k.append(self.rhs(r + c * h, Y))
        return Y

    def lie_rk4(self, r, y, h):
        """Commutator-free Lie RK4 (Celledoni, Marthinsen and Owren 2003)."""
        G1 = self.gen(r, y)
        y2 = self.exp(h / 2 * G1, y)
        G2 = self.gen(r + h / 2, y2)
        G3 = self.gen(r + h / 2, self.exp(h / 2 * G2, y))
        G4 = self.gen(r + h, self.exp(h * (G3 - G1 / 2), y2))
        y = self.exp(h * (G1 / 4 + (G2 + G3) / 6 - G4 / 12), y)
        return self.exp(h * (-G1 / 12 + (G2 + G3) / 6 + G4 / 4), y)

    def lie_adaptive(self, r, y, h):
        return self.lie_rk4(r + h / 2, self.lie_rk4(r, y, h / 2), h / 2)

    def steps(self, method, y, r0, h, n, half):
        """n steps of h, the last one h / 2 long where `half`."""
        r = r0
        for i in range(n):
            if not half:
                r = r0 + i * h
            y = getattr(self, method)(r, y, h if i < n - 1 or not half else r0 + (n - 0.5) * h - r)
            r = r + h
        return y

    def pee(self, y):
        """The electron-flavour survival probability of every neutrino beam, and its number-weighted mean."""
        P = (1 + y[2, 0]) / 2 if self.p.nf == 2 else y[0, ..., 0, 0].real
        return (self.N[0, 0] * P).sum() / (self.N[0, 0].sum() * len(self.u))

    def flux(self, y):
        out = []
        for s in range(2):
            P = [(1 + y[2, s]) / 2, (1 - y[2, s]) / 2] if self.p.nf == 2 else [y[s, ..., a, a].real for a in range(3)]
            out.append(torch.stack([(self.du * (self.N[s, 0] * Q + self.N[s, 1] * (1 - Q))).sum(0) for Q in P]))
        return torch.stack(out)


def exact(case, seed):
    with torch.no_grad():
        if case["kind"] == "batch":
            ps = _instances(case, seed)
            h = min(p.step(case["phase"]) for p in ps)
            out = []
            for p in ps:
                e = _Exact(p)
                out.append(e.native(e.steps("dp45", e.start(None), case["r0"], h, case["steps"], True)).reshape(-1))
            return {"rho": torch.cat(out)}
        p = _problem(case, seed)
        e = _Exact(p)
        if case["kind"] == "adjoint":
            return _exact_adjoint(e, case)
        coherent = case["kind"] == "readout" or case["start"] == "coherent"
        y = e.start(_coherent(p.nf, _beams(p), case.get("prec", "fp64"), seed) if coherent else None)
        if case["kind"] == "readout":
            n = e.native(y)
            J0, J1 = e.moments(case["r0"], y)
            if p.nf == 2:
                m = torch.stack([torch.complex((1 + n[2]) / 2, 0 * n[2]), torch.complex(n[0] / 2, -n[1] / 2),
                                 torch.complex(n[0] / 2, n[1] / 2), torch.complex((1 - n[2]) / 2, 0 * n[2])], -1).reshape(-1, 2, 2)
            else:
                m = e.matrix(n)
            half = m.shape[0] // 2
            m = torch.cat([m[:half], m[half:].conj().resolve_conj()])            # antineutrinos: the paper's own matrices
            return {"rho": torch.view_as_real(m), "J0": J0, "J1": J1, "flux": e.flux(y), "pee": e.pee(y)}
        h = p.step(case["phase"])
        y = e.steps(case["integ"], y, case["r0"], h, case["steps"], _adaptive(case))
        out = {"rho": e.native(y), "pee": e.pee(y)}
        if case["prec"] == "fp64":
            out["J0"], out["J1"] = e.moments(case["r0"] + (case["steps"] - (0.5 if _adaptive(case) else 0.0)) * h, y)
        return out


def _exact_adjoint(e, case):
    """Reverse mode, one step at a time from the stored step starts."""
    h, at = e.p.step(case["phase"]), []
    y = e.start(None)
    for n in range(case["steps"]):
        at.append(y)
        y = e.rk4(case["r0"] + n * h, y, h)
    with torch.enable_grad():
        N, th = e.N.requires_grad_(), e.theta.requires_grad_()
        y = y.requires_grad_()
        J = e.pee(y)
        a, dN, dth = (*torch.autograd.grad(J, (y, N)), torch.zeros_like(th))
        for n in reversed(range(case["steps"])):
            y = at[n].requires_grad_()
            a, gN, gth = torch.autograd.grad(e.rk4(case["r0"] + n * h, y, h), (y, N, th), a)
            dN, dth = dN + gN, dth + gth
    return {"J": J.detach(), "dJ_dN": dN, "dJ_dtheta": dth.reshape(())}
