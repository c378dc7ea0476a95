"""The work a user of this package has it do, as cases that can be timed and compared.

A case is one call sequence of a solve through the package's public entry points: a check
interval of imaginary-time steps of one lattice (``Lattice.step_n``), the same with the
excited-state record and a parity projection, with the upload of a new start field, a
chunk of a served batch (``Batch.step``), or one allocation-free step
(``qf_fft_step_static``).  Sizes, kinetic terms, potentials and precisions are those of the
workloads in ``paper_2211_10185_gb300/inputs.py``, of the served mix in ``serve.py`` and of
the tests.  ``exact`` restates each sequence in plain torch with 64-bit numbers.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2211_10185_gb300 import inputs as I
from paper_2211_10185_gb300 import qfdtd as Q
from paper_2211_10185_gb300.lattice import Lattice
from paper_2211_10185_gb300.serve import Batch

KINETIC = {"fdtd": I.FDTD, "naive": I.FFT_NAIVE, "symanzik": I.FFT_SYMANZIK, "rel": I.FFT_REL}
FFT_SIZES = (8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512)
INTERVAL = 64  # steps between checks, as the benchmark and the server use


def _case(kind, n, kinetic, a, mass, potential, precision="c64", steps=INTERVAL, dtau=0.0, **more):
    return dict(kind=kind, n=n, kinetic=kinetic, a=a, mass=mass, potential=potential, precision=precision,
                steps=steps, dtau=dtau, **more)


def listed():
    return [
        # the smallest call: one step for a caller that owns no workspace
        _case("static", 32, "rel", 0.25, 0.5, "cornell", steps=1, dtau=0.02, name="static_n32_rel"),
        # the smallest lattice of the served mix, alone: launches and latency count
        _case("step", 32, "symanzik", 0.25, 1.0, "oscillator", name="step_n32_symanzik"),
        # the middle of the served mix, alone
        _case("step", 64, "rel", 0.25, 0.8, "cornell", name="step_n64_rel"),
        # a size with a factor 3 and a complex (non-equilibrium) potential
        _case("step", 96, "naive", 0.1, 1.2, "gaussmix", name="step_n96_naive_complex"),
        # Cornell workload, k^2 term: an interval, the three-state record, a parity projection
        _case("excited", 128, "naive", 0.1, 1.5, "cornell", name="excited_n128_naive"),
        # the benchmark's step: relativistic workload with the same record and projection
        _case("excited", 256, "rel", 0.05, 0.3, "cornell", dtau=0.0125, name="excited_n256_rel"),
        # the largest lattice: Gaussian-mix workload, complex potential
        _case("step", 512, "symanzik", 0.04, 1.0, "gaussmix", name="step_n512_symanzik_complex"),
        # oscillator workload: Dirichlet stencil in FP64
        _case("step", 32, "fdtd", 0.15, 1.0, "oscillator", "c128", dtau=0.15 ** 2 / 8, name="step_n32_fdtd_c128"),
        # Dirichlet stencil in FP32 on a size that no tile divides
        _case("step", 250, "fdtd", 0.06, 0.5, "cornell", name="step_n250_fdtd"),
        # the FP64 form of an FFT term, which excited states of close levels are taken from
        _case("step", 64, "rel", 0.25, 0.8, "cornell", "c128", name="step_n64_rel_c128"),
        # a new start field from page-locked host memory, then an interval
        _case("host", 192, "symanzik", 1.0 / 12, 0.9, "cornell", name="host_n192_symanzik"),
        # one chunk of the served mix: sizes and kinetic terms of waiting requests together
        _case("batch", 192, "mixed", 0.0, 0.0, "cornell", name="batch_served_mix",
              members="32:rel 48:fdtd 32:naive 64:symanzik 96:rel 48:symanzik 64:fdtd 128:naive 32:fdtd 96:naive "
                      "128:rel 192:symanzik"),
    ]


def _log_even(rng, lo, hi):
    """An even number in [lo, hi], even in the logarithm."""
    return max(lo, min(hi, 2 * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2)))


def draw(rng):
    c = _draw(rng)
    if c["kind"] != "batch":
        # no coarser than the time step resolves: the wells of a Gaussian mix, or the mean of a
        # confining potential (on which a start field of noise decays)
        depth = {"gaussmix": 15.0, "oscillator": 0.18 * (c["n"] * c["a"]) ** 2, "cornell": 0.12 * c["n"] * c["a"]}
        while 0.5 * _default_dtau(c["kinetic"], c["a"], c["mass"]) * depth[c["potential"]] > 0.2:
            c["a"] = round(0.7 * c["a"], 4)
            c["dtau"] = round(0.5 * c["dtau"], 6)
            depth["oscillator"] *= 0.49
            depth["cornell"] *= 0.7
    return c


def _draw(rng):
    kind = rng.choice(("step", "step", "step", "fdtd", "fdtd", "fp64", "static", "excited", "host", "batch"))
    fft = rng.choice(("naive", "symanzik", "rel"))
    mass = round(rng.uniform(0.3, 3.0), 3)
    potential = rng.choice(("cornell", "cornell", "oscillator", "gaussmix"))
    box = rng.uniform(8.0, 16.0)
    if kind == "static":
        n = rng.choice([s for s in FFT_SIZES if s <= 64])
        return _case("static", n, fft, round(box / n, 4), mass, potential, steps=1,
                     dtau=round(rng.uniform(0.2, 0.6) * _default_dtau(fft, box / n, mass), 6))
    if kind == "batch":
        sizes = [rng.choice((32, 32, 48, 48, 64, 64, 96, 96, 128, 192)) for _ in range(rng.randint(4, 16))]
        return _case("batch", max(sizes), "mixed", 0.0, 0.0, "cornell",
                     members=" ".join("%d:%s" % (s, rng.choice(("fdtd", "naive", "symanzik", "rel"))) for s in sizes))
    if kind == "fdtd":
        n = _log_even(rng, 16, 400)
        return _case("step", n, "fdtd", round(box / n, 4), mass, potential, steps=INTERVAL)
    if kind == "fp64":
        if rng.random() < 0.5:
            n = _log_even(rng, 16, 160)
            return _case("step", n, "fdtd", round(box / n, 4), mass, potential, "c128", steps=rng.choice((16, 32)))
        n = rng.choice([s for s in FFT_SIZES if 16 <= s <= 128])
        return _case("step", n, fft, round(box / n, 4), mass, potential, "c128", steps=rng.choice((16, 32)))
    if kind == "excited":
        # nearby snapshots: the states of a record are differences of them
        n = rng.choice([s for s in FFT_SIZES if 96 <= s <= 256])
        return _case("excited", n, fft, round(box / n, 4), mass, "cornell", steps=rng.choice((16, 24, 32)))
    if kind == "host":
        n = rng.choice([s for s in FFT_SIZES if 48 <= s <= 256])
        return _case("host", n, fft, round(box / n, 4), mass, potential)
    n = rng.choice([s for s in FFT_SIZES if s <= 384])
    return _case("step", n, fft, round(box / n, 4), mass, potential, steps=rng.choice((32, 48, INTERVAL)))


# ---- inputs ---------------------------------------------------------------------------

def _radius(n, a):
    x = (torch.arange(n, dtype=torch.float64, device="cuda") - n // 2) * a
    return torch.sqrt(x[:, None, None] ** 2 + x[None, :, None] ** 2 + x[None, None, :] ** 2)


def _potential(kind, n, a, seed):
    """V(r) of a solve: parameters from the seed, in the ranges of the workloads."""
    rng = np.random.default_rng(seed)
    if kind == "gaussmix":
        L = n * a
        centres = rng.uniform(-L / 4, L / 4, size=(32, 3))
        widths, depths = rng.uniform(0.2, 1.0, 32), rng.uniform(-5.0, 0.0, 32)
        x = (torch.arange(n, dtype=torch.float64, device="cuda") - n // 2) * a
        v = torch.zeros((n, n, n), dtype=torch.float64, device="cuda")
        for (cx, cy, cz), w, d in zip(centres, widths, depths):
            gx, gy, gz = (torch.exp(-(x - float(c)) ** 2 / (2 * float(w) ** 2)) for c in (cx, cy, cz))
            v += float(d) * gz[:, None, None] * (gy[:, None] * gx[None, :])[None]
        return torch.complex(v, -0.05 * v.abs())
    r = _radius(n, a)
    if kind == "oscillator":
        return 0.5 * float(rng.uniform(0.8, 1.2)) ** 2 * r ** 2
    r[r == 0] = a / 2
    return -float(rng.uniform(0.3, 0.6)) / r + float(rng.uniform(0.1, 0.25)) * r


def _noise(n, seed, dirichlet):
    """Start field: independent normal real and imaginary parts."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    psi = torch.complex(*(torch.randn((n, n, n), generator=g, dtype=torch.float64, device="cuda") for _ in range(2)))
    if dirichlet:
        psi[0], psi[:, 0], psi[:, :, 0] = 0, 0, 0
    return psi


def _blob(n, a, mass, seed, dirichlet):
    """Start field of a served request: a Gaussian of a seeded width."""
    w = float(np.random.default_rng(seed).uniform(0.5, 2.0)) / math.sqrt(mass)
    psi = torch.exp(-0.5 * (_radius(n, a) / w) ** 2).to(torch.complex128)
    if dirichlet:
        psi[0], psi[:, 0], psi[:, :, 0] = 0, 0, 0
    return psi


def _members(case, seed):
    """The solves of a batch: (n, a, kinetic, mass, seed) with the served mix's box and masses."""
    rng = np.random.default_rng(seed)
    return [(int(s), 16.0 / int(s), k, float(rng.uniform(0.3, 5.0)), seed * 100 + i)
            for i, (s, k) in enumerate(m.split(":") for m in case["members"].split())]


def _lattice(n, a, kinetic, mass, dtau, v, psi, precision="c64"):
    lat = Lattice(n, a, precision=precision)
    lat.set_potential(v.cpu().numpy())
    lat.set_kinetic(KINETIC[kinetic], mass, dtau or None)
    if psi is not None:
        lat.set_wavefunction(psi.cpu().numpy())
    return lat


def _energy_type(v, precision):
    """The energy as a number of the lattice's precision; complex where the potential is."""
    if not v.is_complex():
        return lambda e: e.real
    return np.complex64 if precision == "c64" else np.complex128


def prepare(case, seed):
    n, a = case["n"], case["a"]
    if case["kind"] == "batch":
        batch = Batch()
        for n, a, kin, mass, s in _members(case, seed):
            lat = _lattice(n, a, kin, mass, 0.0, _potential("cornell", n, a, s), _blob(n, a, mass, s, kin == "fdtd"))
            batch.add(lat, 1 << 40, 0.0)
        return dict(case=case, batch=batch)
    v = _potential(case["potential"], n, a, seed)
    psi = _noise(n, seed, case["kinetic"] == "fdtd")
    if case["kind"] == "static":
        return dict(case=case, lib=Q.load(), psi=psi.to(torch.complex64).contiguous(),
                    v=v.to(torch.complex64 if v.is_complex() else torch.float32).contiguous())
    state = dict(case=case, energy=_energy_type(v, case["precision"]))
    if case["kind"] == "host":
        host = torch.empty((2 * n ** 3,), dtype=torch.float64, pin_memory=True)
        host.copy_(torch.view_as_real(psi).reshape(-1))
        state["host"] = host.numpy()
        state["pinned"] = host
        psi = None
    lat = state["lat"] = _lattice(n, a, case["kinetic"], case["mass"], case["dtau"], v, psi, case["precision"])
    if case["kind"] == "excited":
        lat.step_n(2 * case["steps"], 0.0, check_every=case["steps"])  # two of the record's three snapshots
    return state


# ---- one pass -------------------------------------------------------------------------

def run(state):
    case = state["case"]
    if case["kind"] == "static":
        v, psi = state["v"], state["psi"]
        st = state["lib"].qf_fft_step_static(
            case["n"], case["a"], KINETIC[case["kinetic"]], case["mass"], case["dtau"], ctypes.c_void_p(psi.data_ptr()),
            ctypes.c_void_p(v.data_ptr()), int(v.is_complex()), 1.0, None,
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if st != Q.QF_OK:
            raise Q.QFError(st, "qf_fft_step_static")
        return {"psi": psi}
    if case["kind"] == "batch":
        batch = state["batch"]
        batch.step(case["steps"], check_every=case["steps"])
        return [{"psi": m.field_tensor(), "energy": m.energies()["e"].real} for m in batch.members]
    lat, steps = state["lat"], case["steps"]
    if case["kind"] == "host":
        lat.set_wavefunction_raw(state["host"])
    lat.step_n(steps, 0.0, check_every=steps, snap_every=steps if case["kind"] == "excited" else 0)
    e = lat.energies()["e"]
    out = {"psi": lat.field_tensor(), "energy": state["energy"](e)}
    if case["kind"] == "excited":
        rec = lat.track_excited(3)
        lat.parity_project(Q.QF_P_MINUS_PK, 3, 1)
        out["energies"] = [r["e"].real for r in rec]
        out["states"] = [lat.field_tensor(i) for i in range(3)]
    return out


# ---- what a pass cannot do without ----------------------------------------------------

def _sites_work(n, kinetic, precision, cplx, steps):
    sites, real = n ** 3, 4 if precision == "c64" else 8
    # forward and inverse transforms of 3 axes, the momentum multiply and the update; or the
    # 7-point sum and the update
    flops = 30 * math.log2(n) + 14 if kinetic != "fdtd" else 26
    return sites * real * (4 + (2 if cplx else 1)), sites * steps * flops


def work(case):
    """Each input read once and each output written once; the arithmetic of every step."""
    if case["kind"] == "batch":
        parts = [_sites_work(n, k, "c64", False, case["steps"]) for n, _, k, _, _ in _members(case, 0)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    n, cplx = case["n"], case["potential"] == "gaussmix"
    b, f = _sites_work(n, case["kinetic"], case["precision"], cplx, case["steps"])
    if case["kind"] == "host":
        b += 16 * n ** 3  # the field as it lies in host memory
    if case["kind"] == "excited":
        # two snapshots and the field read, three states written; three energies, the inner
        # products and the projection
        b += 5 * 8 * n ** 3
        f += n ** 3 * (3 * 15 * math.log2(n) + 150)
    return {"bytes": b, "flops": f}


# ---- the same in 64 bits --------------------------------------------------------------

def _default_dtau(kinetic, a, m):
    top = {"fdtd": 6 / (m * a * a), "symanzik": 6 / (m * a * a), "naive": 3 * math.pi ** 2 / (2 * m * a * a),
           "rel": math.sqrt(12 + (a * m) ** 2) / a}[kinetic]
    return 0.75 / top


class _Exact:
    """The iteration on a field kept in 64 bits: psi' = s ((2 - d) psi - dtau H_K psi) / d with
    d = 1 + dtau V / 2, s the documented output scale (a power of two, after a check also
    1 / sqrt(norm))."""

    def __init__(self, n, a, kinetic, m, dtau, v, psi):
        self.n, self.a, self.m, self.v, self.psi = n, a, m, v, psi
        self.fdtd = kinetic == "fdtd"
        self.dt = dtau if dtau > 0 else _default_dtau(kinetic, a, m)
        if not self.fdtd:
            j = torch.arange(n, dtype=torch.float64, device="cuda")
            k = 2 * math.pi * torch.where(j <= n // 2, j, j - n) / n
            s = k ** 2 if kinetic == "naive" else 4 * torch.sin(k / 2) ** 2
            s = s[:, None, None] + s[None, :, None] + s[None, None, :]
            self.t = torch.sqrt(s + (a * m) ** 2) / a if kinetic == "rel" else s / (2 * a * a * m)
        self.step, self.renorm, self.k, self.j, self.scale = 0, -1, 0, 0, 1.0

    def kinetic(self, f):
        if not self.fdtd:
            return torch.fft.ifftn(self.t * torch.fft.fftn(f))
        h = 6 * f
        for d in range(3):
            h -= torch.roll(f, 1, d)
            h -= torch.roll(f, -1, d)
        h /= 2 * self.m * self.a ** 2
        h[0], h[:, 0], h[:, :, 0] = 0, 0, 0
        return h

    def energy(self, f, h=None):
        h = self.kinetic(f) if h is None else h
        norm = torch.linalg.vector_norm(f).item() ** 2
        return complex((torch.vdot(f.reshape(-1), h.reshape(-1)) + (f.abs() ** 2 * self.v).sum()).item()) / norm, norm

    def advance(self, steps, check_every):
        e = None
        d = 1 + 0.5 * self.dt * self.v
        after_check = False
        for _ in range(steps):
            h = self.kinetic(self.psi)
            out = 2.0 ** self.k
            if after_check:
                out = self.scale
                self.renorm = self.step
                after_check = False
            if check_every and self.step % check_every == 0:
                e, norm = self.energy(self.psi, h)
                if self.renorm >= 0 and self.step > self.renorm:
                    lam = (0.5 * math.log2(norm) - self.j) / (self.step - self.renorm) - self.k
                    self.k = min(max(round(-lam), -30), 30)
                    self.j = min(max(-round(0.5 * (lam + self.k) * (self.step - self.renorm - 1)), -60), 60)
                else:
                    q = abs((1 - 0.5 * self.dt * e.real) / (1 + 0.5 * self.dt * e.real))
                    self.k, self.j = min(max(round(-math.log2(q)), -30), 30), 0
                self.scale = 2.0 ** (self.k + self.j) / math.sqrt(norm)
                after_check = True
            self.psi = ((2 - d) * self.psi - self.dt * h) / d * out
            if self.fdtd:
                self.psi[0], self.psi[:, 0], self.psi[:, :, 0] = 0, 0, 0
            self.step += 1
        return e


def _mirror(f, axes):
    """f at the mirrored sites (index i -> (N - i) mod N on each of the axes)."""
    return torch.roll(torch.flip(f, axes), [1] * len(axes), axes)


def _excited(x, snaps):
    """Classical Gram-Schmidt, twice, latest snapshot first; the energies of the states."""
    states, energies = [], []
    for s in snaps:
        w = s.clone()
        for _ in range(2):
            c = [torch.vdot(u.reshape(-1), w.reshape(-1)) for u in states]
            for u, k in zip(states, c):
                w -= k * u
        states.append(w / torch.linalg.vector_norm(w))
        energies.append(x.energy(states[-1])[0].real)
    return states, energies


def exact(case, seed):
    n, a, steps = case["n"], case["a"], case["steps"]
    if case["kind"] == "batch":
        out = []
        for n, a, kin, mass, s in _members(case, seed):
            x = _Exact(n, a, kin, mass, 0.0, _potential("cornell", n, a, s), _blob(n, a, mass, s, kin == "fdtd"))
            e = x.advance(steps, steps)
            out.append({"psi": x.psi, "energy": e.real})
        return out
    x = _Exact(n, a, case["kinetic"], case["mass"], case["dtau"], _potential(case["potential"], n, a, seed),
               _noise(n, seed, case["kinetic"] == "fdtd"))
    if case["kind"] == "static":
        x.advance(1, 0)
        return {"psi": x.psi}
    if case["kind"] == "excited":
        snaps = []
        for _ in range(3):
            e = x.advance(steps, steps)
            snaps.insert(0, x.psi)
        states, energies = _excited(x, snaps)
        f = states[1]
        p = (f + _mirror(f, (1, 2))) - (_mirror(f, (0,)) + _mirror(f, (0, 1, 2)))
        states[1] = p / torch.linalg.vector_norm(p)
        return {"psi": x.psi, "energy": e.real, "energies": energies, "states": states}
    e = x.advance(steps, steps)
    return {"psi": x.psi, "energy": np.complex128(e) if x.v.is_complex() else e.real}
