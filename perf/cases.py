"""What a user of the framework has it do, as cases that can be timed and compared.

A case is one call, or one short run of calls, of the public entry points on lattices that live on
the GPU: leapfrog steps of classical phi^4 fields (one to six real components, FP64, FP32 with the
Kahan-compensated drift, plain FP32), with the kernel the library takes by itself or with the plan
lf2_tune made, steps with an energy record each, energies alone, batched ensembles, field
derivatives and power spectra.  Buffers are torch tensors lent to the library (lf2_field_wrap), as
a program built around torch does it; a state keeps its fields and plan from pass to pass.
"""
import math

import numpy as np
import torch

from paper_1508_05610_gb300 import inputs, lf2

DX, ETA = 1.0, 1.0
SIGMA = 0.1  # standard deviation of phi_0 per component
SIZES = ("nx", "ny", "nz")


def listed():
    return [
        # The smallest workload in earnest: a 32^3 real FP64 run that reports energy and checksums
        # at every one of its 100 steps.  Latency and the barrier between steps count.
        dict(name="energy_every_step_32_f64", kind="step_energy", nx=32, ny=32, nz=32, ncomp=1, prec="f64",
             steps=100, dt=0.1, lam=1.0),
        # A small lattice stepped by the kernel the library takes by itself: one launch per step.
        dict(name="small_48x40x36_f32k", kind="leapfrog", nx=48, ny=40, nz=36, ncomp=1, prec="f32k", steps=50,
             dt=0.05, lam=1.0, tuned=False, field="gauss"),
        # The plain FP64 path of the 256^3 complex workload.
        dict(name="leapfrog_256_complex_f64", kind="leapfrog", nx=256, ny=256, nz=256, ncomp=2, prec="f64", steps=8,
             dt=0.05, lam=1.0, tuned=False, field="gauss"),
        # Diagnostics at every step of a production FP64 run on a lattice that is no power of two:
        # one launch per step with its energy.
        dict(name="energy_every_step_180x150x126_complex_f64", kind="step_energy", nx=180, ny=150, nz=126, ncomp=2,
             prec="f64", steps=10, dt=0.05, lam=1.0),
        # A lattice with odd sides, whose rows are no whole vectors: the kernel for any shape.
        dict(name="odd_257x193x161_f32k", kind="leapfrog", nx=257, ny=193, nz=161, ncomp=1, prec="f32k", steps=16,
             dt=0.05, lam=1.0, tuned=False, field="gauss"),
        # The large FP32 + Kahan real workload: Gaussian random field with a k^-2 spectrum, tuned
        # temporal blocking.  The largest case.
        dict(name="tuned_1024_grf_f32k", kind="leapfrog", nx=1024, ny=1024, nz=1024, ncomp=1, prec="f32k", steps=24,
             dt=0.05, lam=1.0, tuned=True, field="grf"),
        # The complex FP32 + Kahan workload (the benchmark's, at a size of which several states fit).
        dict(name="tuned_512_complex_f32k", kind="leapfrog", nx=512, ny=512, nz=512, ncomp=2, prec="f32k", steps=24,
             dt=0.05, lam=1.0, tuned=True, field="gauss"),
        # An O(4) field.
        dict(name="tuned_256_o4_f32k", kind="leapfrog", nx=256, ny=256, nz=256, ncomp=4, prec="f32k", steps=24,
             dt=0.05, lam=1.0, tuned=True, field="gauss"),
        # 64 independent lattices of uneven sizes, advanced together.
        dict(name="ensemble_64_f32k", kind="ensemble", count=64, ncomp=1, prec="f32k", steps=50, dt=0.05),
        # The FP64 energy of an FP32 field: what a long FP32 run is checked by.
        dict(name="energy_512_f32k", kind="energy", nx=512, ny=512, nz=512, ncomp=1, prec="f32k", dt=0.05, lam=1.0),
        # The paper's benchmarked field operation: symmetric differences of a three-component field
        # along each dimension.
        dict(name="gradient_256_c3_f32", kind="gradient", nx=256, ny=256, nz=256, ncomp=3, prec="f32"),
        # The power spectrum that initial conditions and results are checked by.
        dict(name="spectrum_256_f32", kind="spectrum", n=256, ncomp=1, prec="f32", nbins=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, ncomp, most):
    """Three sides, each spread over its logarithm, odd and even, with at most `most` values in all;
    half of them with rows of whole vectors, as most production lattices have."""
    while True:
        n = [_log_int(rng, 12, 640) for _ in range(3)]
        if rng.random() < 0.5:
            n = [max(16, 8 * round(v / 8)) for v in n]
        if 4096 <= n[0] * n[1] * n[2] * ncomp <= most:
            return dict(zip(SIZES, n))


def draw(rng):
    kind = rng.choice(["leapfrog"] * 4 + ["step_energy"] * 2 + ["energy", "ensemble", "gradient", "spectrum"])
    prec = rng.choice(["f64", "f64", "f32k", "f32k", "f32"])
    ncomp = rng.choice([1, 1, 2, 2, 3, 4, 5, 6])
    dt, lam = round(rng.uniform(0.02, 0.1), 3), round(rng.uniform(0.5, 2.0), 3)
    if kind == "leapfrog":
        # lf2_tune has something to choose from for these; other fields it may refuse, by their sides
        tunable = ncomp <= 2 or (ncomp != 5 and prec != "f64")
        return dict(kind=kind, **_sides(rng, ncomp, 1 << 25), ncomp=ncomp, prec=prec, steps=rng.randint(1, 24), dt=dt,
                    lam=lam, tuned=tunable and rng.random() < 0.6, field="gauss")
    if kind == "step_energy":
        return dict(kind=kind, **_sides(rng, ncomp, 1 << 23), ncomp=ncomp, prec=prec, steps=_log_int(rng, 2, 60), dt=dt,
                    lam=lam)
    if kind == "energy":
        return dict(kind=kind, **_sides(rng, ncomp, 1 << 27), ncomp=ncomp, prec=prec, dt=dt, lam=lam)
    if kind == "ensemble":
        return dict(kind=kind, count=_log_int(rng, 4, 64), ncomp=rng.choice([1, 1, 2]),
                    prec=rng.choice(["f32k", "f32k", "f32"]), steps=rng.randint(4, 25), dt=dt)
    if kind == "gradient":
        return dict(kind=kind, **_sides(rng, ncomp, 1 << 27), ncomp=ncomp, prec=prec)
    return dict(kind=kind, n=_log_int(rng, 32, 384), ncomp=rng.choice([1, 2]), prec=rng.choice(["f64", "f32"]),
                nbins=rng.choice([32, 64, 128]))


# ------------------------------------------------------------------------------- inputs
def _dtype(prec):
    return torch.float64 if prec == "f64" else torch.float32


def _normal(shape, sigma, seed, dtype):
    """FP64 draws, rounded once for FP32 storage."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    out = torch.empty(shape, dtype=dtype, device="cuda")
    flat = out.view(-1)
    for at in range(0, flat.numel(), 1 << 26):
        part = flat[at:at + (1 << 26)]
        part.copy_(torch.randn(part.shape, generator=gen, dtype=torch.float64, device="cuda").mul_(sigma))
    return out


def _fields(case, seed):
    """phi_0 and pi_0, (nz, ny, nx, ncomp).  pi_0 is small noise where the state is one of a run
    in progress (energies), else 0."""
    shape = (case["nz"], case["ny"], case["nx"], case["ncomp"])
    dtype = _dtype(case["prec"])
    if case.get("field") == "grf":
        phi = inputs.grf_field_device(case["nx"], sigma=SIGMA, seed=seed, dtype=dtype)
    else:
        phi = _normal(shape, SIGMA, seed, dtype)
    pi = _normal(shape, SIGMA, seed + 7919, dtype) if case["kind"] == "energy" else torch.zeros_like(phi)
    return phi, pi


def _members(case, seed):
    """(side, lambda) of an ensemble's lattices: the sizes belong to the case, the couplings to the seed."""
    sides = [s for s, _, _ in inputs.ensemble_members(case["count"])]
    lams = [lam for _, lam, _ in inputs.ensemble_members(case["count"], seed=seed)]
    return list(zip(sides, lams))


def _params(case, lam=None):
    return lf2.params(dx=DX, dt=case["dt"], lam=case["lam"] if lam is None else lam, eta=ETA, m2=0.0)


class State:
    """A lattice with its fields on torch buffers."""

    def __init__(self, case):
        self.case = case
        self.lats, self.handles, self.ens, self.own = [], [], None, []

    def lattice(self, sizes):
        self.lats.append(lf2.lf2_lattice_create(sizes))
        return self.lats[-1]

    def field(self, lat, buffers):
        f = lf2.lf2_field_wrap(lat, self.case["ncomp"], lf2.PRECISIONS[self.case["prec"]],
                               [b.data_ptr() for b in buffers])
        self.handles.append(f)
        return f

    def __del__(self):
        if self.ens is not None:
            lf2.lf2_ensemble_destroy(self.ens)
        for f in self.handles:
            lf2.lf2_field_free(f)
        for lat in self.lats:
            lf2.lf2_lattice_destroy(lat)


def _phi_buffers(case, phi):
    """Value and back buffer, and with the compensated drift the compensation and its back buffer."""
    bufs = [phi, torch.empty_like(phi)]
    if case["prec"] == "f32k":
        bufs += [torch.zeros_like(phi), torch.zeros_like(phi)]
    return bufs


def _current(f, which, buffers):
    """The one of the lent buffers that holds the field's current values (which = 0) or compensation (2)."""
    at = lf2.lf2_field_buffer(f, which)
    return next(b for b in buffers if b.data_ptr() == at)


def _evolved(s):
    out = {"phi": _current(s.phi, 0, s.phi_bufs[:2]), "pi": _current(s.pi, 0, s.pi_bufs)}
    if s.case["prec"] == "f32k":
        out["comp"] = _current(s.phi, 2, s.phi_bufs[2:])
    return out


def prepare(case, seed):
    lf2.load()
    s = State(case)
    kind = case["kind"]
    stream = torch.cuda.current_stream()
    if kind == "ensemble":
        members = _members(case, seed)
        total = sum(n ** 3 for n, _ in members) * case["ncomp"]
        s.phi_bufs = _phi_buffers(case, _normal((total,), SIGMA, seed, torch.float32))
        s.pi_bufs = [torch.zeros_like(s.phi_bufs[0]), torch.empty_like(s.phi_bufs[0])]
        phis, pis, plist, at = [], [], [], 0
        for n, lam in members:
            count = n ** 3 * case["ncomp"]
            lat = s.lattice((n, n, n))
            phis.append(s.field(lat, [b[at:at + count] for b in s.phi_bufs]))
            pis.append(s.field(lat, [b[at:at + count] for b in s.pi_bufs]))
            plist.append(_params(case, lam))
            lf2.lf2_leapfrog_init(phis[-1], pis[-1], plist[-1], stream)
            at += count
        s.phi, s.pi = phis[0], pis[0]  # every member's buffers swap together
        s.ens = lf2.lf2_ensemble_create(phis, pis, plist)
        return s
    if kind == "spectrum":
        n = case["n"]
        s.phi_bufs = [_normal((n, n, n, case["ncomp"]), SIGMA, seed, _dtype(case["prec"]))]
        s.phi = s.field(s.lattice((n, n, n)), s.phi_bufs)
        return s
    lat = s.lattice(tuple(case[k] for k in SIZES))
    if kind == "gradient":
        phi, _ = _fields(case, seed)
        s.phi_bufs = [phi]
        s.phi = s.field(lat, s.phi_bufs)
        s.out = [torch.empty_like(phi) for _ in range(3)]
        s.dst = [s.field(lat, [o]) for o in s.out]
        return s
    phi, pi = _fields(case, seed)
    s.phi_bufs, s.pi_bufs = _phi_buffers(case, phi), [pi, torch.empty_like(pi)]
    s.phi, s.pi = s.field(lat, s.phi_bufs), s.field(lat, s.pi_bufs)
    s.params = _params(case)
    lf2.lf2_leapfrog_init(s.phi, s.pi, s.params, stream)
    if kind == "leapfrog" and case["tuned"]:
        lf2.lf2_tune(s.phi, s.pi, s.params, stream=stream)  # kept by the library for this shape
    if kind in ("energy", "step_energy"):
        s.rec = torch.zeros((case.get("steps", 1), 16), dtype=torch.float64, device="cuda")
    return s


def run(s):
    case, kind = s.case, s.case["kind"]
    stream = torch.cuda.current_stream()
    if kind == "leapfrog":
        lf2.lf2_leapfrog(s.phi, s.pi, s.params, case["steps"], stream)
        return _evolved(s)
    if kind == "step_energy":
        lf2.lf2_leapfrog_energy(s.phi, s.pi, s.params, case["steps"], s.rec.data_ptr(), stream)
        return {**_evolved(s), "records": s.rec}
    if kind == "energy":
        lf2.lf2_energy_device(s.phi, s.pi, s.params, s.rec.data_ptr(), stream)
        return {"record": s.rec}
    if kind == "ensemble":
        lf2.lf2_ensemble_run(s.ens, case["steps"], stream)
        return _evolved(s)
    if kind == "gradient":
        for dim in range(3):
            lf2.lf2_field_derivative(s.phi, s.dst[dim], dim, DX, stream)
        return list(s.out)
    power, kmean, count = lf2.lf2_power_spectrum(s.phi, comp=-1, nbins=case["nbins"], dx=DX, stream=stream)
    return {"power": power, "kmean": kmean, "count": count}


# ------------------------------------------------------------------------ compulsory work
def work(case):
    """Bytes: the state read once and written once.  Flops: the arithmetic of the method per
    site, an fma as two."""
    kind, size = case["kind"], 8 if case["prec"] == "f64" else 4
    c = case["ncomp"]
    # |phi|^2 and the potential's coefficient; per component the Laplacian (6), force (4), kick and
    # drift (4) and the compensation (3)
    per_site = 2 * c + 3 + c * (14 + (3 if case["prec"] == "f32k" else 0))
    # energy: synchronised momentum (10), its square (2), three squared differences (9), sums (3)
    per_energy = 2 * c + 6 + 24 * c
    if kind == "spectrum":
        sites = case["n"] ** 3
        return {"bytes": sites * c * size, "flops": c * (2.5 * sites * math.log2(sites) + 4 * sites)}
    if kind == "ensemble":
        sites = sum(n ** 3 for n, _ in _members(case, 0))
    else:
        sites = case["nx"] * case["ny"] * case["nz"]
    values = sites * c
    if kind == "gradient":
        return {"bytes": values * size * 4, "flops": values * 6}
    if kind == "energy":
        return {"bytes": values * size * 2, "flops": sites * per_energy}
    arrays = 6 if case["prec"] == "f32k" else 4
    flops = sites * case["steps"] * (per_site + (per_energy if kind == "step_energy" else 0))
    return {"bytes": values * size * arrays, "flops": flops}


# -------------------------------------------------------------- the same in 64 bits, in torch
def _neighbours(phi):
    """phi(x + i) and phi(x - i) for i = x, y, z of a (nz, ny, nx, ncomp) array."""
    return [(torch.roll(phi, -1, d), torch.roll(phi, 1, d)) for d in (2, 1, 0)]


def _force(phi, lam):
    s2 = (phi * phi).sum(-1, keepdim=True)
    f = phi * (-lam * (s2 - ETA * ETA) - 6.0 / DX ** 2)
    for d in (2, 1, 0):
        f += torch.roll(phi, -1, d)
        f += torch.roll(phi, 1, d)
    return f


def _record(phi, pi, dt, lam):
    """lf2_energy_t: kinetic, gradient, potential, total, then sums and sums of squares, six each."""
    pin = pi + 0.5 * dt * _force(phi, lam)
    kin = 0.5 * float((pin * pin).sum())
    grad = 0.0
    for d in (2, 1, 0):
        e = torch.roll(phi, -1, d) - phi
        grad += 0.5 / DX ** 2 * float((e * e).sum())
        del e
    w = (phi * phi).sum(-1) - ETA * ETA
    pot = 0.25 * lam * float((w * w).sum())
    c = phi.shape[-1]
    sums = [float(phi[..., a].sum()) for a in range(c)] + [0.0] * (6 - c)
    squares = [float((phi[..., a] ** 2).sum()) for a in range(c)] + [0.0] * (6 - c)
    return [kin, grad, pot, kin + grad + pot] + sums + squares


def _evolve(phi, pi, steps, dt, lam, records=None):
    pi -= 0.5 * dt * _force(phi, lam)  # the half kick of lf2_leapfrog_init
    for _ in range(steps):
        if records is not None:
            records.append(_record(phi, pi, dt, lam))
        pi += dt * _force(phi, lam)
        phi += dt * pi
    return phi, pi


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        members = _members(case, seed)
        total = sum(n ** 3 for n, _ in members) * case["ncomp"]
        phi = _normal((total,), SIGMA, seed, torch.float32).double()
        pi, at = torch.zeros_like(phi), 0
        for n, lam in members:
            count = n ** 3 * case["ncomp"]
            shape = (n, n, n, case["ncomp"])
            _evolve(phi[at:at + count].view(shape), pi[at:at + count].view(shape), case["steps"], case["dt"], lam)
            at += count
        out = {"phi": phi, "pi": pi}
        return {**out, "comp": None} if case["prec"] == "f32k" else out
    if kind == "spectrum":
        n, nbins = case["n"], case["nbins"]
        phi = _normal((n, n, n, case["ncomp"]), SIGMA, seed, _dtype(case["prec"])).double()
        power = sum(torch.fft.fftn(phi[..., a]).abs().square_() for a in range(case["ncomp"])) / n ** 3
        m = torch.fft.fftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64).round().long()
        m2 = m[:, None, None] ** 2 + m[None, :, None] ** 2 + m[None, None, :] ** 2
        root = m2.double().sqrt()
        shell = root.long()  # exact: m2 is far below 2^52
        keep = shell < nbins
        shell = shell[keep]
        count = torch.bincount(shell, minlength=nbins).double()
        psum = torch.bincount(shell, weights=power[keep], minlength=nbins)
        ksum = torch.bincount(shell, weights=root[keep], minlength=nbins) * (2 * math.pi / (n * DX))
        some = count.clamp_min(1.0)
        return {"power": (psum / some).cpu().numpy(), "kmean": (ksum / some).cpu().numpy(),
                "count": count.cpu().numpy().astype(np.float64)}
    if kind == "gradient":
        phi = _fields(case, seed)[0].double()
        return [(up - dn) * (0.5 / DX) for up, dn in _neighbours(phi)]
    phi, pi = (f.double() for f in _fields(case, seed))
    if kind == "energy":
        pi -= 0.5 * case["dt"] * _force(phi, case["lam"])
        if case["prec"] != "f64":
            pi = pi.float().double()  # the state holds the half-kicked momentum in FP32
        return {"record": torch.tensor([_record(phi, pi, case["dt"], case["lam"])], dtype=torch.float64)}
    records = [] if kind == "step_energy" else None
    phi, pi = _evolve(phi, pi, case["steps"], case["dt"], case["lam"], records)
    out = {"phi": phi, "pi": pi}
    if case["prec"] == "f32k":
        out["comp"] = None
    if records is not None:
        out["records"] = torch.tensor(records, dtype=torch.float64)
    return out
