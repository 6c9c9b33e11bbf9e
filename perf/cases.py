"""The work that users of this library have it do, as measurable cases.

A case is one simulation in progress: ``prepare`` builds the lattice (or batch) and its
initial state from a seed, ``run`` advances it by the steps between two records and reads
the record through the public API, the way the experiments, the benchmark and the server
do, and returns it whole. A second ``run`` goes on from where the first stopped.

Sizes are this repository's own (its workloads, tests, benchmark and profiles) or, in
``draw``, spread over the ranges that they span. ``exact`` evolves the same initial
densities in FP64 with plain torch.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1701_03637_gb300 as sc
from paper_1701_03637_gb300.ncomp import NLattice

Q = 19
# the library's direction order (include/sc_lbm.h: rest, +-x, +-y, +-z, the diagonals in
# opposite pairs); only the populations of the N-component case depend on it
E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
     (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
     (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
W = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
SIZE = {"f32": 4, "f16": 2, "bf16": 2, "f16s": 2}
MOST_UPDATES = 512 ** 3 * 20  # site updates of the largest listed case


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the planar film of Sec. III B: thousands of short calls of a 2,048-site lattice,
        # the interface position and the evaporated mass recorded after each
        dict(name="film_4x4x128", kind="film", nx=4, ny=4, nz=128, storage="f32", steps=100),
        # the diffusion column of Sec. III A watched closely: a few steps, then the flux profile
        dict(name="column_4x4x125", kind="column", nx=4, ny=4, nz=125, storage="f32", steps=10),
        # a droplet of the precision study and of the tests
        dict(name="droplet_64", kind="droplet", nx=64, ny=64, nz=64, storage="f32", layout="two", sink="planar",
             tune=False, steps=100),
        # the benchmark's 128^3 line, tuned as the benchmark tunes it
        dict(name="droplet_128", kind="droplet", nx=128, ny=128, nz=128, storage="f32", layout="two", sink="planar",
             tune=True, steps=100),
        # the paper's own droplet runs (Sec. III C): 256^3 with the spherical sink
        dict(name="droplet_256_sphere", kind="droplet", nx=256, ny=256, nz=256, storage="f32", layout="two",
             sink="sphere", tune=False, steps=50),
        # FP16 offset storage, two lattices
        dict(name="droplet_256_f16", kind="droplet", nx=256, ny=256, nz=256, storage="f16", layout="two",
             sink="planar", tune=False, steps=50),
        # the benchmark's default line: 512^3 updated in place
        dict(name="droplet_512_aa", kind="droplet", nx=512, ny=512, nz=512, storage="f32", layout="aa",
             sink="planar", tune=False, steps=20),
        # BF16 offset storage in place
        dict(name="droplet_256_aa_bf16", kind="droplet", nx=256, ny=256, nz=256, storage="bf16", layout="aa",
             sink="planar", tune=False, steps=50),
        # extents that no tile or vector width divides, a wall, self couplings (the multiphase
        # model) and two relaxation times
        dict(name="ragged_walls", kind="ragged", nx=151, ny=93, nz=67, storage="f32", layout="two", steps=100),
        # the 64-lattice ensemble of the benchmark: one batched launch per step, tuned
        dict(name="ensemble_64", kind="ensemble", members=64, lo=32, hi=96, cubic=False, storage="f32", tune=True,
             steps=100),
        # what the server does between two records: FP16 cubes of the request stream
        dict(name="served_16_f16", kind="served", members=16, lo=32, hi=160, cubic=True, storage="f16", tune=False,
             steps=100),
        # three components, from one checkpoint to the next
        dict(name="three_components_64", kind="ncomp", nx=64, ny=64, nz=64, ncomp=3, steps=1000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["film", "column", "droplet", "droplet", "droplet", "droplet", "ragged", "ensemble", "served",
                       "ncomp"])
    storage = rng.choice(["f32", "f32", "f16", "bf16", "f16s"])
    if kind in ("film", "column"):
        n = _log_int(rng, 4, 24)
        return dict(kind=kind, nx=n, ny=n, nz=_log_int(rng, 64, 256), storage="f32",
                    steps=_log_int(rng, 50, 200) if kind == "film" else _log_int(rng, 5, 50))
    if kind == "droplet":
        n = _log_int(rng, 32, 384)
        if rng.random() < 0.6:  # edges are usually round numbers
            n = max(32, n // 16 * 16)
        nx, ny, nz = n, n, n
        if rng.random() < 0.3:  # a box that is not a cube
            ny, nz = max(32, int(n * rng.uniform(0.6, 1.0))), max(32, int(n * rng.uniform(0.6, 1.0)))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, storage=storage, layout=rng.choice(["two", "two", "aa"]),
                    sink=rng.choice(["planar", "planar", "sphere"]), tune=rng.random() < 0.3,
                    steps=max(10, min(100, MOST_UPDATES // (2 * nx * ny * nz))))
    if kind == "ragged":
        nx, ny, nz = (_log_int(rng, 24, 220) for _ in range(3))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, storage=storage, layout=rng.choice(["two", "aa"]),
                    steps=_log_int(rng, 50, 100))
    if kind == "ncomp":
        nx, ny, nz = (_log_int(rng, 24, 80) for _ in range(3))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, ncomp=rng.choice([2, 3, 3, 4]), steps=_log_int(rng, 500, 1000))
    m = _log_int(rng, 8, 48)
    if kind == "ensemble":
        return dict(kind=kind, members=m, lo=32, hi=96, cubic=False, storage="f32", tune=rng.random() < 0.5,
                    steps=_log_int(rng, 50, 100))
    return dict(kind=kind, members=max(4, m // 3), lo=32, hi=160, cubic=True, storage=rng.choice(["f16", "f32"]),
                tune=False, steps=100)


# ------------------------------------------------------------------ initial states and parameters

def _rng(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _two_phase(inside, hi, lo, gen, noise=1e-4):
    """(rho^r, rho^b) [2, nz, ny, nx] FP32: hi / lo inside, lo / hi outside, plus noise."""
    rho = torch.stack([torch.where(inside, hi, lo), torch.where(inside, lo, hi)]).float()
    return rho + noise * (2.0 * torch.rand(rho.shape, generator=gen, device="cuda") - 1.0)


def _ball(nx, ny, nz, radius, gen):
    """A ball near the middle of the box (its centre moves by up to two sites with the seed)."""
    c = (torch.rand(3, generator=gen, device="cuda") * 4.0 - 2.0).tolist()
    x = (torch.arange(nx, device="cuda") - nx / 2.0 - c[0]) ** 2
    y = (torch.arange(ny, device="cuda") - ny / 2.0 - c[1]) ** 2
    z = (torch.arange(nz, device="cuda") - nz / 2.0 - c[2]) ** 2
    return (z[:, None, None] + y[None, :, None] + x[None, None, :]) < radius * radius


def _slab(nx, ny, nz, top):
    return (torch.arange(nz, device="cuda") < top)[:, None, None].expand(nz, ny, nx)


def _single(case, seed):
    """Parameters and initial densities of a one-lattice case."""
    kind, nx, ny, nz = case["kind"], case["nx"], case["ny"], case["nz"]
    gen = _rng(seed)
    p = dict(nx=nx, ny=ny, nz=nz, tau_r=1.0, tau_b=1.0, G=3.6, rho_H=0.03, storage=case["storage"])
    if kind == "film":  # a wall of thickness 2, the film above it, the sink plane at the far end
        p.update(geometry=1, sink_z0=nz - 1, sink_layers=1, wall_z0=0, wall_thickness=2, rho_H=0.02)
        return p, _two_phase(_slab(nx, ny, nz, nz // 4), 0.7, 0.04, gen)
    if kind == "column":  # component r diffuses in from the boundary plane z = 0
        p.update(geometry=1, sink_z0=0, sink_layers=1, wall_z0=nz - 2, wall_thickness=2, rho_H=0.001)
        rho = torch.zeros(2, nz, ny, nx, device="cuda")
        rho[1] = 0.7 + 1e-4 * (2.0 * torch.rand(nz, ny, nx, generator=gen, device="cuda") - 1.0)
        return p, rho
    if kind == "ragged":  # a multiphase mixture between walls
        p.update(layout=case["layout"], G=3.4, G_rr=-1.1, G_bb=0.5, tau_r=0.9, tau_b=1.15, geometry=1,
                 sink_z0=nz - 1, sink_layers=1, wall_z0=0, wall_thickness=1)
        return p, _two_phase(_ball(nx, ny, nz, 0.3 * min(nx, ny, nz), gen), 0.7, 0.04, gen)
    p.update(layout=case["layout"])
    if case["sink"] == "sphere":
        p.update(geometry=2, sphere_cx=nx / 2.0, sphere_cy=ny / 2.0, sphere_cz=nz / 2.0,
                 R_H=min(nx, ny, nz) / 2.0 - 2.0, rho_H=0.02)
        return p, _two_phase(_ball(nx, ny, nz, 0.25 * min(nx, ny, nz), gen), 0.7, 0.04, gen)
    p.update(geometry=1, sink_z0=nz - 1, sink_layers=2)
    return p, _two_phase(_ball(nx, ny, nz, 0.1875 * min(nx, ny, nz), gen), 1.0, 0.03, gen)


def _members(case):
    """Parameters of an ensemble's lattices: its make-up belongs to the case, not to the seed."""
    r = random.Random(1000003 * case["members"] + int(case["hi"]))
    edge = lambda: _log_int(r, case["lo"], case["hi"])  # noqa: E731
    out = []
    for k in range(case["members"]):
        nx = edge()
        ny, nz = (nx, nx) if case["cubic"] else (edge(), edge())
        tau = r.uniform(0.8, 1.2)
        p = dict(nx=nx, ny=ny, nz=nz, tau_r=tau, tau_b=tau, G=r.uniform(3.2, 3.8), rho_H=0.03,
                 storage=case["storage"], geometry=1, sink_z0=nz - 1)
        if k % 2 == 0:
            p.update(sink_layers=1, wall_z0=0, wall_thickness=2)
        else:
            p.update(sink_layers=2)
        out.append((p, r.uniform(0.2, 0.35)))
    return out


def _member_rho(k, p, share, gen):
    nx, ny, nz = p["nx"], p["ny"], p["nz"]
    inside = _slab(nx, ny, nz, max(3, nz // 4)) if k % 2 == 0 else _ball(nx, ny, nz, share * min(nx, ny, nz), gen)
    return _two_phase(inside, 1.0, 0.03, gen)


def _components(case, seed):
    """tau, couplings and initial densities [c, nz, ny, nx] of an N-component case: a droplet of
    component 0 in component 1, the others dissolved."""
    nx, ny, nz, nc = case["nx"], case["ny"], case["nz"], case["ncomp"]
    gen = _rng(seed)
    two = _two_phase(_ball(nx, ny, nz, 0.1875 * min(nx, ny, nz), gen), 0.7, 0.04, gen)
    rest = 0.1 + 1e-4 * (2.0 * torch.rand(nc - 2, nz, ny, nx, generator=gen, device="cuda") - 1.0)
    g = [[0.0 if a == b else (3.6 if a + b == 1 else 1.0) for b in range(nc)] for a in range(nc)]
    return [1.0] * nc, g, torch.cat([two, rest])


# ------------------------------------------------------------------ prepare and run

def _fill(lat, rho):
    host = rho.cpu()
    lat.init_fields_from(host[0], host[1])


def prepare(case, seed):
    if case["kind"] == "ncomp":
        tau, g, rho = _components(case, seed)
        lat = NLattice(case["nx"], case["ny"], case["nz"], tau, g)
        lat.init_fields(rho.cpu().numpy())
        return dict(case=case, lat=lat)
    if case["kind"] in ("ensemble", "served"):
        gen, members = _rng(seed), _members(case)
        batch = sc.Batch(sum(sc.required_bytes(p) + 256 for p, _ in members) + (1 << 20), case["storage"])
        lats, out = [], []
        for k, (p, share) in enumerate(members):
            _, lat = batch.add(p)
            _fill(lat, _member_rho(k, p, share, gen))
            lats.append(lat)
            out.append(torch.empty(2, *lat.shape, device="cuda"))
        if case["tune"]:
            batch.tune()
        return dict(case=case, batch=batch, lats=lats, out=out)
    p, rho = _single(case, seed)
    lat = sc.Lattice(p)
    _fill(lat, rho)
    if case.get("tune"):
        lat.tune(20)
    return dict(case=case, lat=lat, out=torch.empty(2, *lat.shape, device="cuda"))


def run(state):
    case, steps = state["case"], state["case"]["steps"]
    if case["kind"] == "ncomp":
        state["lat"].step(steps)
        return state["lat"].read_populations()
    if case["kind"] in ("ensemble", "served"):
        state["batch"].step(steps)
        fields = [lat.read_fields_device(o) for lat, o in zip(state["lats"], state["out"])]
        if case["kind"] == "ensemble":
            return fields
        series = [lat.diagnostics() for lat in state["lats"]]
        keys = ("mass_r", "evaporated_mass", "flux_last", "interface_z", "radius")
        return dict(fields=fields, series=np.array([[d[k] for k in keys] for d in series], np.float32))
    lat = state["lat"]
    lat.step(steps)
    fields = lat.read_fields_device(state["out"])
    if case["kind"] == "film":
        return dict(fields=fields, diagnostics=lat.diagnostics())
    if case["kind"] == "column":
        return dict(fields=fields, flux=lat.flux_profile())
    return fields


# ------------------------------------------------------------------ the work of a pass

def work(case):
    """Each step reads and writes every population of the state once, unless the state
    (one lattice) is small enough to stay on the chip (126 MB of L2), where only the pass
    as a whole has to; the record is written once. Operations per component and site: the
    density and momentum sums (39), the force (36), the relaxation (130)."""
    if case["kind"] in ("ensemble", "served"):
        sites = sum(p["nx"] * p["ny"] * p["nz"] for p, _ in _members(case))
    else:
        sites = case["nx"] * case["ny"] * case["nz"]
    nc = case.get("ncomp", 2)
    state = nc * Q * SIZE[case.get("storage", "f32")] * sites
    moves = case["steps"] if state > 126e6 else 1
    record = nc * Q * 8 * sites if case["kind"] == "ncomp" else 8 * sites
    return dict(bytes=2 * state * moves + record, flops=205.0 * nc * sites * case["steps"])


# ------------------------------------------------------------------ the same in FP64

def _planes(p, nz):
    z = torch.arange(nz, device="cuda")
    return (z >= p.get("wall_z0", 0)) & (z < p.get("wall_z0", 0) + p.get("wall_thickness", 0))


def _sink(p, solid):
    """Sink sites [nz, ny, nx] (broadcastable) or None."""
    nx, ny, nz = p["nx"], p["ny"], p["nz"]
    z = torch.arange(nz, device="cuda")
    if p.get("geometry", 0) == 1:
        m = ((z - p["sink_z0"]) % nz < p["sink_layers"])[:, None, None]
    elif p.get("geometry", 0) == 2:
        ax = lambda n, c: (torch.arange(n, device="cuda", dtype=torch.float64) - c) ** 2  # noqa: E731
        r2 = (ax(nx, p["sphere_cx"])[None, None, :] + ax(ny, p["sphere_cy"])[None, :, None]) + \
            ax(nz, p["sphere_cz"])[:, None, None]
        m = r2 >= p["R_H"] ** 2
    else:
        return None
    return m & ~solid[:, None, None]


def _shift(a, e):
    """a(x - e) (periodic) for [..., z, y, x]."""
    dims = [(d, s) for d, s in ((-1, e[0]), (-2, e[1]), (-3, e[2])) if s]
    return torch.roll(a, [s for _, s in dims], [d for d, _ in dims]) if dims else a


def _evolve(rho0, tau, g, steps, p):
    """`steps` steps of the method from rest populations of rho0 [c, nz, ny, nx], in FP64.
    Returns densities, populations, and the evaporated mass (total, last step)."""
    nc, nz, ny, nx = rho0.shape
    solid = _planes(p, nz)
    walls = bool(solid.any())
    fluid_z = (~solid).double()[:, None, None]
    sink = _sink(p, solid)
    rho = rho0.double() * fluid_z
    rho_h = float(p.get("rho_H", 0.0))

    def reset(rho):
        gone = torch.where(sink, rho[0] - rho_h, 0.0).sum()
        total = rho[0] + rho[1]
        rho[0] = torch.where(sink, rho_h, rho[0])
        rho[1] = torch.where(sink, total - rho_h, rho[1])
        return gone

    if sink is not None:
        reset(rho)
    f = torch.empty(nc, Q, nz, ny, nx, dtype=torch.float64, device="cuda")
    for i in range(Q):
        f[:, i] = W[i] * rho
    om = [1.0 / t for t in tau]
    evaporated, last = torch.zeros((), dtype=torch.float64, device="cuda"), None
    stay = None if sink is None else sink.expand(nz, ny, nx)
    for _ in range(steps):
        psi = (1.0 - torch.exp(-rho)) * fluid_z
        a = torch.zeros(nc, 3, nz, ny, nx, dtype=torch.float64, device="cuda")
        m = torch.zeros_like(a)
        for i in range(1, Q):
            s = _shift(psi, tuple(-v for v in E[i]))
            for d in range(3):
                if E[i][d]:
                    a[:, d].add_(s, alpha=W[i] * E[i][d])
                    m[:, d].add_(f[:, i], alpha=E[i][d])
        den = sum(rho[c] * om[c] for c in range(nc))
        up = sum(m[c] * om[c] for c in range(nc)) / torch.where(den > 0, den, torch.inf)
        del m, den
        for c in range(nc):
            q = torch.where(rho[c] > 0, psi[c] / rho[c], 0.0) * (-tau[c])
            u = up + q * sum(g[c][b] * a[b] for b in range(nc))
            base = 1.0 - 1.5 * (u * u).sum(0)
            for i in range(Q):
                cu = sum(E[i][d] * u[d] for d in range(3)) if i else torch.zeros_like(base)
                new = (cu * (3.0 + 4.5 * cu) + base) * rho[c] * (W[i] * om[c]) + (1.0 - om[c]) * f[c, i]
                f[c, i] = new if stay is None else torch.where(stay, f[c, i], new)
                del cu, new
            del u, base, q
        del a, up, psi
        f[:, 0] *= fluid_z
        for i in range(1, Q, 2):  # opposite pairs
            fwd, bwd = _shift(f[:, i], E[i]), _shift(f[:, i + 1], E[i + 1])
            if walls and E[i][2]:
                up_src = torch.roll(solid, E[i][2])  # plane z - e_z is solid
                dn_src = torch.roll(solid, -E[i][2])
                fwd = torch.where(up_src[:, None, None], f[:, i + 1], fwd)
                bwd = torch.where(dn_src[:, None, None], f[:, i], bwd)
            f[:, i], f[:, i + 1] = fwd * fluid_z, bwd * fluid_z
            del fwd, bwd
        rho = f.sum(1)
        if sink is not None:
            last = reset(rho)
            evaporated += last
            for i in range(Q):
                f[:, i] = torch.where(stay, W[i] * rho, f[:, i])
    return rho, f, evaporated, last


def _matrix(p):
    return [[p.get("G_rr", 0.0), p["G"]], [p["G"], p.get("G_bb", 0.0)]]


def _flux(rho, f, p):
    """Plane means of rho^r (U^r - U) (Eqs. (flux), (velw) at tau = 1), 0 at sinks and walls."""
    nz = rho.shape[1]
    solid = _planes(p, nz)
    fluid = ~solid[:, None, None] & ~_sink(p, solid)
    psi = (1.0 - torch.exp(-rho)) * (~solid).double()[:, None, None]
    total = rho[0] + rho[1]
    out = torch.zeros(3, nz, dtype=torch.float64, device="cuda")
    for d in range(3):
        a = sum(W[i] * E[i][d] * _shift(psi, tuple(-v for v in E[i])) for i in range(1, Q) if E[i][d])
        m = sum(E[i][d] * f[:, i] for i in range(1, Q) if E[i][d])
        F = [-psi[0] * p["G"] * a[1], -psi[1] * p["G"] * a[0]]
        U = (m[0] + m[1] + 0.5 * (F[0] + F[1])) / total
        Ur = (m[0] + F[0] + rho[0] * (m[0] + m[1]) / total) / (2.0 * rho[0])
        j = torch.where(fluid.expand_as(U) & (rho[0] > 0), rho[0] * (Ur - U), 0.0)
        out[d] = j.mean((1, 2))
    return out


def _observables(rho, evaporated, last, p):
    """The floating observables of a diagnostics record (None for the integers)."""
    nz = rho.shape[1]
    solid = _planes(p, nz)
    phi = (rho[0] - rho[1]).mean((1, 2)).tolist()
    hard = solid.tolist()
    z0 = p.get("wall_z0", 0) + p.get("wall_thickness", 0) if any(hard) else 0
    at = -1.0
    for z in range(z0, nz - 1):
        if not hard[z] and not hard[z + 1] and phi[z] > 0.0 >= phi[z + 1]:
            at = z + phi[z] / (phi[z] - phi[z + 1])
            break
    v = float(((rho[0] > rho[1]) & ~solid[:, None, None]).sum())
    return dict(step=None, mass_r=float(rho[0].sum()), mass_b=float(rho[1].sum()), evaporated_mass=float(evaporated),
                flux_last=float(last), interface_z=at, radius=(3.0 * v / (4.0 * math.pi)) ** (1.0 / 3.0),
                droplet_sites=None, status=None)


def exact(case, seed):
    if case["kind"] == "ncomp":
        tau, g, rho = _components(case, seed)
        return _evolve(rho, tau, g, case["steps"], case)[1].cpu().numpy()
    if case["kind"] in ("ensemble", "served"):
        gen, out = _rng(seed), []
        for k, (p, share) in enumerate(_members(case)):
            rho = _member_rho(k, p, share, gen)
            out.append(_evolve(rho, [p["tau_r"], p["tau_b"]], _matrix(p), case["steps"], p)[0])
        # the records of reduced-precision runs drift with the storage's rounding: fields only
        return out if case["kind"] == "ensemble" else dict(fields=out, series=None)
    p, rho = _single(case, seed)
    rho, f, evaporated, last = _evolve(rho, [p["tau_r"], p["tau_b"]], _matrix(p), case["steps"], p)
    if case["kind"] == "film":
        return dict(fields=rho, diagnostics=_observables(rho, evaporated, last, p))
    if case["kind"] == "column":
        return dict(fields=rho, flux=_flux(rho, f, p).cpu().numpy())
    return rho
