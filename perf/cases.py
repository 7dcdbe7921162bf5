"""Workloads of the library as a program that uses it runs them, for timing.

A case is one lattice (or a batch of lattices in one handle), a storage
precision and a number of time steps.  A pass of most cases advances the handle
by that many steps and reads the state back into device buffers the caller
owns (cell types, fill levels, density, velocity) with, for single small
lattices, the bubble table: what a program does that follows a simulation.  The
reduced storage forms hand their floating results on in FP32.  Two cases do
something else: `run` is a whole short simulation from the creation of the
handle to its end, `label` the allocation-free labelling of one lattice.

The inputs have the shapes of the repository's own workloads (static bubble,
gas thread, orifice, bubble populations, foam), made on the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_1604_01632_gb300 import fsl

DEV = "cuda" if torch.cuda.is_available() else "cpu"
LIQ, IFC, GAS, OBS, LID = 0, 1, 2, 3, 4
F64 = torch.float64

# D3Q19 in the library's order
C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
     (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
     (0, -1, 1)]
W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
OPP = [0] + [a + 1 if a % 2 else a - 1 for a in range(1, 19)]

# steps every handle has behind it when a pass begins: the library tunes its
# kernels on the first steps of a shape, and a program's steps come after that
WARM_STEPS = 20

BYTES = {"fp64": 8, "fp32": 4, "f16s": 2, "bf16s": 2}


# --------------------------------------------------------------------- cases

def _case(name, scene, nx, ny, nz, precision, steps, domains=1):
    return {"name": name, "scene": scene, "nx": nx, "ny": ny, "nz": nz, "precision": precision, "steps": steps,
            "domains": domains}


def listed():
    return [
        # the Laplace test: one bubble at rest in a 32^3 box, where launches and barriers count
        _case("bubble32_fp64", "bubble", 32, 32, 32, "fp64", 50),
        # a small ragged box of moving bubbles: odd sides, conversions, merges and splits
        _case("bubbles61_fp32", "bubbles", 61, 47, 53, "fp32", 50),
        # capillary breakup of a gas thread between walls (the 1 M-cell workload of the benchmark)
        _case("thread256_f16s", "thread", 256, 64, 64, "f16s", 50),
        # bubble formation at an orifice: plate, gravity, draining reservoir, atmosphere
        _case("orifice128_fp32", "orifice", 128, 128, 256, "fp32", 20),
        # a batch of bubble-population domains in one handle (the benchmark's batch)
        _case("population64_f16s", "population", 32, 48, 96, "f16s", 20, 64),
        # a batch of small domains with odd sides
        _case("population24_odd_bf16s", "population", 21, 33, 49, "bf16s", 50, 24),
        # the headline foam
        _case("foam512_f16s", "foam", 512, 512, 512, "f16s", 10),
        # the plain FP32 baseline of the metric on a medium foam
        _case("foam256_fp32", "foam", 256, 256, 256, "fp32", 10),
        # a foam of odd sides in BF16 storage
        _case("foam243_bf16s", "foam", 243, 251, 247, "bf16s", 10),
        # the parity path: FP64 storage and arithmetic
        _case("foam160_fp64", "foam", 160, 160, 160, "fp64", 5),
        # a whole short run as a parameter sweep does it: create, upload, step, read back, destroy
        _case("run128_f16s", "run", 128, 128, 128, "f16s", 50),
        # labelling for a caller that cannot allocate, on the largest lattice it takes
        _case("label128", "label", 128, 128, 128, "fp64", 0),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    scene = rng.choice(["foam", "foam", "foam", "bubbles", "population", "thread", "orifice", "bubble", "run", "label"])
    prec = rng.choice(["f16s", "f16s", "fp32", "bf16s", "fp64"])
    steps = rng.randint(10, 60)
    if scene == "foam":
        hi = 176 if prec == "fp64" else 400
        return _drop(_case("", scene, log(96, hi), log(96, hi), log(96, hi), prec, rng.randint(5, 10)))
    if scene == "bubbles":
        return _drop(_case("", scene, log(24, 96), log(24, 96), log(24, 96), prec, steps))
    if scene == "population":
        lo = rng.choice([20, 24, 32])
        return _drop(_case("", scene, lo, lo + rng.randint(4, 24), lo + rng.randint(28, 64), prec, steps,
                           log(4, 12 if prec == "fp64" else 64)))
    if scene == "thread":
        return _drop(_case("", scene, log(96, 512), log(32, 96), log(32, 96), prec, steps))
    if scene == "orifice":
        return _drop(_case("", scene, log(48, 144), log(48, 144), log(96, 256), prec, steps))
    if scene == "bubble":
        n = log(20, 96)
        return _drop(_case("", scene, n, n, n, prec, steps))
    if scene == "run":
        return _drop(_case("", scene, log(48, 160), log(48, 160), log(48, 160), prec, steps))
    return _drop(_case("", "label", log(32, 128), log(32, 128), log(32, 128), "fp64", 0))


def _drop(case):
    del case["name"]
    return case


def _cells(case):
    if case["scene"] == "population":
        m = (case["nx"] + case["ny"] + case["nz"]) / 3.0   # each side is one of the three
        return case["domains"] * m ** 3
    return case["nx"] * case["ny"] * case["nz"]


def work(case):
    """Bytes and operations of a pass: per step one byte of type per cell, 19
    PDFs read and written per liquid and interface cell, 37 B more per interface
    cell (mass read and written, fill level, density, mark); then the PDFs and
    fill levels read and 41 B written per cell by the read-back."""
    n, s = _cells(case), BYTES[case["precision"]]
    if case["scene"] == "label":
        return {"bytes": 9.0 * n, "flops": 0.0}
    liquid, interface = {"foam": (0.70, 0.09), "run": (0.70, 0.09), "bubbles": (0.70, 0.13), "population": (0.70, 0.13),
                         "thread": (0.88, 0.015), "orifice": (0.68, 0.01), "bubble": (0.91, 0.03)}[case["scene"]]
    step = n * (1.0 + (liquid + interface) * 38.0 * s + interface * 37.0)
    b = case["steps"] * step + n * (19.0 * s + 9.0 + 41.0)
    if case["scene"] == "run":
        b += n * (41.0 + 19.0 * s)
    return {"bytes": b, "flops": case["steps"] * n * (liquid + interface) * 300.0}


# -------------------------------------------------------------------- inputs

class Geometry:
    """One lattice: flat device arrays, parameters, bubble sources."""

    def __init__(self, nx, ny, nz, fill, obstacle=None, lid_mask=None, rho=None, u=None, sources=(), **par):
        shape = (nz, ny, nx)
        flags = torch.full(shape, IFC, dtype=torch.uint8, device=DEV)
        flags[fill >= 1.0] = LIQ
        flags[fill <= 0.0] = GAS
        if obstacle is not None:
            flags[obstacle] = OBS
        if lid_mask is not None:
            flags[lid_mask] = LID
        near, gas = torch.zeros(shape, dtype=torch.bool, device=DEV), flags == GAS
        for c in C[1:]:
            near |= torch.roll(gas, shifts=(c[2], c[1], c[0]), dims=(0, 1, 2))
        flags[(flags == LIQ) & near] = IFC      # the interface layer is closed
        self.dims, self.n = (nx, ny, nz), nx * ny * nz
        self.flags = flags.reshape(-1)
        self.fill = torch.where(flags == LIQ, 1.0, torch.where(flags == IFC, fill, 0.0)).reshape(-1).to(F64)
        fluid = (flags == LIQ) | (flags == IFC)
        self.rho = torch.ones(self.n, dtype=F64, device=DEV) if rho is None else torch.where(fluid, rho, 1.0).reshape(-1)
        if u is None:
            self.u = torch.zeros(3 * self.n, dtype=F64, device=DEV)
        else:
            self.u = torch.where(gas[None], 0.0, u).reshape(-1)
        self.sources = list(sources)
        self.par = dict(nx=nx, ny=ny, nz=nz, collision=1, tau=0.8, magic=3.0 / 16.0, sigma=0.0, gravity=(0.0, 0.0, 0.0),
                        eps=1e-3, lid=(0.0, 0.0, 0.0), normal_rule=1, lonely_rule=1)
        self.par.update(par)


def _axes(nx, ny, nz):
    ax = [torch.arange(k, dtype=F64, device=DEV) + 0.5 for k in (nx, ny, nz)]
    return ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]


def _offsets():
    return (torch.arange(4, dtype=F64, device=DEV) + 0.5) / 4 - 0.5


def _sampled(shape, sdf):
    """Liquid fraction of every cell from 4^3 sample points of a signed distance
    (negative in gas)."""
    nz, ny, nx = shape
    x, y, z = _axes(nx, ny, nz)
    d = sdf(x, y, z).expand(shape)
    fill = (d >= 0.0).to(F64)
    k, j, i = torch.nonzero(d.abs() <= 1.5, as_tuple=True)
    o = _offsets()
    xs = (i.to(F64) + 0.5)[:, None, None, None] + o[None, None, None, :]
    ys = (j.to(F64) + 0.5)[:, None, None, None] + o[None, None, :, None]
    zs = (k.to(F64) + 0.5)[:, None, None, None] + o[None, :, None, None]
    fill[k, j, i] = (sdf(xs, ys, zs) >= 0.0).expand(-1, 4, 4, 4).reshape(k.numel(), 64).sum(1).to(F64) / 64.0
    return fill


def _pack(rng, dims, radii, gap, bounded_z):
    """Spheres placed at random with a liquid gap, the largest first: groups of
    similar size draw centres in rounds, a sphere taking its draw when it keeps
    the gap to those placed and to the earlier draws of the round."""
    radii = np.sort(np.asarray(radii))[::-1]
    if len(radii) <= 256:                          # few spheres: one after the other on the host
        pc, pr, L, wrap = np.zeros((0, 3)), np.zeros(0), np.asarray(dims, dtype=np.float64), np.array([1, 1, not bounded_z])
        for r in radii:
            c = rng.uniform(0.0, 1.0, (64, 3)) * L
            if bounded_z:
                c[:, 2] = np.clip(c[:, 2], 1.0 + gap + r, max(1.0 + gap + r, dims[2] - 1.0 - gap - r))
            d = c[:, None, :] - pc[None]
            d -= wrap * L * np.round(d / L)
            ok = np.nonzero(((d * d).sum(-1) >= (r + pr + gap) ** 2).all(1))[0]
            if len(ok):
                pc, pr = np.concatenate([pc, c[ok[:1]]]), np.append(pr, r)
        return torch.tensor(pc, device=DEV), torch.tensor(pr, device=DEV)
    L = torch.tensor(dims, dtype=torch.float32, device=DEV)
    per = torch.tensor([1.0, 1.0, 0.0 if bounded_z else 1.0], device=DEV)
    pc, pr = torch.zeros((0, 3), device=DEV), torch.zeros(0, device=DEV)

    def apart(ca, ra, cb, rb):
        d = ca[:, None, :] - cb[None, :, :]
        d = d - per * L * torch.round(d / L)
        return (d * d).sum(-1) >= (ra[:, None] + rb[None, :] + gap + 1e-3) ** 2

    for group in np.array_split(radii, 12):
        left = torch.tensor(group.copy(), dtype=torch.float32, device=DEV)
        for _ in range(12):
            if not len(left):
                break
            draw_ = torch.tensor(rng.uniform(0.0, 1.0, (len(left), 3)), dtype=torch.float32, device=DEV)
            c = draw_ * L
            if bounded_z:
                lo, hi = 1.0 + gap + left, dims[2] - 1.0 - gap - left
                c[:, 2] = lo + draw_[:, 2] * (hi - lo).clamp(min=0.0)
            ok = apart(c, left, pc, pr).all(1) if len(pr) else torch.ones(len(left), dtype=torch.bool, device=DEV)
            if bounded_z:
                ok &= hi > lo
            clash = ~apart(c, left, c, left) & ok[None, :]
            ok &= ~torch.tril(clash, diagonal=-1).any(1)
            pc, pr = torch.cat([pc, c[ok]]), torch.cat([pr, left[ok]])
            left = left[~ok]
    return pc.to(F64), pr.to(F64)


def _stamped(shape, centres, radii):
    """Liquid fraction of a periodic box holding gas spheres, from 4^3 sample
    points per cell of the band around each surface."""
    nz, ny, nx = shape
    fill = torch.ones(nz * ny * nx, dtype=F64, device=DEV)
    box = torch.ceil(2.0 * radii + 3.0).to(torch.int64)
    off, reach = _offsets(), 0.5 * math.sqrt(3.0) * 0.75 + 1e-9
    for b in sorted(set(box.tolist())):
        ids = torch.nonzero(box == b).reshape(-1)
        per = max(1, (1 << 23) // b ** 3)
        o = torch.arange(b, dtype=F64, device=DEV)
        for s in range(0, len(ids), per):
            c, r = centres[ids[s:s + per]], radii[ids[s:s + per]]
            base = torch.floor(c - r[:, None] - 1.0)
            X, Y, Z = (base[:, a:a + 1] + o[None, :] for a in range(3))
            dist = torch.sqrt(((Z + 0.5 - c[:, 2:3]) ** 2)[:, :, None, None] + ((Y + 0.5 - c[:, 1:2]) ** 2)[:, None, :, None]
                              + ((X + 0.5 - c[:, 0:1]) ** 2)[:, None, None, :]) - r[:, None, None, None]
            flat = ((X.to(torch.int64) % nx)[:, None, None, :] + nx * ((Y.to(torch.int64) % ny)[:, None, :, None]
                    + ny * (Z.to(torch.int64) % nz)[:, :, None, None]))
            fill[flat[dist < -reach]] = 0.0
            m, k, j, i = torch.nonzero(dist.abs() <= reach, as_tuple=True)
            ax = (X[m, i][:, None] + 0.5 + off - c[m, 0][:, None]) ** 2
            ay = (Y[m, j][:, None] + 0.5 + off - c[m, 1][:, None]) ** 2
            az = (Z[m, k][:, None] + 0.5 + off - c[m, 2][:, None]) ** 2
            d2 = az[:, :, None, None] + ay[:, None, :, None] + ax[:, None, None, :]
            cnt = (d2 < (r[m] ** 2)[:, None, None, None]).reshape(m.numel(), 64).sum(1)
            fill.scatter_reduce_(0, flat[m, k, j, i], 1.0 - cnt.to(F64) / 64.0, "amin")
    return fill.reshape(shape)


def _waves(rng, dims, u_max):
    """One Fourier mode per velocity component."""
    x, y, z = _axes(*dims)
    k, ph = rng.integers(1, 3, size=(3, 3)), rng.uniform(0.0, 2.0 * np.pi, size=3)
    amp = u_max * rng.uniform(0.3, 1.0) / math.sqrt(3.0)
    return torch.stack([amp * torch.sin(2.0 * np.pi * (float(k[c, 0]) * x / dims[0] + float(k[c, 1]) * y / dims[1]
                                                       + float(k[c, 2]) * z / dims[2]) + float(ph[c])) for c in range(3)])


def _bubbles(rng, dims, sigma, u_max, per_cell=4e-4, r_lo=3.0, r_hi=8.0):
    """A periodic box of bubbles in a smooth random flow.  (The liquid gap and, in
    the populations, the surface tension keep films from bursting all at once:
    a pass runs hundreds of times on one handle, and the violent coalescence
    of a closer packing can drive the scheme itself to a NaN.)"""
    n = dims[0] * dims[1] * dims[2]
    r_hi = min(r_hi, 0.25 * min(dims))
    radii = rng.uniform(min(r_lo, r_hi), r_hi, max(2, min(200, int(n * per_cell))))
    c, r = _pack(rng, dims, radii, 3.0, False)
    return Geometry(*dims, _stamped(dims[::-1], c, r), u=_waves(rng, dims, u_max), sigma=sigma)


def _foam(rng, dims):
    """Dense packing of lognormal bubbles, no-slip bottom, moving lid, gravity."""
    nx, ny, nz = dims
    target, radii, vol = 0.4 * nx * ny * nz, [], 0.0
    while vol < target:
        r = np.clip(np.exp(np.log(8.0) + 0.3 * rng.standard_normal(256)), 4.0, min(16.0, 0.2 * min(dims)))
        radii.append(r)
        vol += float((4.0 / 3.0 * np.pi * r ** 3).sum())
    c, r = _pack(rng, dims, np.concatenate(radii), 3.0, True)
    obs = torch.zeros((nz, ny, nx), dtype=torch.bool, device=DEV)
    lid = obs.clone()
    obs[0], lid[-1] = True, True
    return Geometry(nx, ny, nz, _stamped((nz, ny, nx), c, r), obstacle=obs, lid_mask=lid, sigma=3e-3,
                    gravity=(0.0, 0.0, -1e-5), lid=(0.05, 0.0, 0.0))


def _thread(rng, dims):
    nx, ny, nz = dims
    R, amp, ph = min(ny, nz) / 8.0, rng.uniform(0.05, 0.15), rng.uniform(0.0, 2.0 * np.pi)
    waves = max(1, round(nx / 64.0))
    cy, cz = ny / 2.0 + rng.uniform(-1.0, 1.0), nz / 2.0 + rng.uniform(-1.0, 1.0)

    def sdf(x, y, z):
        return torch.sqrt((y - cy) ** 2 + (z - cz) ** 2) - R * (1.0 + amp * torch.sin(2.0 * np.pi * waves * x / nx + ph))

    obs = torch.zeros((nz, ny, nx), dtype=torch.bool, device=DEV)
    obs[0] = obs[-1] = True
    obs[:, 0] = obs[:, -1] = True
    return Geometry(nx, ny, nz, _sampled((nz, ny, nx), sdf), obstacle=obs, sigma=5e-3)


def _orifice(rng, dims):
    nx, ny, nz = dims
    pz, hole, cap = max(4, nz // 32), min(nx, ny) * 6.0 / 128.0 + 1.0, min(nx, ny) * rng.uniform(5.0, 7.0) / 128.0 + 1.0
    g, top, ph = 1e-5, pz + 1 + int(nz * 200 / 256), rng.uniform(0.0, 2.0 * np.pi, 2)
    hx, hy = nx / 2.0 + rng.uniform(-1.0, 1.0), ny / 2.0 + rng.uniform(-1.0, 1.0)

    def sdf(x, y, z):
        rr = torch.sqrt((x - hx) ** 2 + (y - hy) ** 2)
        wave = 0.4 * torch.sin(2.0 * np.pi * x / nx + ph[0]) * torch.sin(2.0 * np.pi * y / ny + ph[1])
        gas = torch.maximum(pz + 0.5 - z, z - top - wave)
        gas = torch.maximum(gas, cap - torch.sqrt(rr ** 2 + (z - (pz + 1.0)) ** 2))
        return -torch.maximum(gas, torch.where((z - (pz + 0.5)).abs() <= 0.5, hole - rr, -1e9))

    x, y, z = _axes(nx, ny, nz)
    obs = torch.zeros((nz, ny, nx), dtype=torch.bool, device=DEV)
    obs[0] = obs[-1] = True
    obs[:, 0] = obs[:, -1] = True
    obs[:, :, 0] = obs[:, :, -1] = True
    obs[pz] |= (torch.sqrt((x - hx) ** 2 + (y - hy) ** 2) > hole)[0]
    rho = 1.0 + 3.0 * g * (top - z) + torch.zeros((nz, ny, nx), dtype=F64, device=DEV)
    at = int(hx) + nx * int(hy)
    return Geometry(nx, ny, nz, _sampled((nz, ny, nx), sdf), obstacle=obs, rho=rho, sigma=2e-3, gravity=(0.0, 0.0, -g),
                    sources=[(at + nx * ny * 2, 2e4, 0.02, 0), (at + nx * ny * (nz - 3), 0.0, 0.0, 1)])


def _bubble(rng, dims):
    n = min(dims)
    c = torch.tensor([[d / 2.0 + rng.uniform(-1.0, 1.0) for d in dims]], dtype=F64, device=DEV)
    r = torch.tensor([n / 4.0 * rng.uniform(0.9, 1.1)], dtype=F64, device=DEV)
    return Geometry(*dims, _stamped(dims[::-1], c, r), collision=0, sigma=1e-3)


def _geometries(case, seed):
    rng = np.random.default_rng(seed)
    dims = (case["nx"], case["ny"], case["nz"])
    scene = case["scene"]
    if scene == "population":
        out = []
        sides = np.random.default_rng(0).choice(dims, (case["domains"], 3))   # the sizes belong to the case
        for side in sides:
            out.append(_bubbles(rng, tuple(int(v) for v in side), float(rng.uniform(1e-3, 1.5e-3)), u_max=0.01))
        return out
    if scene == "bubbles":
        return [_bubbles(rng, dims, 5e-3, u_max=0.05)]
    return [{"foam": _foam, "run": _foam, "label": _foam, "thread": _thread, "orifice": _orifice,
             "bubble": _bubble}[scene](rng, dims)]


# ------------------------------------------------------------------- passes

def _simulation(geoms, precision):
    sim = fsl.Simulation([g.par for g in geoms], precision=precision)
    for d, g in enumerate(geoms):
        sim.init_geometry(d, g.flags, g.fill, g.rho, g.u, on_device=True)
    for d, g in enumerate(geoms):
        for s in g.sources:
            sim.set_source(d, *s)
    return sim


class State:
    """The handle of a running simulation and the caller's buffers for its state."""

    def __init__(self, case, geoms, sim):
        self.case, self.sim, self.geoms = case, sim, geoms
        n = [g.n for g in geoms]
        at = np.concatenate([[0], np.cumsum(n)])
        tot = int(at[-1])
        self.flags = torch.empty(tot, dtype=torch.uint8, device=DEV)
        self.fill = torch.empty(tot, dtype=F64, device=DEV)
        self.rho = torch.empty(tot, dtype=F64, device=DEV)
        self.u = torch.empty(3 * tot, dtype=F64, device=DEV)
        self.views = [{"flags": self.flags[at[d]:at[d + 1]], "fill": self.fill[at[d]:at[d + 1]],
                       "rho": self.rho[at[d]:at[d + 1]], "u": self.u[3 * at[d]:3 * at[d + 1]]} for d in range(len(n))]
        self.pdf = None
        if case["scene"] == "bubble":                 # small: the distributions too
            self.pdf = self.views[0]["pdf"] = torch.empty(19 * tot, dtype=F64, device=DEV)


def prepare(case, seed):
    geoms = _geometries(case, seed)
    if case["scene"] == "label":
        g = geoms[0]
        return {"flags": g.flags, "dims": g.dims, "labels": torch.empty(g.n, dtype=torch.int64, device=DEV)}
    if case["scene"] == "run":
        return State(case, geoms, None)
    sim = _simulation(geoms, case["precision"])
    sim.step(WARM_STEPS)
    st = State(case, geoms, sim)
    for g in geoms:
        g.flags = g.fill = g.rho = g.u = None     # the handle holds the state from here on
    return st


def _table_rows(case):
    return 16 + _cells(case) // 4096


def _read_back(st, sim):
    """The state in the caller's buffers; FP64 as it is, the reduced forms in FP32."""
    for d, v in enumerate(st.views):
        sim.fields_to(d, v)
    out = {"flags": st.flags, "fill": st.fill, "rho": st.rho, "u": st.u}
    if st.pdf is not None:
        out["pdf"] = st.pdf
    reduced = st.case["precision"] != "fp64"
    if st.case["scene"] in ("bubble", "thread", "orifice", "run"):
        b, real = sim.bubbles(0), np.float32 if reduced else np.float64
        for name, field, dtype in (("bubble_id", "id", np.int64), ("bubble_cells", "n_cells", np.int64),
                                   ("bubble_volume", "volume", real), ("bubble_pressure", "pressure", real)):
            out[name] = np.zeros(_table_rows(st.case), dtype=dtype)     # a table of a fixed number of rows
            out[name][:len(b)] = b[field]
    if reduced:
        for k in ("fill", "rho", "u", "pdf"):
            if k in out:
                out[k] = out[k].float()
    return out


def run(state):
    if isinstance(state, dict):
        fsl.label_bubbles_static(state["flags"], *state["dims"], state["labels"])
        return {"labels": state["labels"]}
    if state.sim is None:
        sim = _simulation(state.geoms, state.case["precision"])
        sim.step(state.case["steps"])
        out = _read_back(state, sim)
        sim.close()
        return out
    state.sim.step(state.case["steps"])
    return _read_back(state, state.sim)


# -------------------------------------------------- the method in 64 bits

class Reference:
    """The time step in plain torch FP64, for any number of lattices side by side."""

    def __init__(self, geoms, precision):
        self.off = np.concatenate([[0], np.cumsum([g.n for g in geoms])])
        self.N, self.D = int(self.off[-1]), len(geoms)
        par = [g.par for g in geoms]

        def per_cell(v, dtype=F64):
            return torch.repeat_interleave(torch.tensor(v, dtype=dtype, device=DEV),
                                           torch.tensor([g.n for g in geoms], device=DEV))

        self.dom = per_cell(list(range(self.D)), torch.int64)
        self.nx, self.ny, self.nz = (torch.tensor([g.dims[a] for g in geoms], device=DEV) for a in range(3))
        self.o = torch.tensor(self.off[:-1], device=DEV)
        l = torch.arange(self.N, device=DEV) - self.o[self.dom]
        nx, ny = self.nx[self.dom], self.ny[self.dom]
        self.x, self.y, self.z = (l % nx).int(), ((l // nx) % ny).int(), (l // (nx * ny)).int()
        self.p = par[0]
        self.omp = 1.0 / self.p["tau"]
        self.omm = 1.0 / (self.p["magic"] / (self.p["tau"] - 0.5) + 0.5) if self.p["collision"] == 1 else self.omp
        self.sigma2 = torch.tensor([2.0 * p["sigma"] for p in par], dtype=F64, device=DEV)
        self.flag = torch.cat([g.flags for g in geoms])
        fill = torch.cat([g.fill for g in geoms])
        rho = torch.cat([g.rho for g in geoms])
        u = [torch.cat([g.u[a * g.n:(a + 1) * g.n] for g in geoms]) for a in range(3)]
        fluid = (self.flag == LIQ) | (self.flag == IFC)
        self.f = [torch.where(fluid, e, W[a]) for a, e in enumerate(self.feq(rho, u))]
        shifted = precision in ("f16s", "bf16s")     # a buffer of zeros holds f = w in the shifted forms
        self.g = [torch.full((self.N,), W[a] if shifted else 0.0, dtype=F64, device=DEV) for a in range(19)]
        self.phi = torch.where(self.flag == LIQ, 1.0, torch.where(self.flag == IFC, fill, 0.0))
        self.m = torch.where(fluid, torch.where(self.flag == IFC, fill * rho, rho), 0.0)
        self.rhoi = torch.where(fluid, rho, 0.0)
        self.pool = torch.zeros(self.D, dtype=torch.int64, device=DEV)
        self.seed = self.rate = None
        self.id = None
        self.bubbles(initial=True)
        for d, g in enumerate(geoms):
            for cell, extra, rate, const in g.sources:
                b = self.id[int(self.off[d]) + cell]
                if const:
                    self.bconst[b] = True
                else:
                    v = int(round(extra * 2 ** 32))
                    self.bextra[b] += v
                    self.bstar[b] += v
                    self.seed, self.rate = int(self.off[d]) + cell, int(round(rate * 2 ** 32))

    def nb(self, i, c):
        """Cells i + c."""
        d = self.dom[i] if self.D > 1 else None
        nx, ny, nz = (v[d] if self.D > 1 else int(v[0]) for v in (self.nx, self.ny, self.nz))
        x, y, z = ((self.x[i] + c[0]) % nx).long(), ((self.y[i] + c[1]) % ny).long(), ((self.z[i] + c[2]) % nz).long()
        return (self.o[d] if self.D > 1 else 0) + x + nx * (y + ny * z)

    @staticmethod
    def dot(a, v):
        return sum(c * x for c, x in zip(C[a], v) if c) if a else 0.0

    def feq(self, rho, u):
        usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        out = []
        for a in range(19):
            cu = self.dot(a, u)
            out.append(W[a] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq))
        return out

    @staticmethod
    def moments(f):
        r = sum(f[1:], f[0])
        return r, [sum(C[a][k] * f[a] for a in range(1, 19) if C[a][k]) for k in range(3)]

    def volume(self, i):
        t = self.flag[i]
        part = torch.round((1.0 - self.phi[i].clamp(0.0, 1.0)) * 2.0 ** 32).long()
        return torch.where(t == GAS, 1 << 32, torch.where(t == IFC, part, 0))

    def bubbles(self, initial=False):
        """Components of gas and interface cells (18-neighbourhood) and the bubble table."""
        fg = torch.nonzero((self.flag == GAS) | (self.flag == IFC)).reshape(-1)
        pos = torch.full((self.N,), -1, dtype=torch.int64, device=DEV)
        pos[fg] = torch.arange(len(fg), device=DEV)
        lab = torch.arange(len(fg), device=DEV)
        near = [pos[self.nb(fg, C[a])] for a in range(1, 19)]
        while True:
            new = lab.clone()
            for p in near:
                new = torch.where(p >= 0, torch.minimum(new, lab[p.clamp(min=0)]), new)
            low = lab.clone()
            low.scatter_reduce_(0, lab, new, "amin")      # the old root takes the lowest label seen
            new = torch.minimum(new, low[new])
            for _ in range(4):
                new = new[new]
            if bool((new == lab).all()):
                break
            lab = new
        root, comp = torch.unique(lab, return_inverse=True)
        k, t = len(root), self.volume(fg)
        vol = torch.zeros(k, dtype=torch.int64, device=DEV).index_add_(0, comp, t)
        extra, const = torch.zeros_like(vol), torch.zeros(k, dtype=torch.bool, device=DEV)
        if initial:
            star = vol.clone()
        else:
            old = self.id[fg]
            key, pair = torch.unique(comp * len(self.bvol) + old, return_inverse=True)
            pc, pb = key // len(self.bvol), key % len(self.bvol)
            pv = torch.zeros(len(key), dtype=torch.int64, device=DEV).index_add_(0, pair, t)
            if self.seed is not None and int(pos[self.seed]) >= 0:
                q = pair[pos[self.seed]]
                pv[q] += self.bextra[pb[q]]
                extra[pc[q]] = self.bextra[pb[q]]
            tot = torch.zeros_like(self.bvol).index_add_(0, pb, pv)
            first = torch.full_like(self.bvol, 1 << 40).scatter_reduce_(0, pb, pc, "amin")
            s = self.bstar[pb]
            share = torch.where(tot[pb] == 0, torch.where(pc == first[pb], s, 0),
                                torch.where(pv == tot[pb], s, torch.round(s.to(F64) * (pv.to(F64) / tot[pb].to(F64))).long()))
            star = torch.zeros_like(vol).index_add_(0, pc, share)
            const[pc[self.bconst[pb]]] = True
        self.bvol, self.bextra, self.bstar, self.bconst = vol, extra, star, const
        self.id = torch.full((self.N,), -1, dtype=torch.int64, device=DEV)
        self.id[fg] = comp
        self.bid, self.bcells = fg[root], torch.bincount(comp, minlength=k)

    def pressure(self):
        V = (self.bvol + self.bextra).to(F64) * 2.0 ** -32
        p = torch.where(V <= 1e-3, 1.0, self.bstar.to(F64) * 2.0 ** -32 / V)
        return torch.where(self.bconst, 1.0, p) / 3.0

    def gradient(self, i):
        st = self.stencil
        g = [0.0, 0.0, 0.0]
        for b in (-1, 0, 1):
            for a in (-1, 0, 1):
                w = 4.0 if a == b == 0 else 2.0 if a == 0 or b == 0 else 1.0
                g[0] = g[0] + w * (st[self.nb(i, (1, a, b))] - st[self.nb(i, (-1, a, b))])
                g[1] = g[1] + w * (st[self.nb(i, (a, 1, b))] - st[self.nb(i, (a, -1, b))])
                g[2] = g[2] + w * (st[self.nb(i, (a, b, 1))] - st[self.nb(i, (a, b, -1))])
        return g

    def normal(self, i, k):
        g = self.gradient(i)
        n = torch.sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2])
        return torch.where(n > 0.0, -g[k] / n, 0.0)

    def step(self):
        F, G, p, flag = self.f, self.g, self.p, self.flag
        t_if, all_ = flag == IFC, torch.arange(self.N, device=DEV)
        lid = p["lid"]
        I = torch.nonzero(t_if).reshape(-1)
        L = torch.nonzero((flag == LIQ) | t_if).reshape(-1)
        self.stencil = torch.where(flag == GAS, 0.0, torch.where(t_if, self.phi.clamp(0.0, 1.0), 1.0))
        # interface cells: gas density, equilibrium with the cell's own velocity
        own = [F[a][I] for a in range(19)]
        r, j = self.moments(own)
        kappa = 0.25 * sum(self.normal(self.nb(I, C[2 * k + 1]), k) - self.normal(self.nb(I, C[2 * k + 2]), k) for k in range(3))
        rg = 3.0 * (self.pressure()[self.id[I]] + self.sigma2[self.dom[I]] * kappa)
        gas_eq = self.feq(rg, [v / r for v in j])
        grad = self.gradient(I)
        at = torch.searchsorted(L, I)
        fin, dm, has_gas, has_liq = [F[0][L]], 0.0, False, False
        for a in range(1, 19):
            b = OPP[a]
            y = self.nb(L, tuple(-v for v in C[a]))
            ty = flag[y]
            wall = (ty == OBS) | (ty == LID)
            v = torch.where(wall, F[b][L], F[a][y])
            lidt = 6.0 * W[a] * self.dot(a, lid)
            if lidt:
                v = torch.where(ty == LID, v + lidt, v)
            tz = ty[at]
            rebuild = (tz == GAS) | ((tz <= IFC) & (self.dot(a, grad) > 0.0))
            pulled = F[a][y[at]]
            # the link a - bar reaches the same neighbour y
            ex = pulled - own[b]
            dm = dm + torch.where(tz == LIQ, ex, torch.where(tz == IFC, 0.5 * (self.phi[I] + self.phi[y[at]]) * ex, 0.0))
            has_gas, has_liq = has_gas | (tz == GAS), has_liq | (tz == LIQ)
            v[at] = torch.where(rebuild, gas_eq[a] + gas_eq[b] - own[b], v[at])
            fin.append(v)
        # collision
        r, j = self.moments(fin)
        gv = p["gravity"]
        force = [r * c for c in gv]
        u = [(j[k] + 0.5 * force[k]) / r for k in range(3)]
        usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        uF = sum(u[k] * force[k] for k in range(3))
        cp, cm = 1.0 - 0.5 * self.omp, 1.0 - 0.5 * self.omm
        G[0][L] = fin[0] - self.omp * (fin[0] - W[0] * r * (1.0 - 1.5 * usq)) - cp * W[0] * 3.0 * uF
        for a in range(1, 19, 2):
            b, w = a + 1, W[a]
            cu, cF = self.dot(a, u), self.dot(a, force)
            A = self.omp * (0.5 * (fin[a] + fin[b]) - w * r * (1.0 + 4.5 * cu * cu - 1.5 * usq))
            B = self.omm * (0.5 * (fin[a] - fin[b]) - w * r * 3.0 * cu)
            sp, sm = cp * w * (9.0 * cu * cF - 3.0 * uF), cm * w * 3.0 * cF
            G[a][L] = fin[a] - A - B + sp + sm
            G[b][L] = fin[b] - A + B + sp - sm
        # marks
        rho = r[at]
        self.m[I] += dm
        self.rhoi[I] = rho
        m = self.m[I]
        filled, emptied = m > (1.0 + p["eps"]) * rho, m < -p["eps"] * rho
        lonely = ~filled & ~emptied
        filled = filled | (lonely & ~has_gas)
        emptied = ~filled & (emptied | (lonely & ~has_liq))
        FILLED, EMPTIED = (torch.zeros(self.N, dtype=torch.bool, device=DEV) for _ in range(2))
        fc = I[filled]
        FILLED[fc] = True
        EMPTIED[I[emptied]] = True
        new = flag.clone()
        fresh = torch.zeros(self.N, dtype=torch.bool, device=DEV)
        for a in range(1, 19):
            z = self.nb(fc, C[a])
            EMPTIED[z] = False
            fresh[z[flag[z] == GAS]] = True
        ec = torch.nonzero(EMPTIED).reshape(-1)
        drops = torch.cat([self.nb(ec, C[a]) for a in range(1, 19)]) if len(ec) else ec
        drops = torch.unique(drops[flag[drops] == LIQ])
        for a in range(18, 0, -1):
            z = self.nb(drops, C[a])
            self.id[drops] = torch.where(EMPTIED[z], self.id[z], self.id[drops])
        if len(drops):
            self.m[drops] = self.rhoi[drops] = self.moments([G[a][drops] for a in range(19)])[0]
        nc = torch.nonzero(fresh).reshape(-1)
        if len(nc):
            sr, su, cnt = 0.0, [0.0, 0.0, 0.0], 0.0
            for a in range(1, 19):
                z = self.nb(nc, C[a])
                use = (flag[z] == LIQ) | ((flag[z] == IFC) & ~EMPTIED[z])
                rr, jj = self.moments([G[q][z] for q in range(19)])
                sr = sr + torch.where(use, rr, 0.0)
                su = [su[k] + torch.where(use, jj[k] / rr, 0.0) for k in range(3)]
                cnt = cnt + use
            for a, e in enumerate(self.feq(sr / cnt, [v / cnt for v in su])):
                G[a][nc] = e
            self.m[nc] = 0.0
            self.rhoi[nc] = sr / cnt
        new[fc], new[ec], new[drops], new[nc] = LIQ, GAS, IFC, IFC
        # excess mass
        conv = torch.cat([fc, ec])
        over = torch.cat([self.m[fc] - self.rhoi[fc], self.m[ec]])
        k = sum(((new[self.nb(conv, C[a])] == IFC).long() for a in range(1, 19)), torch.zeros_like(conv))
        ex = torch.zeros(self.N, dtype=F64, device=DEV)
        ex[conv] = torch.where(k > 0, over / k.clamp(min=1), 0.0)
        lost = torch.where(k > 0, 0, torch.round(over * 2.0 ** 40).long())
        self.pool.index_add_(0, self.dom[conv], lost)
        R = torch.nonzero(new == IFC).reshape(-1)
        count = torch.bincount(self.dom[R], minlength=self.D)
        sm = self.m[R]
        for a in range(1, 19):
            sm = sm + ex[self.nb(R, C[a])]
        sm = sm + (self.pool.to(F64) * 2.0 ** -40 / count.clamp(min=1))[self.dom[R]]
        self.pool[count > 0] = 0
        self.m[R] = sm
        self.phi[R] = sm / self.rhoi[R]
        self.phi[fc], self.phi[ec], self.m[ec], self.id[fc] = 1.0, 0.0, 0.0, -1
        self.flag = new
        if self.seed is not None and int(self.id[self.seed]) >= 0:
            self.bextra[self.id[self.seed]] -= self.rate
        self.bubbles()
        self.f, self.g = G, F


def exact(case, seed):
    """What `run` returns, in 64 bits; no value for labels, types, ids and counts,
    nor for lattices that would take minutes."""
    if case["scene"] == "label" or _cells(case) > 2.0e7:
        return None
    geoms = _geometries(case, seed)
    ref = Reference(geoms, case["precision"])
    for _ in range(case["steps"] + (0 if case["scene"] == "run" else WARM_STEPS)):
        ref.step()
    r, j = ref.moments(ref.f)
    u = [torch.where(r != 0.0, v / r, 0.0) for v in j]
    u = torch.cat([torch.cat([v[ref.off[d]:ref.off[d + 1]] for v in u]) for d in range(ref.D)])
    out = {"flags": None, "fill": ref.phi, "rho": r, "u": u}
    if case["scene"] in ("bubble", "thread", "orifice", "run"):
        v, p = (torch.zeros(_table_rows(case), dtype=F64, device=DEV) for _ in range(2))
        v[:len(ref.bvol)], p[:len(ref.bvol)] = (ref.bvol + ref.bextra).to(F64) * 2.0 ** -32, ref.pressure()
        out.update(bubble_id=None, bubble_cells=None, bubble_volume=v, bubble_pressure=p)
    if case["scene"] == "bubble":
        out["pdf"] = torch.cat(ref.f)
    return out
