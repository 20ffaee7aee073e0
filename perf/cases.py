"""Performance cases of the boosted-frame PIC step: what a program built on this package
has it do, through the package's public calls.

A pass of a "step" case advances a loaded simulation (or a batch of them) some steps and
reads its state out, as a run does between two outputs; the state goes on evolving from
pass to pass.  The small and middle boxes are periodic along z, the direction the boosted
plasma streams in, so that a long run keeps its particles; the full stage has open ends,
as it is run.  FP32 fields are returned in FP32, the precision the run stores.

exact() steps the same loaded state in 64 bits with plain torch (class _Ref below).
"""
import ctypes
import math

import numpy as np
import torch

import paper_0909_5603_gb300 as pic

FIELDS = [pic.PIC_EX, pic.PIC_EY, pic.PIC_EZ, pic.PIC_BX, pic.PIC_BY, pic.PIC_BZ]


def _case(name, kind, n, ppc, **kw):
    c = dict(name=name, kind=kind, n0=n[0], n1=n[1], n2=n[2], ppc=ppc, order=2, fp64=False, passes=0, steps=10,
             gamma=1.0, ck=False, boris=False, periodic_z=True)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest run: a 2D3V thermal plasma of 65,536 particles (launches and gaps count)
        _case("plasma_2d", "plasma", (128, 1, 128), 4, steps=16),
        # the same in all-FP64, the precision such a reference run is made in
        _case("plasma_2d_fp64", "plasma", (128, 1, 128), 4, steps=16, fp64=True),
        # a parameter scan: uneven independent 2D3V instances stepped as one batch
        _case("scan_2d_batch", "scan", (64, 1, 512), 16, steps=10, instances=32, passes=1),
        # a laser wakefield stage scaled down for a quick look (0.5M particles)
        _case("lwfa_small", "lwfa", (32, 32, 256), 2, steps=20, gamma=13.0, passes=3),
        # linear shape, sizes that are no multiple of any tile, one filter pass
        _case("lwfa_ragged_linear", "lwfa", (90, 70, 331), 3, steps=10, gamma=5.0, passes=1, order=1),
        # the stage under the low-dispersion solver, taken against the boosted-frame instability
        _case("lwfa_low_dispersion", "lwfa", (64, 64, 512), 4, steps=10, gamma=13.0, passes=3, ck=True),
        # a relativistic electron bunch with its self-field: particles crowded into few cells
        _case("beam", "beam", (64, 64, 256), 0, steps=20, particles=1 << 20, beam_gamma=1000.0),
        # a dense hot plasma, 16 particles per cell
        _case("plasma_3d_dense", "plasma", (64, 64, 64), 16, steps=10),
        # the stage in all-FP64, what FP32 runs are checked against
        _case("lwfa_fp64", "lwfa", (48, 48, 128), 2, steps=8, gamma=13.0, passes=3, fp64=True),
        # the full laser wakefield stage, 33.5M particles, open boundaries
        _case("lwfa_stage", "lwfa", (128, 128, 1024), 2, steps=20, gamma=13.0, passes=3, periodic_z=False),
        # what a run reads to judge itself: charge density, Gauss residual, energies
        _case("read_density", "read", (64, 64, 512), 2, gamma=13.0, passes=3),
        # exchange of the particle set with the host: load (sorted by tile) and read-out
        _case("load_particles", "load", (128, 128, 128), 2),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plasma2", "plasma3", "scan", "lwfa", "lwfa", "lwfa", "lwfa", "beam", "fp64", "read", "load"])
    gamma = math.exp(rng.uniform(math.log(1.5), math.log(30.0)))
    passes, order = rng.choice([0, 1, 2, 3, 3, 4]), rng.choice([1, 2, 2])
    if kind == "plasma2":
        c = _case("", "plasma", (_size(rng, 48, 700), 1, _size(rng, 48, 700)), _size(rng, 1, 16), order=order,
                  fp64=rng.random() < 0.3, passes=passes, steps=rng.randint(8, 20), boris=rng.random() < 0.3)
    elif kind == "plasma3":
        c = _case("", "plasma", tuple(_size(rng, 24, 100) for _ in range(3)), _size(rng, 2, 16), order=order,
                  steps=rng.randint(5, 12), passes=passes, boris=rng.random() < 0.3)
    elif kind == "scan":
        c = _case("", "scan", (64, 1, 512), 16, steps=rng.randint(5, 12), instances=_size(rng, 4, 48),
                  passes=rng.choice([0, 1, 3]), order=order)
    elif kind == "lwfa":
        c = _case("", "lwfa", (_size(rng, 24, 128), _size(rng, 24, 128), _size(rng, 64, 512)), rng.randint(1, 4),
                  steps=rng.randint(6, 16), gamma=gamma, passes=passes, order=order, ck=rng.random() < 0.3)
    elif kind == "beam":
        c = _case("", "beam", (_size(rng, 40, 80), _size(rng, 40, 80), _size(rng, 200, 300)), 0, order=order,
                  steps=rng.randint(8, 20), particles=_size(rng, 1 << 16, 1 << 21),
                  beam_gamma=math.exp(rng.uniform(math.log(10.0), math.log(1e4))), passes=rng.choice([0, 1]))
    elif kind == "fp64":
        c = _case("", "lwfa", (_size(rng, 24, 64), _size(rng, 24, 64), _size(rng, 64, 160)), rng.randint(1, 3),
                  steps=rng.randint(4, 10), gamma=gamma, passes=passes, order=order, fp64=True)
    elif kind == "read":
        c = _case("", "read", (_size(rng, 32, 100), _size(rng, 32, 100), _size(rng, 64, 700)), rng.randint(1, 4),
                  gamma=gamma, passes=passes, order=order)
    else:
        c = _case("", "load", tuple(_size(rng, 32, 160) for _ in range(3)), rng.randint(1, 3))
    del c["name"]
    return c


# ---- the runs -------------------------------------------------------------------------
def _lwfa_inputs(c, seed):
    """Cells of a 1/16 boosted wavelength along z and 2 lab wavelengths across, the plasma
    at 1/900 of the critical density: behind a ramp two cells long with the laser ahead of
    it (open z), or filling the periodic box with a two-period pulse in the middle."""
    g = c["gamma"]
    doppler = g * (1.0 + math.sqrt(1.0 - 1.0 / g ** 2))
    dz, dx = doppler / 16.0, 2.0
    if c["ck"]:
        dt = 0.9 * min(dx, dz)
    else:
        dt = min(0.5 * dz, 0.9 / math.sqrt(2.0 / dx ** 2 + 1.0 / dz ** 2))
    dens = (2.0 * math.pi) ** 2 / 900.0
    if c["periodic_z"]:
        laser = (2.0, 1.0, 20.0, 2.0, 0.5 * c["n2"] * dz / doppler)
        plasma = (dens, -1e9, 0.0, c["ppc"], (0.0, 0.0, 0.0), seed)
    else:
        laser = (2.0, 1.0, 20.0, 10.0, 20.0)
        plasma = (dens, 0.0, 2.0 * dz * g, c["ppc"], (0.0, 0.0, 0.0), seed)
    return (dx, dx, dz), dt, laser, plasma


def _scan_inputs(c, i):
    """Instance i of the scan: log2 of the side and the boost spread over the range, the
    density over two decades, a short pulse in the middle of the periodic plasma.  The
    instances of a scan are set by its plan; the seed places their particles."""
    rng = np.random.default_rng(5000 + i)
    side = max(48, int(round(2.0 ** rng.uniform(math.log2(c["n0"]), math.log2(c["n2"])) / 16)) * 16)
    ppc, g = int(rng.integers(1, c["ppc"] + 1)), float(rng.uniform(1.0, 50.0))
    dens = float(rng.uniform(1e-4, 1e-2)) * (2.0 * math.pi) ** 2
    doppler = g * (1.0 + math.sqrt(1.0 - 1.0 / g ** 2))
    dz, dx = doppler / 16.0, 2.0
    dt = min(0.5 * dz, 0.9 / math.sqrt(1.0 / dx ** 2 + 1.0 / dz ** 2))
    laser = (1.0, 1.0, 0.25 * side * dx, 2.0, 0.5 * side * dz / doppler)
    return side, ppc, g, (dx, 1.0, dz), dt, laser, dens


def _sim(c, n, dx, dt, gamma, bc, ids=False):
    return pic.Simulation(2 if n[1] == 1 else 3, n, bc, dx, dt, gamma_boost=gamma, order=c["order"],
                          precision=pic.PIC_PREC_FP64 if c["fp64"] else pic.PIC_PREC_FP32, filter_passes=c["passes"],
                          pusher=pic.PIC_PUSHER_BORIS if c["boris"] else pic.PIC_PUSHER_VAY, track_ids=ids,
                          solver=pic.PIC_SOLVER_CK if c["ck"] else pic.PIC_SOLVER_YEE)


def _pinned(shape, dtype):
    return torch.empty(shape, dtype=dtype, pin_memory=True)


def _particle_room(n, vt):
    vt = torch.float64 if vt == np.float64 else torch.float32
    room = dict(cell=_pinned(n, torch.int32), off=_pinned((n, 3), vt), u=_pinned((n, 3), vt), w=_pinned(n, vt),
                id=_pinned(n, torch.int32))
    return {k: v.numpy() for k, v in room.items()}


def prepare(case, seed):
    c, n, kind = case, (case["n0"], case["n1"], case["n2"]), case["kind"]
    rng = np.random.default_rng(seed)
    s = dict(case=c, n=n)
    if kind == "plasma":
        # thermal electrons at 0.01 (2D) or 0.1 (3D) of mc per axis, uniform in the cells
        two = n[1] == 1
        ncell = n[0] * n[1] * n[2]
        npart = ncell * c["ppc"]
        off = rng.random((npart, 3), dtype=np.float32)
        if two:
            off[:, 1] = 0.0
        u = rng.standard_normal((npart, 3), dtype=np.float32) * np.float32(0.01 if two else 0.1)
        dt = 0.5
        sim = _sim(c, n, (1.0, 1.0, 1.0), dt, 1.0, (0, 0, 0), ids=c["fp64"])
        sim.load_particles(np.repeat(np.arange(ncell, dtype=np.int32), c["ppc"]), off, u,
                           np.full(npart, 1.0 / c["ppc"], np.float32))
        s.update(sim=sim, dx=(1.0, 1.0, 1.0), dt=dt, bc=(0, 0, 0), gamma=1.0, ion=None)
    elif kind == "scan":
        s["sims"], s["of"] = [], []
        for i in range(c["instances"]):
            side, ppc, g, dx, dt, laser, dens = _scan_inputs(c, i)
            sim = _sim(c, (side, 1, side), dx, dt, g, (0, 0, 0))
            sim.load_lab_frame(laser=laser, plasma=(dens, -1e9, 0.0, ppc, (0.0, 0.0, 0.0), seed + i))
            s["sims"].append(sim)
            s["of"].append(dict(n=(side, 1, side), dx=dx, dt=dt, bc=(0, 0, 0), gamma=g, ion=(dens, -1e9, 0.0)))
        s["batch"] = pic.Batch(s["sims"])
    elif kind in ("lwfa", "read"):
        dx, dt, laser, plasma = _lwfa_inputs(c, seed)
        bc = (1, 1, 0 if c["periodic_z"] else 1)
        sim = _sim(c, n, dx, dt, c["gamma"], bc, ids=c["fp64"])
        sim.load_lab_frame(laser=laser, plasma=plasma)
        if kind == "read":
            sim.step(4)
        s.update(sim=sim, dx=dx, dt=dt, bc=bc, gamma=c["gamma"], ion=plasma[:3])
    elif kind == "beam":
        sz, sr = n[2] / 16.0, n[0] / 16.0
        total = 0.2 * math.sqrt(2 * math.pi) * sz * (sr / 4.0)
        bc = (1, 1, 0)
        sim = _sim(c, n, (1.0, 1.0, 1.0), 0.5, 1.0, bc, ids=True)
        sim.load_lab_frame(beam=(c["particles"], c["beam_gamma"], 1e-3, sr, sz, 5.0 * sz, total, seed))
        s.update(sim=sim, dx=(1.0, 1.0, 1.0), dt=0.5, bc=bc, gamma=1.0, ion=None)
        s["room"] = _particle_room(c["particles"], np.float32)
    else:
        ncell = n[0] * n[1] * n[2]
        npart = ncell * c["ppc"]
        p = dict(cell=rng.integers(0, ncell, npart, dtype=np.int32), off=rng.random((npart, 3), dtype=np.float32),
                 u=rng.standard_normal((npart, 3), dtype=np.float32), w=rng.random(npart, dtype=np.float32))
        s["host"] = {k: torch.from_numpy(v).pin_memory().numpy() for k, v in p.items()}
        s["sim"] = _sim(c, n, (1.0, 1.0, 1.0), 0.5, 1.0, (0, 0, 0), ids=True)
        s["room"] = _particle_room(npart, np.float32)
    if kind in ("plasma", "lwfa", "beam"):
        # page-locked room for the field read-out, and where an FP32 run keeps it
        s["comps"] = [pic.PIC_EX, pic.PIC_EZ] if n[0] * n[1] * n[2] > (1 << 23) else FIELDS
        s["wide"] = _pinned((len(s["comps"]), n[2], n[1], n[0]), torch.float64)
        s["count"] = c["particles"] if kind == "beam" else n[0] * n[1] * n[2] * c["ppc"]
        if not c["fp64"]:
            s["narrow"] = torch.empty(s["wide"].shape, dtype=torch.float32)
        else:
            s["room"] = _particle_room(s["sim"].num_particles(), np.float64)
    return s


def _read_fields(s):
    sim, wide = s["sim"], s["wide"]
    comps = (ctypes.c_int * len(s["comps"]))(*s["comps"])
    st = pic.lib().pic_get_fields(sim.h, comps, len(s["comps"]), ctypes.c_void_p(wide.data_ptr()), wide.numel())
    if st != pic.PIC_OK:
        raise pic.PicError(st, "pic_get_fields")
    return s["narrow"].copy_(wide) if "narrow" in s else wide


def _energies(d):
    return dict(field=d["field_energy"], kinetic=d["kinetic_energy"], charge=d["total_charge"])


def _by_id(p, n, count):
    """Position (cells) and momentum of every particle at the row of its id (a particle
    that has left the box: zero)."""
    n0, n1, _ = n
    cell, ids = torch.from_numpy(p["cell"]), torch.from_numpy(p["id"]).long()
    pos = torch.from_numpy(p["off"]).clone()
    pos[:, 0] += cell % n0
    pos[:, 1] += (cell // n0) % n1
    pos[:, 2] += cell // (n0 * n1)
    u = torch.from_numpy(p["u"])
    return dict(pos=pos.new_zeros(count, 3).index_copy_(0, ids, pos), u=u.new_zeros(count, 3).index_copy_(0, ids, u))


def run(s):
    c, kind = s["case"], s["case"]["kind"]
    if kind == "scan":
        s["batch"].step(c["steps"])
        s["batch"].synchronize()
        return [sim.get_fields([pic.PIC_EX, pic.PIC_EZ]).astype(np.float32) for sim in s["sims"]]
    sim = s["sim"]
    if kind == "load":
        h = s["host"]
        sim.load_particles(h["cell"], h["off"], h["u"], h["w"])
        p = sim.get_particles(stored=True, out=s["room"])
        return {k: p[k] for k in ("cell", "off", "u", "w", "id")}
    if kind == "read":
        return dict(energies=_energies(sim.diagnostics()), gauss=sim.gauss_residual()[1], rho=sim.get_field(pic.PIC_RHO))
    sim.step(c["steps"])
    out = dict(fields=_read_fields(s), energies=_energies(sim.diagnostics()))
    if c["fp64"] and kind == "plasma":
        out["particles"] = sim.get_particles(out=s["room"])
    elif c["fp64"] or kind == "beam":
        out["particles"] = _by_id(sim.get_particles(stored=True, out=s["room"]), s["n"], s["count"])
    return out


# ---- the work a pass cannot do without ------------------------------------------------
def _step_work(n, npart, c):
    ncell, es, dims = n[0] * n[1] * n[2], 8 if c["fp64"] else 4, 2 if n[1] == 1 else 3
    # the particles read and written once, E and B read and written once
    nbytes = 2 * npart * (4 + es * (dims + 4)) + 12 * es * ncell
    w = c["order"] + 1
    gather = 6 * 2 * (w ** dims + w ** (dims - 1) + w)
    deposit = 3 * (3 * w ** dims + 3 * w ** (dims - 1))
    grid = 70 + 3 * dims * 2 * (2 * c["passes"] + 1) * (c["passes"] > 0)
    return nbytes, npart * (gather + deposit + 160) + ncell * grid


def work(case):
    c, n, kind = case, (case["n0"], case["n1"], case["n2"]), case["kind"]
    ncell = n[0] * n[1] * n[2]
    npart = c["particles"] if kind == "beam" else ncell * c["ppc"]
    if kind == "load":
        return dict(bytes=npart * (32 + 36), flops=0)
    if kind == "read":
        w = (c["order"] + 1) ** 3
        return dict(bytes=npart * 48 + ncell * (24 + 12 + 8), flops=npart * (3 * w + 40) + ncell * 20)
    if kind == "scan":
        # mean side^2 of the log-uniform sides, mean particles per cell
        lo, hi = math.log(c["n0"]), math.log(c["n2"])
        side2 = (math.exp(2 * hi) - math.exp(2 * lo)) / (2 * (hi - lo))
        nb, fl = _step_work((side2, 1, 1), side2 * (c["ppc"] + 1) / 2, c)
        return dict(bytes=c["instances"] * (c["steps"] * nb + side2 * 8), flops=c["instances"] * c["steps"] * fl)
    nb, fl = _step_work(n, npart, c)
    read = ncell * (2 if ncell > (1 << 23) else 6) * (8 if c["fp64"] else 4)
    return dict(bytes=c["steps"] * nb + read, flops=c["steps"] * fl)


# ---- the same in 64 bits --------------------------------------------------------------
class _Ref:
    """The PIC step in FP64 torch tensors (fields (n2, n1, n0), x fastest)."""

    def __init__(self, sim, n, dx, dt, bc, gamma, ion, case):
        f64 = dict(dtype=torch.float64, device="cuda")
        self.n, self.dx, self.dt, self.c = n, dx, dt, case
        self.axes = [a for a in range(3) if not (a == 1 and n[1] == 1)]
        self.per = [b == 0 for b in bc]
        self.F = [torch.as_tensor(f, **f64) for f in sim.get_fields(FIELDS)]
        p = sim.get_particles()
        self.cell0 = torch.as_tensor(p["cell"], device="cuda").long()
        self.l = [self.cell0 % n[0], (self.cell0 // n[0]) % n[1], self.cell0 // (n[0] * n[1])]
        self.o = list(torch.as_tensor(p["off"], **f64).unbind(1))
        self.u = list(torch.as_tensor(p["u"], **f64).unbind(1))
        self.w = torch.as_tensor(p["w"], **f64)
        self.id = torch.as_tensor(p["id"], device="cuda").long()
        self.t, self.gamma, self.ion = 0, gamma, ion
        self.damp = [None] * 3
        for a in self.axes:
            if not self.per[a]:
                i = torch.arange(n[a], **f64)
                d = torch.clamp(torch.maximum(16 - i, i - (n[a] - 17)), min=0)
                self.damp[a] = (1.0 - 0.1 * (d / 16) ** 2).view([-1 if 2 - a == k else 1 for k in range(3)])

    def shift(self, f, a, by):
        """f at index + by along axis a (wrapped, or zero beyond an open face)."""
        if a not in self.axes:
            return f
        g = torch.roll(f, -by, 2 - a)
        if not self.per[a]:
            g.narrow(2 - a, self.n[a] - 1 if by > 0 else 0, 1).zero_()
        return g

    def nodal(self, l, o):
        if self.c["order"] == 1:
            return l, [1 - o, o]
        up = o >= 0.5
        f = o - up.double()
        return l + up.long() - 1, [0.5 * (0.5 - f) ** 2, 0.75 - f * f, 0.5 * (0.5 + f) ** 2]

    def stag(self, l, o):
        if self.c["order"] == 2:
            f = o - 0.5
            return l - 1, [0.5 * (0.5 - f) ** 2, 0.75 - f * f, 0.5 * (0.5 + f) ** 2]
        up = o >= 0.5
        f = torch.where(up, o - 0.5, o + 0.5)
        return torch.where(up, l, l - 1), [1 - f, f]

    def index(self, a, i):
        """Array index of node i along a and whether it is inside."""
        if self.per[a]:
            return i % self.n[a], None
        return i.clamp(0, self.n[a] - 1), (i >= 0) & (i < self.n[a])

    def spread(self, shapes):
        """(flat index, weight) of every node of the product of per-axis (first, weights)."""
        first = {a: shapes[a] for a in self.axes}
        rows = {}
        for a, (b, w) in first.items():
            rows[a] = []
            for m, v in enumerate(w):
                i, ok = self.index(a, b + m)
                rows[a].append((i, v if ok is None else v * ok))
        for iz, wz in rows[2]:
            for iy, wy in rows.get(1, [(None, None)]):
                row = iz if iy is None else iz * self.n[1] + iy
                wyz = wz if wy is None else wz * wy
                for ix, wx in rows[0]:
                    yield row * self.n[0] + ix, wyz * wx

    def gather(self):
        nod = {a: self.nodal(self.l[a], self.o[a]) for a in self.axes}
        sta = {a: self.stag(self.l[a], self.o[a]) for a in self.axes}
        out = []
        for comp in range(6):
            f, a = self.F[comp].reshape(-1), comp % 3
            stag = {b: (b == a) == (comp < 3) for b in self.axes}
            v = torch.zeros_like(self.w)
            for i, w in self.spread({b: (sta if stag[b] else nod)[b] for b in self.axes}):
                v += f[i] * w
            out.append(v)
        return out[:3], out[3:]

    def push(self, E, B):
        h, u = -0.5 * self.dt, self.u

        def cross(a, b):
            return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]

        def dot(a, b):
            return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]

        if self.c["boris"]:
            um = [u[k] + h * E[k] for k in range(3)]
            g = torch.sqrt(1 + dot(um, um))
            t = [h * B[k] / g for k in range(3)]
            f = 2 / (1 + dot(t, t))
            q = cross(um, t)
            q = cross([um[k] + q[k] for k in range(3)], [f * t[k] for k in range(3)])
            self.u = [um[k] + q[k] + h * E[k] for k in range(3)]
            return
        g = torch.sqrt(1 + dot(u, u))
        vb = cross([u[k] / g for k in range(3)], B)
        up = [u[k] + 2 * h * E[k] + h * vb[k] for k in range(3)]
        t = [h * B[k] for k in range(3)]
        tau2, us = dot(t, t), dot(up, t)
        sig = 1 + dot(up, up) - tau2
        q4 = tau2 + us * us
        root = torch.sqrt(sig * sig + 4 * q4)
        g2 = torch.where(sig >= 0, 0.5 * (sig + root), 2 * q4 / torch.where(sig >= 0, torch.ones_like(root), root - sig))
        g = torch.sqrt(g2)
        s = [t[k] / g for k in range(3)]
        f, ut, cr = 1 / (1 + dot(s, s)), dot(up, s), cross(up, s)
        self.u = [f * (up[k] + ut * s[k] + cr[k]) for k in range(3)]

    def shape_change(self, a, l1, o1):
        """Old shape and its change on the common window, and the window's first node."""
        W = self.c["order"] + 2
        (b0, w0), (b1, w1) = self.nodal(self.l[a], self.o[a]), self.nodal(l1, o1)
        ws = torch.minimum(b0, b1)

        def place(b, w):
            late = (b > ws).double()
            z = torch.zeros_like(w[0])
            return [(w[i] if i < W - 1 else z) * (1 - late) + (w[i - 1] if i else z) * late for i in range(W)]

        S0, S1 = place(b0, w0), place(b1, w1)
        return ws, S0, [y - x for x, y in zip(S0, S1)]

    def deposit(self, l1, o1, vy):
        n, W = self.n, self.c["order"] + 2
        dV = self.dx[0] * self.dx[1] * self.dx[2]
        qw = -self.w / dV
        J = [torch.zeros(n[0] * n[1] * n[2], dtype=torch.float64, device="cuda") for _ in range(3)]
        win = {a: self.shape_change(a, l1[a], o1[a]) for a in self.axes}
        at = {a: [self.index(a, win[a][0] + m) for m in range(W)] for a in self.axes}
        run = {}
        for a in self.axes:
            acc, run[a] = torch.zeros_like(self.w), []
            for m in range(W):
                acc = acc + win[a][2][m]
                run[a].append(acc * (-qw * self.dx[a] / self.dt))

        def put(comp, m, v):
            idx = None
            for a in (2, 1, 0):
                if a not in self.axes:
                    continue
                i, ok = at[a][m[a]]
                idx = i if idx is None else idx * n[a] + i
                if ok is not None:
                    v = v * ok
            J[comp].index_add_(0, idx, v)

        def average(a, i, b, j):
            """Time average of the product of the moving weights along a and b."""
            (_, Sa, Da), (_, Sb, Db) = win[a], win[b]
            return Sa[i] * (Sb[j] + 0.5 * Db[j]) + Da[i] * (0.5 * Sb[j] + Db[j] / 3.0)

        for a in self.axes:
            others = [b for b in self.axes if b != a]
            for j in range(W):
                for k in range(W) if len(others) == 2 else [0]:
                    if len(others) == 2:
                        tr = average(others[0], j, others[1], k)
                    else:
                        tr = win[others[0]][1][j] + 0.5 * win[others[0]][2][j]
                    for i in range(W - 1):
                        m = {a: i, others[0]: j, others[-1]: k if len(others) == 2 else j}
                        put(a, m, tr * run[a][i])
        if 1 not in self.axes:
            for i in range(W):
                for k in range(W):
                    put(1, {0: i, 2: k}, qw * vy * average(0, i, 2, k))
        return [j.view(n[2], n[1], n[0]) for j in J]

    def ion_charge_to(self, z):
        """Charge per area of the boosted ion profile between the box's start and z."""
        dens, zs, ramp = self.ion
        g, lz = self.gamma, self.n[2] * self.dx[2]
        if self.per[2]:
            return g * dens * z  # it fills the periodic box
        z = z.clamp(0.0, lz)
        up, top = zs / g, (zs + ramp) / g
        rise = 0.5 * (z.clamp(up, top) - up) ** 2 / (top - up) if ramp > 0 else 0.0
        return g * dens * (rise + (z - top).clamp(min=0.0))

    def ions(self, t, lo, hi):
        """Charge per area that sits in [z + lo dz, z + hi dz] around each plane at t."""
        beta = math.sqrt(1.0 - 1.0 / self.gamma ** 2)
        z = torch.arange(self.n[2], dtype=torch.float64, device="cuda") * self.dx[2] + beta * t
        return self.ion_charge_to(z + hi * self.dx[2]) - self.ion_charge_to(z + lo * self.dx[2])

    def particles(self):
        dt, n = self.dt, self.n
        E, B = self.gather()
        self.push(E, B)
        g = torch.sqrt(1 + self.u[0] ** 2 + self.u[1] ** 2 + self.u[2] ** 2)
        l1, o1 = list(self.l), list(self.o)
        for a in self.axes:
            x = self.o[a] + dt * (self.u[a] / g) / self.dx[a]
            k = torch.floor(x)
            o1[a], l1[a] = x - k, self.l[a] + k.long()
        J = self.deposit(l1, o1, self.u[1] / g)
        if self.ion is not None:
            beta = math.sqrt(1.0 - 1.0 / self.gamma ** 2)
            cross = self.ions((self.t + 0.5) * dt, 0.5 - 0.5 * beta * dt / self.dx[2], 0.5 + 0.5 * beta * dt / self.dx[2])
            J[2] -= (cross / dt).view(-1, 1, 1)
        live = None
        for a in self.axes:
            if self.per[a]:
                l1[a] = l1[a] % n[a]
            else:
                ok = (l1[a] >= 0) & (l1[a] < n[a])
                live = ok if live is None else live & ok
        self.l, self.o = l1, o1
        if live is not None and not bool(live.all()):
            self.l, self.o, self.u = ([v[live] for v in x] for x in (self.l, self.o, self.u))
            self.w, self.id = self.w[live], self.id[live]
        return J

    def diff(self, f, a, by):
        return (self.shift(f, a, 1) - f if by > 0 else f - self.shift(f, a, -1)) / self.dx[a] if a in self.axes else 0.0

    def curl_e(self, a, b):
        """d E_b / d a for the Faraday update (averaged across under the low-dispersion solver)."""
        f = self.diff(self.F[b], a, 1)
        if not self.c["ck"] or a not in self.axes:
            return f
        e = self.F[b]
        total = 0.0
        p, q = (a + 1) % 3, (a + 2) % 3
        for i in (-1, 0, 1):
            for j in (-1, 0, 1):
                g = self.shift(e, p, i) if i else e
                g = self.shift(g, q, j) if j else g
                total = total + (7 / 12, 1 / 12, 1 / 48)[abs(i) + abs(j)] * (self.shift(g, a, 1) - g)
        return total / self.dx[a]

    def damped(self, f):
        for d in self.damp:
            if d is not None:
                f = f * d
        return f

    def step(self):
        J = self.particles()
        for a in self.axes:
            for _ in range(self.c["passes"]):
                J = [0.25 * self.shift(j, a, -1) + 0.5 * j + 0.25 * self.shift(j, a, 1) for j in J]
        F, h = self.F, 0.5 * self.dt

        def faraday():
            return [F[3 + a] - h * (self.curl_e((a + 1) % 3, (a + 2) % 3) - self.curl_e((a + 2) % 3, (a + 1) % 3))
                    for a in range(3)]

        F[3:] = faraday()
        F[:3] = [self.damped(F[a] + self.dt * (self.diff(F[3 + (a + 2) % 3], (a + 1) % 3, -1)
                                               - self.diff(F[3 + (a + 1) % 3], (a + 2) % 3, -1) - J[a])) for a in range(3)]
        F[3:] = [self.damped(b) for b in faraday()]
        self.t += 1

    def energies(self):
        dV = self.dx[0] * self.dx[1] * self.dx[2]
        uu = self.u[0] ** 2 + self.u[1] ** 2 + self.u[2] ** 2
        return dict(field=0.5 * dV * float(sum((f * f).sum() for f in self.F)),
                    kinetic=float((self.w * (uu / (1 + torch.sqrt(1 + uu)))).sum()), charge=-float(self.w.sum()))

    def rho(self):
        dV = self.dx[0] * self.dx[1] * self.dx[2]
        r = torch.zeros(self.n[0] * self.n[1] * self.n[2], dtype=torch.float64, device="cuda")
        for i, w in self.spread({a: self.nodal(self.l[a], self.o[a]) for a in self.axes}):
            r.index_add_(0, i, w * (-self.w / dV))
        r = r.view(self.n[2], self.n[1], self.n[0])
        if self.ion is not None:
            r = r + (self.ions(self.t * self.dt, -0.5, 0.5) / self.dx[2]).view(-1, 1, 1)
        return r

    def canonical(self, tile=16):
        """Particles sorted by tile, in the order they were in before (periodic runs)."""
        t = [self.l[a] // (tile if len(self.axes) == 2 else 8) for a in range(3)]
        nt = [-(-v // (tile if len(self.axes) == 2 else 8)) for v in self.n]
        return torch.argsort(t[0] + nt[0] * (t[1] + nt[1] * t[2]), stable=True)


def exact(case, seed):
    c = case
    s = prepare(c, seed)
    if c["kind"] == "load":
        h, n = s["host"], s["n"]
        cell = torch.from_numpy(h["cell"]).long()
        t = [cell % n[0] // 8, cell // n[0] % n[1] // 8, cell // (n[0] * n[1]) // 8]
        order = torch.argsort(t[0] + -(-n[0] // 8) * (t[1] + -(-n[1] // 8) * t[2]), stable=True).numpy()
        return dict({k: h[k][order] for k in ("cell", "off", "u", "w")}, id=order.astype(np.int32))
    if c["kind"] == "scan":
        out = []
        for sim, of in zip(s["sims"], s["of"]):
            r = _Ref(sim, of["n"], of["dx"], of["dt"], of["bc"], of["gamma"], of["ion"], c)
            for _ in range(c["steps"]):
                r.step()
            out.append(torch.stack([r.F[0], r.F[2]]))
        return out
    r = _Ref(s["sim"], s["n"], s["dx"], s["dt"], s["bc"], s["gamma"], s["ion"], c)
    if c["kind"] == "read":
        r.t = 4
        rho = r.rho()
        gap = sum(r.diff(r.F[a], a, -1) for a in r.axes) - rho
        return dict(energies=r.energies(), gauss=float(torch.sqrt((gap * gap).mean())), rho=rho)
    if len(r.l[0]) * c["steps"] > 300e6:
        return None  # tens of seconds
    for _ in range(c["steps"]):
        r.step()
        if c["fp64"]:
            # the particles are kept sorted by tile after every step
            o = r.canonical()
            r.l, r.o, r.u = ([v[o] for v in x] for x in (r.l, r.o, r.u))
            r.w, r.id = r.w[o], r.id[o]
    out = dict(fields=torch.stack([r.F[k] for k in s["comps"]]), energies=r.energies())
    if c["fp64"] and c["kind"] == "plasma":
        out["particles"] = dict(cell=r.l[0] + s["n"][0] * (r.l[1] + s["n"][1] * r.l[2]), off=torch.stack(r.o, 1),
                                u=torch.stack(r.u, 1), w=r.w, id=r.id)
    elif c["fp64"] or c["kind"] == "beam":
        pos = torch.stack([r.l[a] + r.o[a] for a in range(3)], 1)
        rows = pos.new_zeros(s["count"], 3)
        out["particles"] = dict(pos=rows.index_copy(0, r.id, pos), u=rows.index_copy(0, r.id, torch.stack(r.u, 1)))
    return out
