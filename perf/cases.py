"""Performance cases: the work users have this library do, through its Python
entry points (`paper_1309_7859_gb300.memd`).

A case is a dict of plain values; `kind` says which calls a pass makes:

  md        one system: `steps` thermostatted steps, then its positions,
            velocities, image counters and forces read back (a simulation
            between two samples)
  io        one system driven by a host program: state in, one step, state
            and forces out (`step_io(1, load=True)`)
  batch     `count` independent replicas stepped together `steps` times, then
            every replica's state and forces read back
  batchio   the same batch driven by a host program, one step a call
  setup     a new system from scratch: permittivity mapped and homogenised,
            charges placed, the field solved, forces and energies read
  snapshot  checkpoint of one system, restored into another, whose energies,
            fields and particles are read
  live      a medium that follows its salt: permittivity from the present
            salt density, then `steps` steps, state and forces read back

Sizes, profiles, time step and thermostat are those of the repository's own
workloads (`paper_1309_7859_gb300/inputs.py`, `bench.py`, the tests' ragged
meshes).  `exact` is the method in plain torch and numpy, 64 bits throughout.

The forces, energies and fields of an FP32 system are FP32 numbers that the
interface hands out in FP64 arrays; they are returned in FP32, where every
one of them is exact (the energies, FP64 sums of FP32 fields, are rounded).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1309_7859_gb300 import inputs, memd

TH = (1.0, 1.0)          # Langevin: gamma, kT
DT = 0.005
S = 1 << 16              # sub-cell steps of the fixed point
SALT_RULE = (60.0, -20.0, 40.0, 80.0, 2.0)   # eps0, slope, lowest, highest, sigma


# ------------------------------------------------------------------ the cases
def _one(name, kind, mesh, n, eps, precision, steps, cell=1.0):
    c = {"name": name} if name else {}
    return {**c, "kind": kind, "nx": mesh[0], "ny": mesh[1], "nz": mesh[2], "n": n, "eps": eps,
            "precision": precision, "steps": steps, "cell": cell}


def _many(name, kind, count, meshes, nmin, nmax, precision, steps):
    c = {"name": name} if name else {}
    return {**c, "kind": kind, "count": count, "meshes": meshes, "nmin": nmin, "nmax": nmax,
            "precision": precision, "steps": steps}


def listed():
    return [
        # the smallest system there is, driven step by step from a host
        # program: nothing but latency
        _one("io-8-fp64", "io", (8, 8, 8), 16, "const", "fp64", 1),
        # the paper's kind of slab between two samples: small, in L2
        _one("md-slab32-fp32", "md", (32, 32, 32), 1000, "tanh", "fp32", 50),
        # double precision on a ragged box whose cell is no power of two
        _one("md-ragged-fp64", "md", (45, 38, 51), 3000, "vertices", "fp64", 20, 0.9),
        # an electrolyte with many charges: the particle kernels
        _one("md-salt64-fp32", "md", (64, 64, 64), 32768, "sin", "fp32", 20),
        # an odd width: no rows of whole vectors
        _one("md-odd95-fp32", "md", (95, 95, 95), 20000, "vertices", "fp32", 10),
        # the largest single system: bound by HBM
        _one("md-slab256-fp32", "md", (256, 256, 256), 100000, "tanh", "fp32", 5),
        # many replicas at once, the throughput workload, and the same driven
        # from the host
        _many("batch-64-fp32", "batch", 64, "16,24,32,48", 200, 8000, "fp32", 10),
        _many("batchio-64-fp32", "batchio", 64, "16,24,32,48", 200, 8000, "fp32", 1),
        # setting a system up, as the request server does for every request:
        # an even mesh and an odd one (its stream draws both alike)
        _one("setup-48-fp32", "setup", (48, 48, 48), 2200, "vertices", "fp32", 0),
        _one("setup-77-fp32", "setup", (77, 77, 77), 10000, "vertices", "fp32", 0),
        # checkpoint, restore, energies and fields of a double-precision run
        _one("snapshot-64-fp64", "snapshot", (64, 64, 64), 8000, "sin", "fp64", 2),
        # a medium that is made anew from its salt between blocks of steps
        _one("live-salt60-fp32", "live", (60, 60, 60), 20000, "sin", "fp32", 10),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _even(x, lo=2):
    n = int(round(x))
    return max(lo, n - n % 2)


def _mesh(rng, lo, hi):
    """Three extents around one size, odd ones as likely as even ones."""
    N = _log(rng, lo, hi)
    if rng.random() < 0.4:  # a cube of any width
        return (max(lo, int(round(N))),) * 3
    return tuple(int(min(hi, max(lo, round(N * rng.uniform(0.75, 1.3))))) for _ in range(3))


def draw(rng):
    c = _draw(rng)
    while work(c)["bytes"] > 4.5e9:   # no longer than the largest listed one
        c["steps"] -= 1
    return c


def _draw(rng):
    kind = rng.choice(["md", "md", "md", "io", "batch", "batchio", "setup", "setup",
                       "live", "snapshot"])
    prec = rng.choice(["fp32", "fp32", "fp64"])
    cell = rng.choice([1.0, 1.0, 0.9, 1.25])
    eps = rng.choice(["const", "tanh", "sin", "vertices"])
    if kind in ("md", "io"):
        m = _mesh(rng, 8, 160)
        V = m[0] * m[1] * m[2]
        n = _even(_log(rng, 16, max(32, min(100000, V // 4))))
        steps = 1 if kind == "io" else max(2, min(50, int(rng.uniform(0.3, 1.0) * 4e7 / V)))
        return _one("", kind, m, n, eps, prec, steps, cell)
    if kind == "setup":
        m = _mesh(rng, 12, 110)
        V = m[0] * m[1] * m[2]
        return _one("", kind, m, _even(_log(rng, 100, max(200, min(50000, V // 4)))), eps, prec,
                    0, cell)
    if kind in ("live", "snapshot"):
        m = _mesh(rng, 16, 80)
        V = m[0] * m[1] * m[2]
        return _one("", kind, m, _even(_log(rng, 100, min(32768, V // 4))), eps, prec,
                    rng.randint(1, 5), cell)
    sizes = sorted(rng.sample([12, 16, 20, 24, 27, 32, 37, 40, 48], rng.randint(1, 4)))
    return _many("", kind, rng.randint(4, 64), ",".join(map(str, sizes)), 200,
                 _even(_log(rng, 400, 8000)), prec,
                 1 if kind == "batchio" else rng.randint(5, 20))


# ----------------------------------------------------------------- the inputs
def _eps(rng, kind, mesh, box, cell):
    if kind == "const":
        return inputs.EpsSpec("const", 0, (float(rng.uniform(1.0, 80.0)),))
    if kind == "tanh":   # a slab somewhere, eps 2 to 80 on either side
        ax = int(rng.integers(0, 3))
        L = box[ax]
        e = rng.uniform(2.0, 80.0, size=2)
        return inputs.EpsSpec("tanh", ax, (float(0.5 * (e[0] + e[1])), float(0.5 * (e[1] - e[0])),
                                           float(rng.uniform(0.0, L)),
                                           float(rng.uniform(L / 8, L / 4)), 1.5 * cell))
    if kind == "sin":
        return inputs.EpsSpec("sin", int(rng.integers(0, 3)),
                              (60.0, -20.0, float(rng.uniform(0.0, 6.28))))
    return inputs.EpsSpec("vertices", 0, (), inputs.smooth_random_vertices(rng, mesh))


def _system(mesh, n, eps, precision, cell, seed, steps):
    rng = np.random.default_rng(seed)
    box = tuple(N * cell for N in mesh)
    e = _eps(rng, eps, mesh, box, cell)
    q = inputs.neutral_charges(rng, n)
    if eps == "sin":   # the salt follows its profile
        x = inputs.sine_modulated_positions(rng, n, box, e.axis, 0.5)
    else:
        x = inputs.uniform_positions(rng, n, box)
    return inputs.System(name="", mesh=tuple(mesh), box=box, eps=e, c_light=1.0, dt=DT,
                         precision=precision, x=x, q=q, m=np.ones(n),
                         v=inputs.thermal_velocities(rng, n), steps=steps, thermostat=TH,
                         seed=int(seed))


def _systems(case, seed):
    """The systems of a case; the members of a batch have sizes set by the
    case alone."""
    if "count" not in case:
        return [_system((case["nx"], case["ny"], case["nz"]), case["n"], case["eps"],
                        case["precision"], case["cell"], seed, case["steps"])]
    out = []
    for r, (N, n) in enumerate(_members(case)):
        out.append(_system((N, N, N), n, "tanh", case["precision"], 1.0, seed * 4096 + r,
                           case["steps"]))
    return out


def _members(case):
    """(mesh width, charges) of every replica: the widths in turn, the charges
    spread over their range's logarithm."""
    sizes = [int(t) for t in case["meshes"].split(",")]
    out = []
    for r in range(case["count"]):
        N = sizes[r % len(sizes)]
        n = case["nmin"] * (case["nmax"] / case["nmin"]) ** ((r * 0.7548776662 + 0.17) % 1.0)
        out.append((N, _even(min(n, N ** 3 // 2))))
    return out


# ------------------------------------------------------------ what a user has
class _Held:
    """The library's page-locked arrays live as long as their owner: this
    keeps the owner with the array."""

    def __init__(self, array, owner):
        self.__array_interface__ = array.__array_interface__
        self.owner = owner


def prepare(case, seed):
    kind = case["kind"]
    sys = _systems(case, seed)
    stream = torch.cuda.Stream()
    fp32 = case["precision"] == "fp32"
    st = {"case": case, "sys": sys, "stream": stream, "fp32": fp32}
    if kind == "setup":
        return st
    made = []
    for s in sys:
        g = memd.from_system(s, stream=stream)
        g.init_field(s.x, s.q, s.m, s.v)
        made.append(g)
    st["made"] = made
    if kind == "snapshot":
        made[0].step(case["steps"], TH)
        other = memd.from_system(sys[0], stream=stream)  # where the checkpoint is restored
        other.init_field(sys[0].x[::-1], sys[0].q[::-1], sys[0].m, sys[0].v)
        st["other"] = other
        return st
    if "count" in case:
        st["runner"] = memd.Batch(made)
        io = st["runner"].io_buffers()
    else:
        st["runner"] = made[0]
        io = made[0].io_buffers()
    io["pos"][...] = np.concatenate([s.x for s in sys])
    io["vel"][...] = np.concatenate([s.v for s in sys])
    io["img"][...] = 0
    st["io"] = {k: np.asarray(_Held(a, st["runner"])) for k, a in io.items() if k != "offsets"}
    st["f"] = torch.from_numpy(st["io"]["f"])
    st["f32"] = torch.empty(st["f"].shape, dtype=torch.float32)
    return st


def _fp(st, a):
    """Numbers of the system's field precision."""
    return a.astype(np.float32) if st["fp32"] else a


def _energies(st, e):
    return [_fp(st, np.array([e[k] for k in ("kinetic", "electric", "magnetic", "self", "dipole",
                                             "total", "P0", "P1", "P2")])), int(e["gauss_exact"])]


def _moved(st):
    io = st["io"]
    f = st["f32"].copy_(st["f"]) if st["fp32"] else st["f"]
    return [io["pos"], io["vel"], io["img"], f]


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "setup":
        s = st["sys"][0]
        g = memd.from_system(s, stream=st["stream"])
        g.init_field(s.x, s.q, s.m, s.v)
        out = [_fp(st, g.forces())] + _energies(st, g.energy())
        g.close()
        return out
    if kind == "snapshot":
        g, h = st["made"][0], st["other"]
        h.load_state(g.save_state())
        e = _energies(st, h.energy())
        D, B, Lg = h.fields()
        x, v, img = h.particles()
        return [x, v, img, _fp(st, h.forces()), _fp(st, D), _fp(st, B), Lg] + e
    ev = [st["runner"].eps_from_density(*SALT_RULE)] if kind == "live" else []
    st["runner"].step_io(case["steps"], TH, load=kind in ("io", "batchio"))
    return _moved(st) + ev


def work(case):
    """Bytes: a step reads D, B and 1/eps and writes D and B of every site; a
    charge's state (position, velocity, force, image, valence and three
    constants) is read once and written once, and the transfer, ledger, D
    and 1/eps words of its cell's twelve links are touched once.  A setup
    reads the permittivity and the charges and writes the fields, 1/eps, the
    ledger and the forces once.  Operations: the stencil's and the gather's."""
    es = 4 if case["precision"] == "fp32" else 8
    kind, steps = case["kind"], case["steps"]
    if "count" in case:
        mem = _members(case)
        V, n = sum(N ** 3 for N, _ in mem), sum(k for _, k in mem)
    else:
        V, n = case["nx"] * case["ny"] * case["nz"], case["n"]
    step_b = 15 * es * V + n * (176 + 12 * (16 + 2 * es))
    step_f = 33 * V + 400 * n
    make_b = V * (8 + 3 * 8 + 9 * es + 48) + n * 120
    make_f = 200 * V + 400 * n
    if kind == "setup":
        return {"bytes": make_b, "flops": make_f}
    if kind == "snapshot":   # the state out, in again, then read
        state = V * (6 * es + 24) + n * 120
        return {"bytes": 3 * state, "flops": 40 * V}
    if kind == "live":
        return {"bytes": V * (8 + 3 * es + 24) + steps * step_b, "flops": 60 * V + steps * step_f}
    io = 4 * 24 * n if kind in ("io", "batchio") else 0
    return {"bytes": steps * step_b + io, "flops": steps * step_f}


# --------------------------------------------- the same in plain 64-bit torch
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _up(a, d):     # a at the site one further along axis d (x, y, z)
    return torch.roll(a, -1, dims=-1 - d)


def _dn(a, d):
    return torch.roll(a, 1, dims=-1 - d)


def _eps_links(e, mesh, a):
    """eps of the links, [3, nz, ny, nx]."""
    dev = _dev()
    nx, ny, nz = mesh
    out = torch.empty((3, nz, ny, nx), dtype=torch.float64, device=dev)
    if e.kind == "vertices":
        ev = torch.as_tensor(np.asarray(e.values), dtype=torch.float64, device=dev)
        ev = ev.reshape(nz, ny, nx)
        for d in range(3):
            out[d] = 0.5 * (ev + _up(ev, d))
        return out
    if e.kind == "const":
        out.fill_(e.params[0])
        return out
    p, ax = e.params, e.axis
    L = mesh[ax] * a
    shape = [1, 1, 1]
    shape[2 - ax] = mesh[ax]
    for d in range(3):
        s = (torch.arange(mesh[ax], dtype=torch.float64, device=dev) + (0.5 if d == ax else 0.0)) * a
        if e.kind == "tanh":
            t = s - p[2]
            t = t - L * torch.round(t / L)
            val = p[0] + p[1] * torch.tanh((t.abs() - p[3]) / p[4])
        else:
            val = p[0] + p[1] * torch.sin(2.0 * math.pi * s / L + p[2])
        out[d] = val.reshape(shape)
    return out


def _lambda(mesh):
    """Eigenvalues of -Laplace on the unit lattice, [nz, ny, nx // 2 + 1]."""
    dev = _dev()
    w = [4.0 * torch.sin(math.pi * torch.arange(N, dtype=torch.float64, device=dev) / N) ** 2
         for N in mesh]
    return w[2][:, None, None] + w[1][None, :, None] + w[0][None, None, : mesh[0] // 2 + 1]


def _poisson(eps, f, a):
    """phi_k of zero mean with -div(eps grad phi_k) = f_k, by conjugate gradients."""
    mesh = eps.shape[:0:-1]
    lam = _lambda(mesh)
    lam = torch.where(lam == 0.0, lam[lam > 0].min(), lam)
    dims = (-3, -2, -1)
    vert = sum(eps[d] + _dn(eps[d], d) for d in range(3)) / 6.0
    s = torch.rsqrt(vert) * a

    def op(p):
        return sum(eps[d] * (p - _up(p, d)) + _dn(eps[d], d) * (p - _dn(p, d))
                   for d in range(3)) / (a * a)

    def pre(r):
        z = torch.fft.irfftn(torch.fft.rfftn(r * s, dim=dims) / lam, s=r.shape[-3:], dim=dims) * s
        return z - z.mean(dim=dims, keepdim=True)

    def dot(u, v):
        return (u * v).sum(dim=dims, keepdim=True)

    r = f - f.mean(dim=dims, keepdim=True)
    x = torch.zeros_like(r)
    f2 = dot(r, r).clamp_min(1e-300)
    z = pre(r)
    p = z.clone()
    rz = dot(r, z)
    best, stale = math.inf, 0
    for _ in range(400):
        live = dot(r, r) > 1e-30 * f2      # the others have arrived
        q = op(p)
        pq = dot(p, q)
        al = torch.where(live & (pq > 0), rz / pq.clamp_min(1e-300), torch.zeros_like(pq))
        x = x + al * p
        r = r - al * q
        res = float((dot(r, r) / f2).max())
        stale = 0 if res < 0.5 * best else stale + 1
        best = min(best, res)
        if res < 1e-30 or stale >= 20:
            break
        z = pre(r)
        rz2 = dot(r, z)
        p = z + torch.where(rz > 0, rz2 / rz.clamp_min(1e-300), torch.zeros_like(rz)) * p
        rz = rz2
    return x - x.mean(dim=dims, keepdim=True)


class _Exact:
    """One system of the method in 64 bits."""

    def __init__(self, s):
        dev = _dev()
        self.mesh, self.a, self.seed = s.mesh, s.box[0] / s.mesh[0], s.seed
        self.L = torch.tensor(s.box, dtype=torch.float64, device=dev)
        self.N = torch.tensor(s.mesh, dtype=torch.int64, device=dev)
        self.V = int(np.prod(s.mesh))
        self.box_v = float(np.prod(s.box))
        self.x = torch.as_tensor(s.x, device=dev)
        self.v = torch.as_tensor(s.v, device=dev).clone()
        self.q = torch.as_tensor(s.q, device=dev).to(torch.int64)
        self.m = torch.as_tensor(s.m, device=dev)
        self.img = torch.zeros_like(self.x, dtype=torch.int64)
        self.step_no = 0
        # the lattice Green's function at the offsets {0, 1}^3
        lam = _lambda(self.mesh)
        ghat = torch.where(lam > 0, 1.0 / lam.clamp_min(1e-300), torch.zeros_like(lam))
        g = torch.fft.irfftn(ghat, s=self.mesh[::-1])
        self.G = [[[float(g[k, j, i]) for i in (0, 1)] for j in (0, 1)] for k in (0, 1)]
        self.set_eps(_eps_links(s.eps, s.mesh, self.a))

    def set_eps(self, eps):
        a = self.a
        self.eps, self.ie = eps, 1.0 / eps
        f = torch.stack([-(eps[d] - _dn(eps[d], d)) / a for d in range(3)])
        psi = _poisson(eps, f, a)
        self.cellflux = [torch.stack([eps[e] * ((1.0 if e == d else 0.0)
                                                - (_up(psi[d], e) - psi[d]) / a)
                                      for e in range(3)]) for d in range(3)]
        M = np.array([[float(self.cellflux[d][e].mean()) for d in range(3)] for e in range(3)])
        Mi = np.linalg.inv(M)
        self.Mi, self.Minv = Mi, 0.5 * (Mi + Mi.T)

    def quant(self, x):
        u = x / self.a
        c = torch.floor(u)
        f = torch.floor((u - c) * S).to(torch.int64)
        return c.to(torch.int64), f

    def vid(self, c):
        c = torch.remainder(c, self.N)
        return c[:, 0] + self.mesh[0] * (c[:, 1] + self.mesh[1] * c[:, 2])

    def vertex_charge(self, q):
        """Cloud-in-cell charge of the vertices in units of 2^-48, int64."""
        c, f = self.quant(self.x)
        out = torch.zeros(self.V, dtype=torch.int64, device=self.x.device)
        for t in range(8):
            o = torch.tensor([t & 1, t >> 1 & 1, t >> 2], device=c.device)
            w = torch.where(o == 1, f, S - f).prod(dim=1)
            out.index_add_(0, self.vid(c + o), q * w)
        return out

    def dipole(self):
        c, f = self.quant(self.x)
        u = (self.img * self.N + c) * S + f
        return (self.q[:, None] * u).sum(0).double().cpu().numpy() * (self.a / S)

    def init(self):
        a = self.a
        rho = self.vertex_charge(self.q).double().reshape(self.mesh[::-1]) * 2.0 ** -48
        phi = _poisson(self.eps, (rho / a ** 3)[None], a)[0]
        D = torch.stack([-self.eps[d] * (_up(phi, d) - phi) / a for d in range(3)])
        mean = D.mean(dim=(1, 2, 3)).cpu().numpy()
        E0 = self.Mi @ (-self.dipole() / self.box_v - mean)
        for d in range(3):
            D = D + E0[d] * self.cellflux[d]
        self.D, self.B = D, torch.zeros_like(D)
        self.gather()
        self.Ft = self.F

    def links(self, c, f, d):
        """The four d-links of every charge's cell: field index, weight."""
        e1, e2 = (d + 1) % 3, (d + 2) % 3
        for a2 in (0, 1):
            for a1 in (0, 1):
                cc = c.clone()
                cc[:, e1] += a1
                cc[:, e2] += a2
                w = (f[:, e1] if a1 else S - f[:, e1]) * (f[:, e2] if a2 else S - f[:, e2])
                yield d * self.V + self.vid(cc), w

    def self_terms(self, f):
        t = f.double() / S
        c1 = 2.0 * t * (1.0 - t)
        cc, dc = (1.0 - c1, c1), (4.0 * t - 2.0, 2.0 - 4.0 * t)
        U, g = 0.0, [0.0, 0.0, 0.0]
        for k in (0, 1):
            for j in (0, 1):
                for i in (0, 1):
                    G = self.G[k][j][i]
                    x, y, z = cc[i][:, 0], cc[j][:, 1], cc[k][:, 2]
                    U = U + G * x * y * z
                    g[0] = g[0] + G * dc[i][:, 0] * y * z
                    g[1] = g[1] + G * x * dc[j][:, 1] * z
                    g[2] = g[2] + G * x * y * dc[k][:, 2]
        return U, g

    def cell_ie(self, c, f):
        ie = self.ie.reshape(-1)
        return sum(ie[l] for d in range(3) for l, _ in self.links(c, f, d)) / 12.0

    def gather(self):
        c, f = self.quant(self.x)
        D, ie, q = self.D.reshape(-1), self.ie.reshape(-1), self.q.double()
        MP = self.Minv @ self.dipole() / self.box_v
        ic = self.cell_ie(c, f)
        _, g = self.self_terms(f)
        F = []
        for d in range(3):
            E = sum(D[l] * ie[l] * (w.double() / S ** 2) for l, w in self.links(c, f, d))
            F.append(q * E + q * q / (2.0 * self.a) * ic * g[d] / self.a + q * MP[d])
        self.F = torch.stack(F, dim=1)

    def circ(self):
        E = self.D * self.ie
        out = []
        for d in range(3):
            e1, e2 = (d + 1) % 3, (d + 2) % 3
            out.append(E[e1] + _up(E[e2], e1) - _up(E[e1], e2) - E[e2])
        return torch.stack(out)

    def noise(self):
        n = self.x.shape[0]
        lo32 = np.uint64(0xFFFFFFFF)
        c = [np.arange(n, dtype=np.uint64), np.zeros(n, np.uint64),
             np.full(n, self.step_no, np.uint64), np.zeros(n, np.uint64)]
        k0, k1 = self.seed & 0xFFFFFFFF, (self.seed >> 32) & 0xFFFFFFFF
        for _ in range(10):   # Philox4x32-10 (Salmon et al., SC'11)
            p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
            c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & lo32,
                 (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & lo32]
            k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
        r = np.stack(c[:3], axis=1).astype(np.float64)
        xi = math.sqrt(3.0) * (2.0 * ((r + 0.5) * 2.0 ** -32) - 1.0)
        return torch.as_tensor(xi, device=self.x.device)

    def step(self, gamma=TH[0], kT=TH[1]):
        a, dt, dev = self.a, DT, self.x.device
        h = (0.5 * dt / self.m)[:, None]
        self.v = self.v + h * self.Ft
        self.B = self.B - dt / a * self.circ()
        # drift and charge transfer, axis by axis
        c0, f0 = self.quant(self.x)
        xn = self.x + dt * self.v
        turn = torch.floor(xn / self.L)
        xn = xn - turn * self.L
        turn = turn.to(torch.int64)
        c1, f1 = self.quant(xn)
        T = torch.zeros(3 * self.V, dtype=torch.int64, device=dev)
        cc, cf = c0.clone(), f0.clone()
        for d in range(3):
            hop = c1[:, d] + turn[:, d] * self.N[d] - c0[:, d]   # -1, 0 or 1
            # signed sub-cell distance in the old and in the new cell
            old = torch.where(hop == 0, f1[:, d] - f0[:, d],
                              torch.where(hop > 0, S - f0[:, d], -f0[:, d]))
            new = torch.where(hop == 0, 0, torch.where(hop > 0, f1[:, d], f1[:, d] - S))
            for l, w in self.links(cc, cf, d):
                T.index_add_(0, l, -self.q * old * w)
            there = cc.clone()
            there[:, d] += hop
            for l, w in self.links(there, cf, d):
                T.index_add_(0, l, -self.q * new * w)
            cc[:, d], cf[:, d] = c1[:, d], f1[:, d]
        self.x, self.img = xn, self.img + turn
        D = []
        for d in range(3):
            e1, e2 = (d + 1) % 3, (d + 2) % 3
            D.append(self.D[d] + dt / a * (self.B[e2] - _dn(self.B[e2], e1) - self.B[e1]
                                           + _dn(self.B[e1], e2)))
        self.D = torch.stack(D) + (T.double() * (2.0 ** -48 / (a * a))).reshape(self.D.shape)
        self.gather()
        sig = torch.sqrt(2.0 * gamma * self.m * kT / dt)[:, None]
        self.Ft = self.F + (-gamma * self.m[:, None] * self.v + sig * self.noise())
        self.v = self.v + h * self.Ft
        self.step_no += 1

    def salt_eps(self, eps0, slope, lo, hi, sigma):
        rho = self.vertex_charge(self.q.abs()).double().reshape(self.mesh[::-1]) * 2.0 ** -48
        R = math.ceil(3.0 * sigma)
        w = [math.exp(-j * j / (2.0 * sigma * sigma)) for j in range(-R, R + 1)]
        for d in range(3):
            rho = sum(wj / sum(w) * torch.roll(rho, -j, dims=-1 - d)
                      for j, wj in zip(range(-R, R + 1), w))
        ev = (eps0 + slope * (rho / rho.mean() - 1.0)).clamp(lo, hi)
        self.set_eps(torch.stack([0.5 * (ev + _up(ev, d)) for d in range(3)]))
        self.gather()
        self.Ft = self.F
        return ev

    def energies(self):
        a = self.a
        c, f = self.quant(self.x)
        q = self.q.double()
        U, _ = self.self_terms(f)
        P = self.dipole()
        e = [float((0.5 * self.m[:, None] * self.v ** 2).sum()),
             float((self.D ** 2 * self.ie).sum()) * 0.5 * a ** 3,
             float((self.B * (self.B - DT / a * self.circ())).sum()) * 0.5 * a ** 3,
             float((q * q / (2.0 * a) * self.cell_ie(c, f) * U).sum()),
             float(0.5 * P @ self.Minv @ P / self.box_v)]
        return np.array(e + [e[0] + e[1] + e[2] - e[3] - e[4], *P])


def exact(case, seed):
    kind = case["kind"]
    got, ev = [], []
    for s in _systems(case, seed):
        x = _Exact(s)
        x.init()
        if kind == "live":
            ev = [x.salt_eps(*SALT_RULE)]
        for _ in range(case["steps"]):
            x.step()
        got.append(x)
    if kind == "setup":
        return [got[0].F, got[0].energies(), None]
    if kind == "snapshot":
        x = got[0]
        return [x.x, x.v, None, x.F, x.D, x.B, None, x.energies(), None]
    return [torch.cat([x.x for x in got]), torch.cat([x.v for x in got]), None,
            torch.cat([x.F for x in got])] + ev
