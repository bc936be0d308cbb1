"""Cases that time the voxel electrophysiology step through its public entry points.

A pass restores a checkpoint from pinned host memory (``Sim.write_state``), advances the model
(``Sim.step`` or ``Batch.step``) and takes the new state back (``Sim.read_state``): what a program that
resumes, steps and saves a simulation does, and a pass starts from the same state every time.

Inputs are made on the GPU from the seed alone: masks, fibres and a travelling front (excited tissue
below a tilted plane, gates recovering behind it).  The first guess of v_e is -g v, the elliptic solution
when the two tensors are proportional, so that a solve starts warm, as it does inside a run.

Sizes and parameters follow the repository's own workloads: the 32^3 FP64 slab, the 128^3 shell, the 256^3
biventricular heart, the dense slab, shells of 48 to 160 voxels side by side, and the heart in a conducting
torso (its v_e starts from 0).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2302_12519_gb300 as ep

DEV = "cuda"


class _Params:
    """Parameter set of ``Sim.set_params`` (Mitchell-Schaeffer constants, conductivities, solver)."""

    def __init__(self, c):
        self.tau_in, self.tau_out, self.tau_open, self.tau_close, self.v_gate = 0.3, 6.0, 120.0, 150.0, 0.13
        self.sig_iL, self.sig_iT, self.sig_eL, self.sig_eT = c["siL"], c["siT"], c["seL"], c["seT"]
        self.lam, self.K, self.dt = 1.0, 1.0, c["dt"]
        self.omega = c["omega"]
        self.rel_tol, self.check_every, self.max_iter = 1e-6, 10, 50000
        self.diffusion = ep.EP_IMPLICIT if c["implicit"] else ep.EP_EXPLICIT
        self.solver = {"jacobi": ep.EP_SOLVER_JACOBI, "chebyshev": ep.EP_SOLVER_CHEBYSHEV,
                       "sor": ep.EP_SOLVER_GAUSS_SEIDEL}[c["solver"]]
        self.cheb_lmin = self.cheb_lmax = 0.0


def _case(geom, nx, ny, nz, model, **kw):
    c = {"geom": geom, "nx": nx, "ny": ny, "nz": nz, "model": model, "fp64": False, "implicit": False,
         "solver": "jacobi", "omega": 0.0, "steps": 1, "dx": 0.5, "dt": 0.05, "siL": 0.20, "siT": 0.05,
         "seL": 0.20, "seT": 0.05, "torso": False, "front": 0.45, "members": 0}
    c.update(kw)
    return c


def listed():
    """The work a user of the framework has it do, from the smallest calls to the whole heart."""
    return [
        # the double-precision reference slab of the benchmark problem
        _case("slab", 32, 32, 32, "mono", fp64=True, dx=0.25, dt=0.01, steps=100, name="slab32_mono_fp64"),
        # a small tissue sample, ragged sizes: latency and launches count
        _case("slab", 61, 45, 53, "mono", steps=400, name="slab61_mono"),
        # a dense tissue block, memory far above L2: the fused reaction-diffusion step
        _case("slab", 256, 256, 256, "mono", steps=100, name="slab256_mono"),
        # the same model with implicit diffusion, which allows large steps
        _case("slab", 161, 160, 158, "mono", implicit=True, dt=0.2, steps=20, name="slab160_mono_implicit"),
        # the smallest ventricle shell of the parameter studies, the method's own solve
        _case("shell", 48, 48, 48, "bi", steps=2, name="shell48_jacobi"),
        # the ellipsoidal ventricle
        _case("shell", 128, 128, 128, "bi", name="shell128_jacobi"),
        # the biventricular heart: the framework's main workload
        _case("biv", 256, 256, 256, "bi", name="biv256_jacobi"),
        # the ventricle with the accelerated solve and unequal anisotropy
        _case("shell", 128, 128, 128, "bi", solver="chebyshev", seT=0.10, steps=4, name="shell128_chebyshev"),
        # the heart with the accelerated solve: long production runs
        _case("biv", 256, 256, 256, "bi", solver="chebyshev", steps=4, name="biv256_chebyshev"),
        # the heart at a coarser voxel size with the over-relaxed in-place solve, early in the beat
        _case("biv", 176, 176, 176, "bi", solver="sor", omega=1.8, front=0.05, name="biv176_sor"),
        # the heart in a conducting torso (the ECG set-up), early in the beat
        _case("biv", 144, 144, 144, "bi", solver="chebyshev", torso=True, front=0.02,
              name="biv144_torso_chebyshev"),
        # shells of many sizes and conductivities advanced together (parameter study)
        _case("shell", 160, 160, 160, "bi", solver="chebyshev", members=10, steps=2, name="batch10_chebyshev"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: ragged sizes, other conductivities, every solver and geometry."""
    kind = rng.choice(["mono", "mono", "implicit", "jacobi", "jacobi", "chebyshev", "chebyshev", "sor", "torso",
                       "batch"])
    siL = rng.uniform(0.15, 0.25)
    siT = siL / rng.uniform(3.0, 5.0)
    sig = {"siL": siL, "siT": siT, "seL": siL, "seT": siT}
    if kind in ("mono", "implicit"):
        top = 250 if kind == "mono" else 170
        n = [max(5, int(_log(rng, 24, top) * rng.uniform(0.8, 1.0))) for _ in range(3)]
        vox = n[0] * n[1] * n[2]
        geom = rng.choice(["slab", "slab", "shell"])
        if kind == "implicit":
            return _case(geom, *n, "mono", implicit=True, dt=rng.choice([0.05, 0.1, 0.2]),
                         steps=max(2, min(40, int(8e7 / vox))), **sig)
        fp64 = vox < 300000 and rng.random() < 0.3
        return _case(geom, *n, "mono", fp64=fp64, steps=max(20, min(400, int(2e9 / vox) // (20 if fp64 else 1))),
                     **sig)
    lo, top = {"jacobi": (40, 170), "chebyshev": (48, 230), "sor": (40, 160), "torso": (40, 128),
               "batch": (48, 150)}[kind]
    m = _log(rng, lo, top)
    n = [max(24, int(m * rng.uniform(0.85, 1.0))) for _ in range(3)]
    geom = rng.choice(["shell", "biv"])
    if kind in ("chebyshev", "torso") and rng.random() < 0.7:
        sig["seT"] = siT * rng.uniform(1.2, 2.0)
    if kind == "jacobi":
        return _case(geom, *n, "bi", **sig)
    if kind == "chebyshev":
        return _case(geom, *n, "bi", solver="chebyshev", steps=rng.randint(1, 4), **sig)
    if kind == "sor":
        return _case(geom, *n, "bi", solver="sor", omega=rng.choice([0.0, 1.5, 1.8]), front=0.05, **sig)
    if kind == "torso":
        return _case(geom, *n, "bi", solver="chebyshev", torso=True, front=0.02, **sig)
    return _case("shell", m, m, m, "bi", solver=rng.choice(["chebyshev", "chebyshev", "jacobi"]),
                 members=rng.randint(2, 12), steps=1, **sig)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _grid(c):
    dims = (c["nz"], c["ny"], c["nx"])
    z, y, x = torch.meshgrid(*[torch.arange(n, device=DEV, dtype=torch.float32) + 0.5 - n / 2.0 for n in dims],
                             indexing="ij")
    return x, y, z


def _level(x, y, z, ax, ay, az):
    return torch.sqrt((x / ax) ** 2 + (y / ay) ** 2 + (z / az) ** 2)


def _shell(x, y, z, semi, wall):
    so = _level(x, y, z, *semi)
    si = _level(x, y, z, *[max(a - wall, 0.5) for a in semi])
    return (so <= 1.0) & (si > 1.0), ((1.0 - 1.0 / si.clamp(min=1e-6)) /
                                      (1.0 / so.clamp(min=1e-6) - 1.0 / si.clamp(min=1e-6))).nan_to_num(0.0).clamp(0, 1)


def _helix(x, y, z, depth):
    """Circumferential direction turned about the position vector from +60 to -60 degrees through the wall."""
    r = torch.stack([x, y, z], -1)
    r = r / r.norm(dim=-1, keepdim=True).clamp(min=1e-6)
    h = torch.sqrt(x * x + y * y).clamp(min=1e-6)
    circ = torch.stack([-y / h, x / h, torch.zeros_like(x)], -1)
    a = torch.deg2rad(60.0 - 120.0 * depth)[..., None]
    f = torch.cos(a) * circ + torch.sin(a) * torch.linalg.cross(r, circ)
    return f / f.norm(dim=-1, keepdim=True).clamp(min=1e-6)


def _geometry(c, gen):
    """Tissue mask (bool) and unit fibres, (nz, ny, nx) and (nz, ny, nx, 3)."""
    x, y, z = _grid(c)
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    if c["geom"] == "slab":   # all tissue, fibres in the x-y plane turning from -60 to +60 degrees through z
        th = torch.deg2rad(torch.linspace(-60.0, 60.0, nz, device=DEV))[:, None, None].expand(nz, ny, nx)
        f = torch.stack([torch.cos(th), torch.sin(th), torch.zeros_like(th)], -1)
        return torch.ones((nz, ny, nx), dtype=torch.bool, device=DEV), f
    sx, sy, sz = nx / 256.0, ny / 256.0, nz / 256.0
    if c["geom"] == "shell":   # closed ellipsoidal shell, wall 10 voxels on a 128^3 grid
        wall = max(2.0, 20.0 * min(sx, sy, sz))
        m, d = _shell(x, y, z, (80 * sx, 80 * sy, 110 * sz), wall)
        f = _helix(x, y, z, d)
    else:   # two truncated shells, the right ventricle outside the left
        s = min(sx, sy, sz)
        lv, ld = _shell(x, y + 20 * sy, z, (85 * sx, 85 * sy, 125 * sz), 32 * s)
        rv, rd = _shell(x, y - 30 * sy, z, (100 * sx, 75 * sy, 115 * sz), 18 * s)
        inside = _level(x, y + 20 * sy, z, 85 * sx, 85 * sy, 125 * sz) <= 1.0
        keep = z <= 85 * sz
        lv, rv = lv & keep, rv & ~inside & keep
        m = lv | rv
        f = torch.where(lv[..., None], _helix(x, y + 20 * sy, z, ld), _helix(x, y - 30 * sy, z, rd))
        f = f + torch.randn(f.shape, device=DEV, generator=gen) * math.tan(math.radians(2.5))
        f = f / f.norm(dim=-1, keepdim=True).clamp(min=1e-6)
    return m, f * m[..., None]


def _inputs(c, seed):
    """Everything a pass starts from, as tensors on the GPU."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    m, f = _geometry(c, gen)
    x, y, z = _grid(c)
    u = torch.rand(4, device=DEV, generator=gen).tolist()
    zs = torch.nonzero(m.any(dim=2).any(dim=1))[:, 0]
    z0 = float(z[zs[0], 0, 0]) + c["front"] * (0.8 + 0.4 * u[0]) * float(zs[-1] - zs[0])
    tilt = min(1.0, 2.0 * c["front"])
    d = z - z0 + tilt * ((0.4 * u[1] - 0.2) * x + (0.4 * u[2] - 0.2) * y)   # height above a tilted front
    w = 1.0 - (0.1 + 0.3 * u[3]) * (1.0 - torch.exp((d / 60.0).clamp(max=0.0)))
    plateau = 0.5 + 0.5 * torch.sqrt(1.0 - 4.0 * (0.3 / 6.0) / w)   # where the two currents balance
    v = 0.5 * (1.0 - torch.tanh(d / 1.5)) * plateau
    v = v * (1.0 + 0.002 * torch.rand(m.shape, device=DEV, generator=gen))
    g = c["siL"] / (c["siL"] + c["seL"])
    zero, one = torch.zeros_like(v), torch.ones_like(v)
    v, w = torch.where(m, v, zero), torch.where(m, w, one)
    ve = -g * v if c["model"] == "bi" and not c["torso"] else zero
    return m, f.to(torch.float32).contiguous(), v, w, ve


def _members(c, seed):
    """The single simulations of a case: itself, or the members of a batch, each with its own size and tensors."""
    if not c["members"]:
        return [(c, seed)]
    out = []
    for i in range(c["members"]):
        rng = np.random.default_rng([c["members"], c["nx"], i])
        n = int(round(48 + (c["nx"] - 48) * (i + 0.5) / c["members"])) if c["nx"] > 48 else c["nx"]
        siL, seL = rng.uniform(0.15, 0.25), rng.uniform(0.15, 0.25)
        k = dict(c, members=0, nx=n, ny=n, nz=n, siL=float(siL), siT=float(siL / rng.uniform(3.0, 5.0)),
                 seL=float(seL), seT=float(seL / rng.uniform(3.0, 5.0)))
        out.append((k, seed * 1000 + i))
    return out


class _Run:
    """A handle, its checkpoint and the host memory its states come back to."""

    def __init__(self, c, seed):
        m, f, v, w, ve = _inputs(c, seed)
        s = ep.Sim(c["nx"], c["ny"], c["nz"], c["dx"], ep.EP_BI if c["model"] == "bi" else ep.EP_MONO,
                   ep.EP_FP64 if c["fp64"] else ep.EP_FP32)
        s.set_mask(m.to(torch.uint8).cpu().numpy())
        s.set_fibres(f.cpu().numpy())
        s.set_params(_Params(c))
        s.add_stimulus((0, 0, 0), (4, 4, 4), 0.0, 1.0, 0.5)
        if c["torso"]:
            s.set_torso((~m).to(torch.uint8).cpu().numpy(), 1.0)
        s.set_state(*[a.double().cpu().numpy() for a in (v, w, ve)], 0)
        nb = s.state_bytes()
        self.start = torch.empty(nb, dtype=torch.uint8, pin_memory=True).numpy()
        self.end = torch.empty(nb, dtype=torch.uint8, pin_memory=True).numpy()
        s.read_state(self.start)
        self.sim, self.steps = s, c["steps"]
        self.type, self.head = (np.float64, 32) if c["fp64"] else (np.float32, 32)

    def restore(self):
        self.sim.write_state(self.start)

    def outputs(self):
        f = self.sim.read_state(self.end)[self.head:].view(self.type).reshape(4, -1)
        return {"v": f[0], "w": f[1], "ve": f[2], "tact": f[3]}


class _Batch:
    def __init__(self, c, seed):
        self.runs = [_Run(k, s) for k, s in _members(c, seed)]
        self.batch, self.steps = ep.Batch(len(self.runs)), c["steps"]
        for r in self.runs:
            self.batch.add(r.sim)


def prepare(case, seed):
    return _Batch(case, seed) if case["members"] else _Run(case, seed)


def run(state):
    if isinstance(state, _Run):
        state.restore()
        state.sim.step(state.steps)
        return state.outputs()
    for r in state.runs:
        r.restore()
    state.batch.step(state.steps)
    return [r.outputs() for r in state.runs]


# --------------------------------------------------------------------------
# work and reference
# --------------------------------------------------------------------------
def _fill(c):
    """Share of the box that is tissue."""
    return {"slab": 1.0, "shell": 0.095, "biv": 0.203}[c["geom"]]


def _sweeps(c):
    """Typical sweeps of one solve from these starts (the over-relaxed solve's are eight colour passes)."""
    n = max(c["nx"], c["ny"], c["nz"])
    if c["implicit"]:
        return 5 + 30 * c["dt"]
    if c["torso"]:
        return 40.0 * n
    return {"jacobi": 60.0 * n, "chebyshev": 250 + 2.0 * n, "sor": 8 * 5.0 * n}[c["solver"]]


def work(case):
    """A field read or written once is 4 (8) bytes a voxel, a voxel's fibre and diagonal 16; a sweep reads its
    iterate, right-hand side and record and writes the new iterate."""
    total = {"bytes": 0.0, "flops": 0.0}
    for c, _ in _members(case, 0):
        n, rb = c["nx"] * c["ny"] * c["nz"], 8 if c["fp64"] else 4
        tissue = n * _fill(c)
        domain = n if c["torso"] else tissue
        b = tissue * (4 * rb + 16) * c["steps"] + 7 * rb * n   # reaction and diffusion; the checkpoints
        fl = tissue * 130.0 * c["steps"]
        if c["model"] == "bi" or c["implicit"]:
            s = _sweeps(c) * c["steps"]
            b += domain * (3 * rb + 16) * s
            fl += domain * 110.0 * s
        total["bytes"] += b
        total["flops"] += fl
    return total


class _Operator:
    """The self-dual finite-volume operator in 64 bits: vertex gradients averaged over the valid voxel pairs,
    a vertex tensor that is the mean over the block, and the transpose of the gradient; pairs and tensors of
    the tissue, or with `torso` the isotropic term over tissue + torso."""

    def __init__(self, c, pairs, tissue, f, sT, dS, so=0.0):
        self.shape = tuple(pairs.shape)
        P = self._pad(pairs.double())
        self.pairs = [[(lo, hi, self._cut(P, lo) * self._cut(P, hi)) for lo, hi in self._axis(a)] for a in range(3)]
        self.r = []
        for a in range(3):
            n = sum(p[2] for p in self.pairs[a])
            self.r.append(torch.where(n > 0, 1.0 / n.clamp(min=1.0), torch.zeros_like(n)))
        corners = [(u, t, s) for u in (0, 1) for t in (0, 1) for s in (0, 1)]
        C = 1.0 / (8.0 * c["dx"] ** 2)
        T = self._pad(tissue.double())
        nT = sum(self._cut(T, o) for o in corners)
        self.S = [[None] * 3 for _ in range(3)]
        for i in range(3):
            for j in range(i, 3):
                s = torch.zeros_like(nT)
                if dS != 0.0:
                    ff = self._pad(f[..., i].double() * f[..., j].double() * tissue.double())
                    s = dS * sum(self._cut(ff, o) for o in corners)
                if i == j:
                    s = s + sT * nT
                if so and i == j:
                    s = so * (sum(self._cut(P, o) for o in corners) - nT)   # the block's torso voxels
                elif so:
                    s = torch.zeros_like(nT)
                self.S[i][j] = self.S[j][i] = C * s * self.r[i] * self.r[j]

    @staticmethod
    def _pad(a):
        return torch.nn.functional.pad(a, (1, 1, 1, 1, 1, 1))

    def _cut(self, a, o):
        nz, ny, nx = self.shape
        return a[o[0]:o[0] + nz + 1, o[1]:o[1] + ny + 1, o[2]:o[2] + nx + 1]

    @staticmethod
    def _axis(a):
        """The four voxel pairs of a vertex along axis a (0 = x), as (low corner, high corner)."""
        out = []
        for p in (0, 1):
            for q in (0, 1):
                lo, hi = [p, q], [p, q]
                lo.insert(2 - a, 0)
                hi.insert(2 - a, 1)
                out.append((tuple(lo), tuple(hi)))
        return out

    def __call__(self, u):
        U = self._pad(u)
        g = [sum(m * (self._cut(U, hi) - self._cut(U, lo)) for lo, hi, m in self.pairs[a]) for a in range(3)]
        out = torch.zeros_like(U)
        for a in range(3):
            F = self.S[a][0] * g[0] + self.S[a][1] * g[1] + self.S[a][2] * g[2]
            for lo, hi, m in self.pairs[a]:
                self._cut(out, hi).add_(m * F)
                self._cut(out, lo).sub_(m * F)
        return out[1:-1, 1:-1, 1:-1]

    def diagonal(self):
        out = torch.zeros([n + 2 for n in self.shape], dtype=torch.float64, device=DEV)
        for u in (0, 1):
            for t in (0, 1):
                for s in (0, 1):
                    c = []
                    for a in range(3):
                        k = torch.zeros_like(self.r[0])
                        for lo, hi, m in self.pairs[a]:
                            if hi == (u, t, s):
                                k = m
                            elif lo == (u, t, s):
                                k = -m
                        c.append(k)
                    self._cut(out, (u, t, s)).add_(sum(self.S[a][b] * c[a] * c[b] for a in range(3) for b in range(3)))
        return out[1:-1, 1:-1, 1:-1]


def _components(dom):
    """Takes the mean of every face-connected component off a field (zero off the domain)."""
    lab = torch.where(dom, torch.arange(1, dom.numel() + 1, device=DEV).reshape(dom.shape), 0)
    while True:
        new = lab.clone()
        for a in range(3):
            n = lab.shape[a]
            new.narrow(a, 0, n - 1).copy_(torch.maximum(new.narrow(a, 0, n - 1), lab.narrow(a, 1, n - 1)))
            new.narrow(a, 1, n - 1).copy_(torch.maximum(new.narrow(a, 1, n - 1), lab.narrow(a, 0, n - 1)))
        new = torch.where(dom, new, 0)
        if torch.equal(new, lab):
            break
        lab = new
    where = dom.reshape(-1).nonzero()[:, 0]
    names, inv = torch.unique(lab.reshape(-1)[where], return_inverse=True)
    parts = [where[inv == i] for i in range(len(names))] if len(names) <= 64 else None
    count = torch.bincount(inv).double()

    def centre(a):
        flat, out = a.reshape(-1), torch.zeros(a.numel(), dtype=torch.float64, device=DEV)
        if parts is not None:
            for p in parts:
                out[p] = flat[p] - flat[p].mean()
        else:
            out[where] = flat[where] - (torch.bincount(inv, flat[where]) / count)[inv]
        return out.reshape(a.shape)

    return centre


def _solve(apply, diag, b, x, centre, tol=1e-10):
    """Conjugate gradients in 64 bits, to well below what the library is asked for."""
    inv = torch.where(diag > 0, 1.0 / diag.clamp(min=1e-300), torch.zeros_like(diag))
    b = centre(b)
    x = x.clone()
    r = b - apply(x)
    z = centre(inv * r)
    p, rz, bb = z.clone(), (r * z).sum(), (b * b).sum()
    for it in range(20000):
        q = apply(p)
        a = rz / (p * q).sum()
        x += a * p
        r -= a * q
        if it % 20 == 19 and float((r * r).sum() / bb) <= tol * tol:
            break
        z = centre(inv * r)
        new = (r * z).sum()
        p = z + (new / rz) * p
        rz = new
    return centre(x)


def _exact_one(c, seed):
    m, f, v, w, ve = _inputs(c, seed)
    if c["fp64"]:
        v, w, ve = (a.double() for a in (v, w, ve))
    v, w, ve = v.double(), w.double(), ve.double()
    mono, dt = c["model"] == "mono", c["dt"]
    Li = _Operator(c, m, m, f, c["siT"], c["siL"] - c["siT"])
    a = dt * (0.5 if mono else 1.0)
    tact = torch.full_like(v, -1.0)
    stim = torch.zeros_like(v)
    stim[0:4, 0:4, 0:4] = 0.5
    equal = c["seL"] == c["siL"] and c["seT"] == c["siT"] and not c["torso"]
    dom = torch.ones_like(m) if c["torso"] else m
    centre = None if mono else _components(dom)
    if not mono and not equal:
        sT, sL = c["siT"] + c["seT"], c["siL"] + c["seL"]
        Lh = _Operator(c, m, m, f, sT, sL - sT)
        A, D = Lh, Lh.diagonal()
        if c["torso"]:
            Lo = _Operator(c, dom, m, f, 0.0, 0.0, so=1.0)
            A, D = (lambda u: Lh(u * m) * m + Lo(u)), D + Lo.diagonal()
    if c["implicit"]:
        Di = 1.0 + a * Li.diagonal()
    for n in range(c["steps"]):
        js = stim if n * dt < 1.0 else torch.zeros_like(stim)
        vs = v + dt * (v * v * (1 - v) * w / 0.3 - v / 6.0 + js)
        w1 = w + dt * torch.where(v < 0.13, (1 - w) / 120.0, -w / 150.0)
        if c["implicit"]:
            v1 = _solve(lambda u: u + a * Li(u), Di, vs * m, vs * m, lambda u: u)
        else:
            v1 = vs - a * Li((vs if mono else vs + ve) * m)
        v1, w = torch.where(m, v1, torch.zeros_like(v1)), torch.where(m, w1, torch.ones_like(w1))
        up = m & (v < 0.5) & (v1 >= 0.5) & (tact < 0)
        tact = torch.where(up, n * dt + dt * (0.5 - v) / (v1 - v), tact)
        v = v1
        if not mono and equal:   # proportional tensors: v_e = -v / 2 up to each component's constant
            ve = centre(-0.5 * v)
        elif not mono:
            ve = _solve(A, D, -Li(v) * m, ve * dom, centre)
    return {"v": v.reshape(-1), "w": w.reshape(-1), "ve": ve.reshape(-1), "tact": tact.reshape(-1)}


def exact(case, seed):
    """The state after the pass in 64 bits, its linear systems solved far below the library's tolerance.
    Left out where those solves take over about 20 seconds (unequal tensors on large grids)."""
    vox = case["nx"] * case["ny"] * case["nz"] * case["steps"]
    if case["model"] == "bi" and not case["members"] and vox > 2e7 and (
            case["torso"] or case["seL"] != case["siL"] or case["seT"] != case["siT"]):
        return None
    out = [_exact_one(c, s) for c, s in _members(case, seed)]
    return out if case["members"] else out[0]
