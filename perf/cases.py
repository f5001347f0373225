"""Performance cases of the multiblob library: what its users run, over the sizes they run it at.

Each case goes through the public entry points (`Multiblob`, `rollout_particle_velocities`) and
returns what the call produces whole: the stepped state (blob positions and fluid velocity), the
particle velocities with their gradients, or the grid or blob array of a standalone operator.

`exact` computes the same outputs in plain FP64 PyTorch from the definitions in include/mb.h
(Peskin kernel, MAC operators, Crank-Nicolson solve by FFT, harmonic bonds, soft repulsion,
Philox thermal stress); it shares no code with the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1407_5600_gb300 as mb
from paper_1407_5600_gb300 import workloads as wl
from paper_1407_5600_gb300.autograd import rollout_particle_velocities

DEV = "cuda"
RHO = ETA = 1.0
DT = 0.05


def _sim(name=None, *, nx, ny, nz, batch=1, h=1.0, precision=0, deterministic=0, advection=0,
         mean_mode=0, kT=0.0, integrator=0, place="suspension", a=2.2, particles=1, rep=0, ext=0.0,
         body=0.0, v_rms=0.0, steps=1):
    """A case that steps suspensions: `particles` icosahedra of vertex radius a (in units of h)
    per box, repulsion on or off, external forces and body force of the given sizes, an initial
    smooth solenoidal flow of rms v_rms, `steps` steps a call."""
    c = dict(kind="step", nx=nx, ny=ny, nz=nz, batch=batch, h=h, precision=precision,
             deterministic=deterministic, advection=advection, mean_mode=mean_mode, kT=kT,
             integrator=integrator, place=place, a=a, particles=particles, rep=rep, ext=ext,
             body=body, v_rms=v_rms, steps=steps)
    return dict(c, name=name) if name else c


def _op(kind, name=None, *, nx, ny, nz, h=1.0, precision=0, blobs=0, body=0.0, mean_mode=0):
    """A standalone operator on one box: spread, interp or fluid."""
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, batch=1, h=h, precision=precision, blobs=blobs,
             body=body, mean_mode=mean_mode)
    return dict(c, name=name) if name else c


def _rollout(name=None, *, n, particles, a, K, checkpoint, ext=1e-3, rep=0):
    """A differentiable run: K steps and the gradient of the particle velocities."""
    c = dict(kind="rollout", nx=n, ny=n, nz=n, batch=1, h=1.0, precision=1, place="suspension",
             a=a, particles=particles, rep=rep, ext=ext, body=0.0, v_rms=0.0, K=K,
             checkpoint=checkpoint)
    return dict(c, name=name) if name else c


def _count(phi, a, cells):
    return int(round(phi * cells / (4.0 / 3.0 * math.pi * a ** 3)))


def listed():
    return [
        # the smallest: one particle dragged through a small box in the plain FP64, deterministic
        # method (the Stokeslet / Hasimoto drag run); launches and latency
        _sim("drag_32_fp64", nx=32, ny=32, nz=32, precision=1, deterministic=1, mean_mode=1,
             place="single", a=1.0, ext=1e-3, steps=20),
        # the lubrication curve: 32 independent boxes of two particles in one context
        _sim("gap_sweep_32x64", nx=64, ny=64, nz=64, batch=32, place="gap", a=1.6, particles=2,
             ext=1e-3, steps=10),
        # the dense suspension of the viscosity protocol, the benchmark's workload, on the FP32
        # grid and in FP64
        _sim("dense_128", nx=128, ny=128, nz=128, a=2.2, particles=_count(0.40, 2.2, 128 ** 3),
             rep=1, body=1e-4, v_rms=0.02, steps=10),
        _sim("dense_128_fp64", nx=128, ny=128, nz=128, precision=1, a=2.2,
             particles=_count(0.40, 2.2, 128 ** 3), rep=1, body=1e-4, v_rms=0.02, steps=2),
        # the differentiable run: K = 50 steps of 64 particles, checkpoints every 10, gradients
        # with respect to every blob coordinate and the spring stiffness
        _rollout("rollout_64", n=64, particles=64, a=2.0, K=50, checkpoint=10),
        # the large fluctuating suspension (sides above 128: one FFT pass per axis)
        _sim("thermal_256", nx=256, ny=256, nz=256, a=3.2, particles=_count(0.30, 3.2, 256 ** 3),
             rep=1, kT=1e-3, v_rms=0.02, steps=2),
        # the steady-Stokes integrator of the viscosity runs: the dense suspension, and a dilute
        # one in FP64
        _sim("stokes_128", nx=128, ny=128, nz=128, mean_mode=1, integrator=1, a=2.2,
             particles=_count(0.40, 2.2, 128 ** 3), rep=1, body=1e-4, steps=4),
        _sim("stokes_64_fp64", nx=64, ny=64, nz=64, precision=1, mean_mode=1, integrator=1,
             a=2.2, particles=_count(0.05, 2.2, 64 ** 3), rep=1, body=1e-3, steps=4),
        # every fluid term at once in a box of three different sides: thermal and convective
        # stress, an odd number of particles, external forces
        _sim("convective_64x128x32", nx=64, ny=128, nz=32, a=2.2, particles=331, rep=1, ext=1e-3,
             kT=1e-3, advection=1, v_rms=0.05, steps=5),
        # the operators on their own, for programs that assemble their own scheme
        _op("spread", "spread_128", nx=128, ny=128, nz=128, blobs=99991),
        _op("interp", "interp_256x64x32_fp64", nx=256, ny=64, nz=32, precision=1, blobs=50021),
        _op("fluid", "fluid_256x64x64_fp64", nx=256, ny=64, nz=64, precision=1, body=1e-3),
    ]


def draw(rng):
    kind = rng.choice(["step"] * 5 + ["stokes"] * 2 + ["rollout", "spread", "interp", "fluid"])

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def sides(low, high, most):
        # powers of two whose product stays within `most` cells
        while True:
            n = [2 ** rng.randint(low, high) for _ in range(3)]
            if rng.random() < 0.4:
                n = [n[0]] * 3
            if n[0] * n[1] * n[2] <= most:
                return dict(nx=n[0], ny=n[1], nz=n[2])

    def vol(s):
        return s["nx"] * s["ny"] * s["nz"]

    h = rng.choice([1.0, 1.0, 0.7])
    precision = rng.randint(0, 1)
    if kind == "rollout":
        n = rng.choice([16, 32, 64])
        a = round(rng.uniform(1.0, 2.2), 2)
        most = max(1, _count(0.05, a, n ** 3))
        return _rollout(n=n, particles=log_int(1, most), a=a, K=rng.randint(2, 30),
                        checkpoint=rng.choice([3, 5, 10]), rep=rng.randint(0, 1))
    if kind in ("spread", "interp", "fluid"):
        s = sides(3, 8, 2 ** 21)
        return _op(kind, h=h, precision=precision,
                   blobs=log_int(1, 200000) if kind != "fluid" else 0,
                   body=rng.choice([0.0, 1e-3]) if kind == "fluid" else 0.0,
                   mean_mode=rng.randint(0, 1), **s)
    s = sides(4, 8, 2 ** 21)
    batch = log_int(1, max(1, min(64, 2 ** 22 // vol(s)))) if rng.random() < 0.3 else 1
    lmin = min(s["nx"], s["ny"], s["nz"])
    a = round(rng.uniform(1.0, min(3.2, lmin / 5.0)), 2)
    dense = rng.random() < 0.4
    particles = max(1, int(_count(rng.uniform(0.2, 0.4) if dense else
                                  math.exp(rng.uniform(math.log(0.002), math.log(0.2))), a, vol(s))))
    particles = min(particles, max(1, 18808 // batch))
    c = dict(s, batch=batch, h=h, precision=precision, a=a, particles=particles,
             rep=1 if particles > 8 else 0, ext=rng.choice([0.0, 1e-3]),
             body=rng.choice([0.0, 1e-3]), steps=rng.randint(1, 8))
    if kind == "stokes":
        if not c["ext"]:               # something drives the flow
            c["body"] = 1e-3
        return _sim(integrator=1, mean_mode=1, **c)
    driven = c["ext"] or c["body"]
    return _sim(mean_mode=rng.randint(0, 1), kT=rng.choice([0.0, 0.0, 1e-3]),
                advection=1 if rng.random() < 0.2 else 0,
                deterministic=1 if precision and rng.random() < 0.3 else 0,
                v_rms=rng.choice([0.0, 0.02, 0.05] if driven else [0.02, 0.05]), **c)


# ---------------------------------------------------------------------------------------------
# Inputs.

def _centres(case, rng):
    """Non-overlapping centres: a face-centred lattice of the box with random vacancies, each
    particle displaced by less than half its free space (units of h)."""
    L = np.array([case["nx"], case["ny"], case["nz"]], dtype=np.float64)
    n, a = case["particles"], case["a"]
    if case["place"] == "single":
        return rng.uniform(0.0, 1.0, size=(1, 3)) * L
    tight = 2.0 * a * math.sqrt(2.0)
    n = min(n, 4 * int(np.prod(np.maximum(1, np.floor(L / tight)))))
    c = (4.0 * float(np.prod(L)) / n) ** (1.0 / 3.0)
    m = np.maximum(1, np.floor(L / c))
    while 4 * np.prod(m) < n:
        c *= 0.98
        m = np.maximum(1, np.floor(L / c))
    m = m.astype(int)
    base = np.array([[0, 0, 0], [0.5, 0.5, 0], [0.5, 0, 0.5], [0, 0.5, 0.5]])
    ijk = np.stack(np.meshgrid(*[np.arange(k) for k in m], indexing="ij"), -1)
    sites = ((ijk.reshape(-1, 1, 3) + base[None]).reshape(-1, 3) + 0.25) * (L / m)
    keep = np.sort(rng.permutation(len(sites))[:n])
    cell = np.sort(L / m)
    free = 0.5 * math.hypot(cell[0], cell[1]) - 2.0 * a
    d = rng.normal(size=(n, 3))
    d *= (0.5 * max(0.0, free) * rng.uniform(size=(n, 1)) ** (1 / 3)) / np.linalg.norm(d, axis=1, keepdims=True)
    return sites[keep] + d


def _rotations(n, rng):
    q = rng.normal(size=(n, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    return np.stack([
        1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
        2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
        2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], -1).reshape(n, 3, 3)


def _box(case, b, seed):
    """Blobs of box b: 13-blob icosahedra at rest shape, random orientations."""
    rng = np.random.default_rng([seed, b])
    h = case["h"]
    L = np.array([case["nx"], case["ny"], case["nz"]], dtype=np.float64) * h
    tpl, tb, tr = wl.icosahedron_template(case["a"] * h)
    if case["place"] == "gap":       # surface gaps log-spaced from 0.05h to 4h over the boxes
        gap = 0.05 * 80.0 ** (b / max(case["batch"] - 1, 1)) * h
        sep = np.array([2 * case["a"] * h + gap, 0.0, 0.0])
        off = rng.uniform(-0.5, 0.5, size=3) * h
        centres = np.array([L / 2 + off - sep / 2, L / 2 + off + sep / 2])
    else:
        centres = _centres(case, rng) * h
    n = len(centres)
    pos = centres[:, None, :] + np.einsum("bk,pjk->pbj", tpl, _rotations(n, rng))
    pos = np.mod(pos.reshape(-1, 3), L)
    pos[pos >= L] = 0.0
    pid = np.repeat(np.arange(n, dtype=np.int32), 13)
    bonds = (tb[None] + 13 * np.arange(n, dtype=np.int32)[:, None, None]).reshape(-1, 2)
    ext = None
    if case["ext"]:
        if case["place"] == "single":
            ext = np.zeros_like(pos)
            ext[:, 0] = case["ext"] / 13.0
        elif case["place"] == "gap":
            ext = np.zeros_like(pos)
            ext[:13, 0], ext[13:, 0] = case["ext"] / 13.0, -case["ext"] / 13.0
        else:
            ext = rng.normal(scale=case["ext"], size=pos.shape)
    return dict(pos=pos, pid=pid, bonds=bonds.astype(np.int32), rest=np.tile(tr, n), n=n, ext=ext)


def _shape(case):
    return (case["nz"], case["ny"], case["nx"])


def _grid_dtype(case):
    return torch.float64 if case["precision"] == 1 else torch.float32


def _flow(case, seed):
    """[batch, 3, nz, ny, nx] smooth flow, discretely divergence-free (a MAC curl), rms v_rms."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    nz, ny, nx = _shape(case)
    v = torch.empty((case["batch"], 3, nz, ny, nx), dtype=_grid_dtype(case), device=DEV)
    kz, ky, kx = (torch.fft.fftfreq(n, device=DEV, dtype=torch.float64) for n in (nz, ny, nx))
    k2 = kz[:, None, None] ** 2 + ky[None, :, None] ** 2 + kx[None, None, : nx // 2 + 1] ** 2
    smooth = torch.exp(-k2 * (4.0 * math.pi) ** 2 / 2)
    for b in range(case["batch"]):
        A = torch.randn((3, nz, ny, nx), generator=g, device=DEV, dtype=torch.float64)
        A = torch.fft.irfftn(torch.fft.rfftn(A, dim=(1, 2, 3)) * smooth, s=(nz, ny, nx), dim=(1, 2, 3))

        def up(x, d):
            return torch.roll(x, -1, d) - x

        u = torch.stack([up(A[2], 1) - up(A[1], 0), up(A[0], 0) - up(A[2], 2), up(A[1], 2) - up(A[0], 1)])
        v[b] = (u * (case["v_rms"] / u.square().mean().sqrt())).to(v.dtype)
    return v


def _body(case):
    return (case["body"], 0, 2, 1) if case["body"] else None


def _springs(case):
    h = case["h"]
    return 100.0 * h, (100.0 * h if case["rep"] else 0.0), (h if case["rep"] else 0.0)


def _op_inputs(case, seed):
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    shape = (3,) + _shape(case)
    out = {}
    if case["kind"] in ("spread", "interp"):
        L = torch.tensor([case["nx"], case["ny"], case["nz"]], dtype=torch.float64, device=DEV) * case["h"]
        out["pos"] = torch.rand((case["blobs"], 3), generator=g, device=DEV, dtype=torch.float64) * L
    if case["kind"] == "spread":
        out["F"] = torch.randn((case["blobs"], 3), generator=g, device=DEV, dtype=torch.float64)
    else:
        out["v"] = torch.randn(shape, generator=g, device=DEV, dtype=torch.float64).to(_grid_dtype(case))
    if case["kind"] == "fluid":
        out["f"] = (0.1 * torch.randn(shape, generator=g, device=DEV, dtype=torch.float64)).to(_grid_dtype(case))
    return out


# ---------------------------------------------------------------------------------------------
# The calls.

def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        keys = ("nx", "ny", "nz", "batch", "h", "precision", "deterministic", "advection",
                "mean_mode", "kT", "integrator")
        desc = mb.GridDesc(rho=RHO, eta=ETA, dt=DT, seed=int(seed), **{k: case[k] for k in keys})
        sim = mb.Multiblob(desc)
        boxes = [_box(case, b, seed) for b in range(case["batch"])]
        for b, x in enumerate(boxes):
            sim.set_particles(b, x["pos"], x["pid"], x["bonds"], x["rest"], *_springs(case))
        if case["v_rms"]:
            sim.set_velocity_field(_flow(case, seed))
        ext = None
        if case["ext"]:
            ext = torch.as_tensor(np.concatenate([x["ext"] for x in boxes]), device=DEV)
        return dict(kind=kind, sim=sim, ext=ext, body=_body(case), steps=case["steps"])
    if kind == "rollout":
        sim = mb.Multiblob(mb.GridDesc(case["nx"], case["ny"], case["nz"], rho=RHO, eta=ETA, dt=DT,
                                       precision=1))
        x = _box(case, 0, seed)
        return dict(kind=kind, sim=sim, K=case["K"], checkpoint=case["checkpoint"], x=x,
                    springs=_springs(case), ext=torch.as_tensor(x["ext"], device=DEV),
                    q=torch.as_tensor(x["pos"], device=DEV).requires_grad_(),
                    k=torch.tensor(_springs(case)[0], dtype=torch.float64, device=DEV, requires_grad=True),
                    gU=torch.as_tensor(_cotangent(x, seed), device=DEV))
    sim = mb.Multiblob(mb.GridDesc(case["nx"], case["ny"], case["nz"], h=case["h"], rho=RHO, eta=ETA,
                                   dt=DT, precision=case["precision"], mean_mode=case["mean_mode"]))
    return dict(kind=kind, sim=sim, body=_body(case), **_op_inputs(case, seed))


def _cotangent(x, seed):
    return np.random.default_rng([seed, 1 << 20]).normal(size=(x["n"], 3))


def run(s):
    sim, kind = s["sim"], s["kind"]
    if kind == "step":
        sim.step(s["steps"], ext_blob_force=s["ext"], body_force=s["body"])
        return {"q": sim.blob_positions(), "v": sim.velocity_field()}
    if kind == "rollout":
        x = s["x"]
        U = rollout_particle_velocities(sim, s["q"], s["k"], x["pid"], x["bonds"], x["rest"], s["K"],
                                        s["checkpoint"], ext_blob_force=s["ext"], k_rep=s["springs"][1],
                                        r_cut=s["springs"][2])
        gq, gk = torch.autograd.grad(U, (s["q"], s["k"]), grad_outputs=s["gU"])
        return {"U": U.detach(), "grad_q": gq, "grad_k": gk}
    if kind == "spread":
        return sim.spread(s["pos"], s["F"])
    if kind == "interp":
        return sim.interp(s["pos"], s["v"])
    return sim.fluid_update(s["v"], s["f"], body_force=s["body"])


# ---------------------------------------------------------------------------------------------
# What a pass cannot do without.

def work(case):
    N = case["nx"] * case["ny"] * case["nz"] * case["batch"]
    box = case["nx"] * case["ny"] * case["nz"]
    real = 8 if case["precision"] == 1 else 4
    field = 3 * real * N
    fft = 2.5 * 3 * N * math.log2(box)              # one real transform of three components
    solve = 2 * fft + 3 * N * (14 + 24)             # there and back, stencil, divide, projection
    gather = 81 * 2 + 100                           # 27 nodes x 3 components, the weights
    if case["kind"] == "fluid":
        return {"bytes": 3 * field, "flops": solve}
    if case["kind"] in ("spread", "interp"):
        return {"bytes": field + 48 * case["blobs"], "flops": gather * case["blobs"]}
    nb = 13 * _blob_particles(case) * case["batch"]
    blobs = nb * (3 * gather + 42 / 13 * 40 + (100 if case["rep"] else 0))
    if case["kind"] == "rollout":
        # forward: field and positions read and written; backward: the same with the gradients
        return {"bytes": case["K"] * 3 * (2 * field + 48 * nb), "flops": case["K"] * 3 * (solve + blobs)}
    rounds = 2 if case["integrator"] == 1 else 1
    noise = (9 * N * 40 if case["kT"] else 0) + (9 * N * 6 if case["advection"] else 0)
    per = {"bytes": 2 * field + 48 * nb + (24 * nb if case["ext"] else 0),
           "flops": rounds * (solve + blobs) + noise}
    return {k: case["steps"] * x for k, x in per.items()}


def _blob_particles(case):
    L = np.array([case["nx"], case["ny"], case["nz"]], dtype=np.float64)
    tight = 2.0 * case["a"] * math.sqrt(2.0)
    if case["place"] == "suspension":
        return min(case["particles"], 4 * int(np.prod(np.maximum(1, np.floor(L / tight)))))
    return case["particles"]


# ---------------------------------------------------------------------------------------------
# The same outputs in FP64 from the definitions.

class _Exact:
    """One box: operators on [3, nz, ny, nx] fields and [n, 3] blobs in FP64."""

    def __init__(self, case):
        self.n = (case["nx"], case["ny"], case["nz"])
        self.shape, self.h = _shape(case), case["h"]
        self.L = torch.tensor(self.n, dtype=torch.float64, device=DEV) * self.h
        self.N = self.n[0] * self.n[1] * self.n[2]
        th = [2 * math.pi * torch.arange(n, dtype=torch.float64, device=DEV) / n for n in self.n]
        th[0] = th[0][: self.n[0] // 2 + 1]
        view = ((1, 1, -1), (1, -1, 1), (-1, 1, 1))
        self.D = [((torch.exp(1j * t) - 1) / self.h).view(w) for t, w in zip(th, view)]
        self.lam = sum((4 / self.h ** 2 * torch.sin(t / 2) ** 2).view(w) for t, w in zip(th, view))

    def weights(self, q, a):
        """Node indices [n, 27] and weights [n, 27] of component a."""
        idx, w = [], []
        for d in range(3):
            x = q[:, d] / self.h - (0.0 if d == a else 0.5)
            i0 = torch.floor(x.detach() + 0.5)
            t = x - i0
            s = torch.sqrt(1 - 3 * t * t)
            w.append(torch.stack([(2 - 3 * t - s) / 6, (1 + s) / 3, (2 + 3 * t - s) / 6], 1))
            i = i0.long()[:, None] + torch.arange(-1, 2, device=DEV)
            idx.append(torch.remainder(i, self.n[d]))
        nx, ny, _ = self.n
        at = (idx[2][:, :, None, None] * ny + idx[1][:, None, :, None]) * nx + idx[0][:, None, None, :]
        ww = w[2][:, :, None, None] * w[1][:, None, :, None] * w[0][:, None, None, :]
        return at.reshape(len(q), 27), ww.reshape(len(q), 27)

    def interp(self, q, v):
        u = []
        for a in range(3):
            at, w = self.weights(q, a)
            u.append((v[a].reshape(-1)[at] * w).sum(1))
        return torch.stack(u, 1)

    def spread(self, q, F):
        f = []
        for a in range(3):
            at, w = self.weights(q, a)
            c = (w * F[:, a : a + 1]).reshape(-1) / self.h ** 3
            f.append(torch.zeros(self.N, dtype=torch.float64, device=DEV).index_add(0, at.reshape(-1), c))
        return torch.stack(f).view((3,) + self.shape)

    def project(self, W):
        dw = sum(d * w for d, w in zip(self.D, W))
        lam = self.lam.clone()
        lam[0, 0, 0] = 1.0
        # G = -conj(D); D.G = -lambda, so P W = W + G (D.W) / lambda
        return torch.stack([w - torch.conj(d) * dw / lam for d, w in zip(self.D, W)])

    def body(self, body):
        f = torch.zeros((3,) + self.shape, dtype=torch.float64, device=DEV)
        if body:
            f0, axis, d, j = body
            x = torch.arange(self.n[d], dtype=torch.float64, device=DEV) + (0.0 if axis == d else 0.5)
            view = ((1, 1, -1), (1, -1, 1), (-1, 1, 1))[d]
            f[axis] += f0 * torch.sin(2 * math.pi * j * x / self.n[d]).view(view)
        return f

    def solve(self, v, f, mean=None):
        """Crank-Nicolson update of v with force density f; k = 0 from `mean` (None: from the grid)."""
        V, Fh = (torch.fft.rfftn(x, dim=(1, 2, 3)) for x in (v, f))
        W = ((RHO / DT - 0.5 * ETA * self.lam) * V + Fh) / (RHO / DT + 0.5 * ETA * self.lam)
        return self.back(W, W[:, 0, 0, 0] if mean is None else mean * self.N)

    def back(self, W, zero):
        P = self.project(W)
        keep = torch.ones_like(self.lam)
        keep[0, 0, 0] = 0.0
        at0 = torch.zeros_like(self.lam)
        at0[0, 0, 0] = 1.0
        P = P * keep + at0 * zero.to(P.dtype)[:, None, None, None]
        return torch.fft.irfftn(P, s=self.shape, dim=(1, 2, 3))

    def stokes(self, f):
        lam = self.lam.clone()
        lam[0, 0, 0] = 1.0
        W = torch.fft.rfftn(f, dim=(1, 2, 3)) / (ETA * lam)
        return self.back(W, torch.zeros(3, dtype=torch.float64, device=DEV))

    def image(self, d):
        return d - self.L * torch.round(d.detach() / self.L)

    def forces(self, q, x, k, k_rep, r_cut, ext):
        F = torch.zeros_like(q) if ext is None else ext.clone()
        i, j = x["i"], x["j"]
        r = self.image(q[i] - q[j])
        length = r.norm(dim=1, keepdim=True)
        f = -k * (length - x["r0"][:, None]) * r / length
        F = F.index_add(0, i, f).index_add(0, j, -f)
        if k_rep and r_cut:
            b, c = self.pairs(q.detach(), x["pid"], r_cut)
            if len(b):
                r = self.image(q[b] - q[c])
                length = r.norm(dim=1, keepdim=True)
                F = F.index_add(0, b, k_rep * (r_cut - length) * r / length)
        return F

    def pairs(self, q, pid, r_cut):
        """Ordered pairs (b, c) of blobs of different particles closer than r_cut."""
        m = [max(1, int(math.floor(float(self.L[d]) / r_cut))) for d in range(3)]
        m = [k if k >= 3 else 1 for k in m]
        cell = [torch.clamp((torch.remainder(q[:, d], self.L[d]) / self.L[d] * m[d]).long(), 0, m[d] - 1)
                for d in range(3)]
        cid = (cell[2] * m[1] + cell[1]) * m[0] + cell[0]
        order = torch.argsort(cid)
        cnt = torch.bincount(cid, minlength=m[0] * m[1] * m[2])
        start = torch.cumsum(cnt, 0) - cnt
        got = []
        me = torch.arange(len(q), device=DEV)
        reach = [(-1, 0, 1) if k > 1 else (0,) for k in m]
        for dz in reach[2]:
            for dy in reach[1]:
                for dx in reach[0]:
                    nb = [torch.remainder(c + d, k) for c, d, k in zip(cell, (dx, dy, dz), m)]
                    cc = (nb[2] * m[1] + nb[1]) * m[0] + nb[0]
                    for t in range(int(cnt.max())):
                        has = t < cnt[cc]
                        b = me[has]
                        c = order[start[cc[has]] + t]
                        r = self.image(q[b] - q[c])
                        near = (pid[b] != pid[c]) & (r.square().sum(1) < r_cut ** 2)
                        got.append((b[near], c[near]))
        return torch.cat([g[0] for g in got]), torch.cat([g[1] for g in got])

    def stress_force(self, T):
        """-D.T of stresses [3][3] at centres (T_aa) and edges (T_ab at integer a, b coordinates)."""
        ax = (2, 1, 0)
        f = []
        for a in range(3):
            s = 0
            for b in range(3):
                t = T[a][b]
                s = s + (t - torch.roll(t, 1, ax[b]) if a == b else torch.roll(t, -1, ax[b]) - t)
            f.append(-s / self.h)
        return torch.stack(f)

    def convective(self, v):
        ax = (2, 1, 0)

        def mean(x, d, s):
            return 0.5 * (x + torch.roll(x, s, ax[d]))

        return [[RHO * (mean(v[a], a, -1) ** 2 if a == b else mean(v[a], b, 1) * mean(v[b], a, 1))
                 for b in range(3)] for a in range(3)]

    def thermal(self, kT, seed, step, box):
        amp = math.sqrt(2 * ETA * kT / (self.h ** 3 * DT))
        G = torch.arange(self.N // 4, dtype=torch.int64, device=DEV)
        z = torch.empty((self.N // 4, 36), dtype=torch.float64, device=DEV)
        for j in range(5):
            words = _philox(G, step, box, j, seed)
            for i in range(4):
                p = 4 * j + i
                if p < 18:
                    u1 = ((words[i] & 0xFFFFFFFF).double() + 0.5) / 2.0 ** 32
                    u2 = (_shr(words[i], 32).double() + 0.5) / 2.0 ** 32
                    r = torch.sqrt(-2 * torch.log(u1))
                    z[:, 2 * p], z[:, 2 * p + 1] = r * torch.cos(2 * math.pi * u2), r * torch.sin(2 * math.pi * u2)
        W = (amp * z).view(self.N // 4, 4, 9).permute(2, 0, 1).reshape(9, *self.shape)
        return [[W[3 * a + b] for b in range(3)] for a in range(3)]


def _shr(x, n):
    return (x >> n) & ((1 << (64 - n)) - 1)


def _signed(x):
    x &= (1 << 64) - 1
    return x - (1 << 64) if x >= 1 << 63 else x


def _mulhi(x, m):
    """High 64 bits of the unsigned product of x (int64 bits) and the constant m."""
    x0, x1, m0, m1 = x & 0xFFFFFFFF, _shr(x, 32), m & 0xFFFFFFFF, m >> 32
    w1 = x1 * m0 + _shr(x0 * m0, 32)
    w2 = x0 * m1 + (w1 & 0xFFFFFFFF)
    return x1 * m1 + _shr(w1, 32) + _shr(w2, 32)


def _philox(c0, c1, c2, c3, seed):
    """Philox4x64-10 with key (seed, 0), 64-bit words held as int64 bits."""
    M0, M1 = 0xD2E7470EE14C6C93, 0xCA5A826395121157
    W0, W1 = 0x9E3779B97F4A7C15, 0xBB67AE8584CAA73B
    c = [c0, torch.full_like(c0, c1), torch.full_like(c0, c2), torch.full_like(c0, c3)]
    k0, k1 = seed, 0
    for _ in range(10):
        lo0, lo1 = c[0] * _signed(M0), c[2] * _signed(M1)
        c = [_mulhi(c[2], M1) ^ c[1] ^ _signed(k0), lo1, _mulhi(c[0], M0) ^ c[3] ^ _signed(k1), lo0]
        k0, k1 = k0 + W0, k1 + W1
    return c


def _blobs(x):
    bonds = torch.as_tensor(x["bonds"], device=DEV).long()
    return dict(i=bonds[:, 0], j=bonds[:, 1], r0=torch.as_tensor(x["rest"], device=DEV),
                pid=torch.as_tensor(x["pid"], device=DEV),
                ext=None if x["ext"] is None else torch.as_tensor(x["ext"], device=DEV))


def _exact_step(case, seed):
    E = _Exact(case)
    k, k_rep, r_cut = _springs(case)
    flow = _flow(case, seed).double() if case["v_rms"] else None
    q_out, v_out = [], []
    fb = E.body(_body(case))
    for b in range(case["batch"]):
        x = _box(case, b, seed)
        y, q = _blobs(x), torch.as_tensor(x["pos"], device=DEV)
        v = flow[b] if flow is not None else torch.zeros((3,) + E.shape, dtype=torch.float64, device=DEV)
        mean = v.mean(dim=(1, 2, 3)) * (1.0 if case["mean_mode"] == 0 else 0.0)
        for n in range(case["steps"]):
            if case["integrator"] == 1:
                v = E.stokes(E.spread(q, E.forces(q, y, k, k_rep, r_cut, y["ext"])) + fb)
                qh = q + 0.5 * DT * E.interp(q, v)
                v = E.stokes(E.spread(qh, E.forces(qh, y, k, k_rep, r_cut, y["ext"])) + fb)
                q = torch.remainder(q + DT * E.interp(qh, v), E.L)
                continue
            qh = torch.remainder(q + 0.5 * DT * E.interp(q, v), E.L)
            F = E.forces(qh, y, k, k_rep, r_cut, y["ext"])
            f = E.spread(qh, F) + fb
            if case["kT"]:
                f = f + E.stress_force(E.thermal(case["kT"], int(seed), n, b))
            if case["advection"]:
                f = f + E.stress_force(E.convective(v))
            if case["mean_mode"] == 0:
                mean = mean + DT / (RHO * E.N * E.h ** 3) * F.sum(0)
            v1 = E.solve(v, f, mean)
            q = torch.remainder(q + 0.5 * DT * E.interp(qh, v + v1), E.L)
            v = v1
        q_out.append(q)
        v_out.append(v)
    return {"q": torch.cat(q_out), "v": torch.stack(v_out)}


def _exact_rollout(case, seed):
    E = _Exact(case)
    x = _box(case, 0, seed)
    y = _blobs(x)
    k, k_rep, r_cut = _springs(case)
    q0 = torch.as_tensor(x["pos"], device=DEV).requires_grad_()
    k0 = torch.tensor(k, dtype=torch.float64, device=DEV, requires_grad=True)

    def step(q, v, mean, k):
        qh = q + 0.5 * DT * E.interp(q, v)
        F = E.forces(qh, y, k, k_rep, r_cut, y["ext"])
        mean = mean + DT / (RHO * E.N * E.h ** 3) * F.sum(0)
        v1 = E.solve(v, E.spread(qh, F), mean)
        return q + 0.5 * DT * E.interp(qh, v + v1), v1, mean

    # one state per step kept, each step differentiated on its own from the last to the first
    v = torch.zeros((3,) + E.shape, dtype=torch.float64, device=DEV)
    states = [(q0.detach(), v, torch.zeros(3, dtype=torch.float64, device=DEV))]
    with torch.no_grad():
        for _ in range(case["K"]):
            states.append(step(*states[-1], k0))
    pid = y["pid"].long()
    share = torch.zeros((x["n"], 1), dtype=torch.float64, device=DEV).index_add(
        0, pid, torch.ones((len(pid), 1), dtype=torch.float64, device=DEV))

    def U0(q, v):
        return torch.zeros((x["n"], 3), dtype=torch.float64, device=DEV).index_add(0, pid, E.interp(q, v)) / share

    q, v = (t.clone().requires_grad_() for t in states[-1][:2])
    U = U0(q, v)
    gU = torch.as_tensor(_cotangent(x, seed), device=DEV)
    gq, gv = torch.autograd.grad(U, (q, v), grad_outputs=gU)
    gk, gm = torch.zeros_like(k0), torch.zeros(3, dtype=torch.float64, device=DEV)
    for n in reversed(range(case["K"])):
        q, v, m = (t.clone().requires_grad_() for t in states[n])
        out = step(q, v, m, k0)
        gq, gv, gm, dk = torch.autograd.grad(out, (q, v, m, k0), grad_outputs=(gq, gv, gm),
                                             allow_unused=True)
        gm = torch.zeros(3, dtype=torch.float64, device=DEV) if gm is None else gm
        gk = gk + dk
    return {"U": U.detach(), "grad_q": gq, "grad_k": gk}


def exact(case, seed):
    if case["kind"] == "step" and case["rep"] and case["batch"] * case["steps"] * (1 + case["integrator"]) > 300:
        return None                    # the pair search box by box would take too long
    with torch.set_grad_enabled(case["kind"] == "rollout"):
        if case["kind"] == "step":
            return _exact_step(case, seed)
        if case["kind"] == "rollout":
            return _exact_rollout(case, seed)
        E, x = _Exact(case), _op_inputs(case, seed)
        if case["kind"] == "spread":
            return E.spread(x["pos"], x["F"])[None]
        if case["kind"] == "interp":
            return E.interp(x["pos"], x["v"].double())
        mean = None if case["mean_mode"] == 0 else torch.zeros(3, dtype=torch.float64, device=DEV)
        return E.solve(x["v"].double(), x["f"].double() + E.body(_body(case)), mean)[None]
