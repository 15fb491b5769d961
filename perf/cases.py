"""What a user of this package has it do, as timed cases.

A case is one call sequence of a program that holds an mDPD system: advance a
run and take a frame, evaluate forces for a host program, couple through host
buffers, differentiate an evaluation or a window.  `prepare` makes what such a
program has in hand (positions, velocities, a handle, cotangents), `run` is one
pass through the public entry points, `exact` is the same result in 64 bits
from a plain torch restatement of the method that shares no code with the
package.

Frames of a run with FP32 pair arithmetic are returned as float32 (that is
what such a run determines, and what trajectory files hold); those of a run
with FP64 pair arithmetic as float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1903_10134_gb300 import adjoint as AD
from paper_1903_10134_gb300 import inputs as I
from paper_1903_10134_gb300 import mdpd as M

DEV = "cuda"
RC, RD, DT, KT = 1.0, 0.75, 0.01, 1.0


def listed():
    return [
        # Equation-of-state box (Fig. 3b): 6,000 particles in 10^3, FP64 throughout.
        # The smallest system anybody runs: launches and latency.
        _case("bulk_fp64", kind="step", shape="bulk", lx=10.0, ly=10.0, lz=10.0, n=6000,
              precision=0, steps=50),
        # The liquid-vapour slab of Sec. 4.1 at the benchmark's size, a frame every 20 steps.
        _case("slab", kind="step", shape="slab", lx=60.0, ly=20.0, lz=20.0, n=48000, steps=20,
              tune=True),
        # The same slab in FP64, advanced one step at a time by a program that owns the
        # state in host memory (couples its own fields between the steps).
        _case("slab_fp64_host", kind="host", shape="slab", lx=60.0, ly=20.0, lz=20.0, n=48000,
              precision=0, tune=True),
        # A small porous sample with the wall density phi of Sec. 3.2 switched on.
        _case("rock64_phi", kind="step", shape="rock", nvox=64, porosity=0.15, steps=10, phi=True),
        # Poiseuille slit 100 x 40 x 20 (Sec. 4.2 shape): walls from a voxel image.
        _case("slit", kind="step", shape="slit", lx=100.0, ly=40.0, lz=20.0, n=480000, g=0.02,
              A_fs=-30.0, steps=10, tune=True),
        # The water slab of Sec. 4.1 in its 100^3 box, contracted to its liquid density.
        _case("water_slab", kind="step", shape="slab", lx=100.0, ly=100.0, lz=100.0, n=820000,
              fill=0.1206, A=-50.0, gamma=12.4, steps=5, tune=True),
        # The porous rock of Sec. 5-6, 256^3 voxels: 1.9M fluid and 2.5M wall particles.
        _case("rock256", kind="step", shape="rock", nvox=256, porosity=0.15, steps=5, tune=True),
        # 256 uneven replicas (parameter sweeps), one launch per kernel for all.
        _case("batch256", kind="batch", nrep=256, n_min=2000, n_max=20000, steps=5, tune=True),
        # A host program's evaluation of forces and densities at positions of its own:
        # two types, one reflecting axis, an odd count, no autotuning.
        _case("eval_mixed", kind="eval", shape="bulk", lx=17.3, ly=13.9, lz=14.2, n=20011,
              ntypes=2, perz=False),
        # Local densities for a caller that may not allocate (20^3 liquid).
        _case("density_noalloc", kind="density", shape="bulk", lx=20.0, ly=20.0, lz=20.0,
              n=48000),
        # Gradient of one evaluation (forces, virial, densities): bulk liquid, FP32.
        _case("eval_vjp", kind="vjp", shape="bulk", lx=25.5, ly=25.5, lz=25.5, n=100003),
        # Calibration window of Sec. 4.1's parameters: 64 small slabs, 20 steps, FP64,
        # forward and backward.
        _case("window64", kind="window", nrep=64, n_min=600, n_max=2000, precision=0, steps=20),
    ]


_DEFAULT = dict(shape="", lx=0.0, ly=0.0, lz=0.0, n=0, nvox=0, porosity=0.0, fill=1.0 / 3.0,
                A=-40.0, B=25.0, gamma=4.5, A_fs=-40.0, g=0.0, ntypes=1, perz=True, precision=1,
                xi=0, rho_self=0, phi=False, nrep=0, n_min=0, n_max=0, steps=0, tune=False)


def _case(name, **kw):
    c = dict(_DEFAULT)
    if kw.get("shape") == "rock":
        c["g"] = 0.01
    c.update(kw)
    if name:
        c["name"] = name
    return c


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the families above at another size, odd sizes and options among them."""
    fam = rng.choice(("bulk", "slab", "slab", "slit", "rock", "rock", "batch", "eval", "host",
                      "density", "vjp", "window"))
    f64 = rng.random() < 0.3
    mix = dict(A=-round(rng.uniform(30.0, 50.0), 2), B=round(rng.uniform(15.0, 35.0), 2),
               xi=int(rng.random() < 0.15), rho_self=int(rng.random() < 0.1))
    if fam in ("bulk", "eval", "vjp", "host", "density"):
        top = {"density": 60000, "bulk": 400000, "vjp": 300000}.get(fam, 100000)
        n = int(_log(rng, 500, top if not f64 else min(top, 60000)))
        vol, a, b = n / 6.0, rng.uniform(0.75, 1.35), rng.uniform(0.75, 1.35)
        e = vol ** (1.0 / 3.0)
        box = [max(3.05, round(v, 3)) for v in (e * a, e * b, e / (a * b))]
        kw = dict(kind="step" if fam == "bulk" else fam, shape="bulk", lx=box[0], ly=box[1],
                  lz=box[2], n=n, precision=0 if f64 else 1, ntypes=rng.choice((1, 1, 2, 3)),
                  perz=rng.random() < 0.7, tune=rng.random() < 0.5)
        if fam == "bulk":
            kw["steps"] = rng.randint(5, 30)
        if fam == "density":
            mix["xi"] = 0
            kw["ntypes"] = 1
        return _case("", **kw, **mix)
    if fam == "slab":
        n = int(_log(rng, 3000, 60000 if f64 else 900000))
        ly = round((n / 18.0) ** (1.0 / 3.0) * rng.uniform(0.8, 1.6), 3)
        lz = round((n / 18.0) ** (1.0 / 3.0) * rng.uniform(0.8, 1.6), 3)
        lx = round(max(3.2, n / 6.0 / (ly * lz)) * 3.0, 3)
        return _case("", kind="step", shape="slab", lx=lx, ly=max(3.1, ly), lz=max(3.1, lz), n=n,
                     precision=0 if f64 else 1, steps=rng.randint(2, 4) if f64 else rng.randint(3, 12),
                     tune=rng.random() < 0.7, **mix)
    if fam == "slit":
        n = int(_log(rng, 5000, 700000))
        h = 0.5 * rng.randint(8, 44)
        area = n / 6.0 / h
        ly = 0.5 * max(7, int(2.0 * math.sqrt(area) * rng.uniform(0.5, 1.5)))
        lx = 0.5 * max(7, round(2.0 * area / ly))
        n = int(min(n, 6.2 * lx * ly * h))
        return _case("", kind="step", shape="slit", lx=lx, ly=ly, lz=h, n=n, g=0.02,
                     A_fs=-round(rng.uniform(20.0, 40.0), 2), steps=rng.randint(3, 8),
                     phi=rng.random() < 0.3, tune=rng.random() < 0.6, **mix)
    if fam == "rock":
        nvox = int(_log(rng, 24, 250))
        return _case("", kind="step", shape="rock", nvox=nvox, porosity=round(rng.uniform(0.1, 0.4), 3)
                     if nvox < 160 else 0.15, steps=rng.randint(2, 5), phi=rng.random() < 0.3,
                     precision=0 if f64 and nvox < 96 else 1, tune=rng.random() < 0.6, **mix)
    if fam == "batch":
        lo = int(_log(rng, 200, 4000))
        return _case("", kind="batch", nrep=int(_log(rng, 4, 220)), n_min=lo,
                     n_max=lo * rng.randint(2, 5), steps=rng.randint(2, 8), tune=rng.random() < 0.6)
    lo = rng.randint(400, 900)
    return _case("", kind="window", nrep=rng.randint(4, 64), n_min=lo, n_max=lo + rng.randint(50, 1200),
                 precision=0 if rng.random() < 0.6 else 1, steps=rng.randint(3, 20))


# ---- what a program has in hand ---------------------------------------------------

class _Sys:
    """A plain description of one system: box, tables, particles, walls."""


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _liquid(g, n, lo, hi):
    """n particles of a disordered liquid in the box [lo, hi): sites of a cubic
    lattice (a few left empty at random), each displaced by up to a third of
    the spacing, so that the local density is the liquid's everywhere."""
    e = [h - l for l, h in zip(lo, hi)]
    a = (e[0] * e[1] * e[2] / n) ** (1.0 / 3.0)
    m = [max(1, int(v / a)) for v in e]
    while m[0] * m[1] * m[2] < n:
        k = min(range(3), key=lambda q: m[q] / e[q])
        m[k] += 1
    site = torch.randperm(m[0] * m[1] * m[2], generator=g, device=DEV)[:n].sort().values
    q = torch.stack([site % m[0], site // m[0] % m[1], site // (m[0] * m[1])], 1)
    h = torch.tensor([v / k for v, k in zip(e, m)], device=DEV, dtype=torch.float64)
    x = (q + 0.5 + 0.66 * (_rand(g, n, 3) - 0.5)) * h
    x = x[torch.randperm(n, generator=g, device=DEV)]
    return x + torch.tensor(lo, device=DEV, dtype=torch.float64)


def _rock_mask(g, nvox, porosity, corr=4.0):
    """Periodic Gaussian random field (covariance exp(-r^2 / 2 corr^2) in
    voxels), its lowest `porosity` quantile the pores; uint8, 1 = solid."""
    w = torch.randn(nvox, nvox, nvox, generator=g, device=DEV, dtype=torch.float32)
    k = torch.fft.fftfreq(nvox, device=DEV) * 2 * math.pi
    kr = torch.fft.rfftfreq(nvox, device=DEV) * 2 * math.pi
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + kr[None, None, :] ** 2
    f = torch.fft.irfftn(torch.fft.rfftn(w) * torch.exp(-k2 * corr * corr / 4.0), s=w.shape)
    thr = f.reshape(-1).kthvalue(max(1, int(porosity * nvox ** 3))).values
    return (f > thr).to(torch.uint8)


def _velocities(g, n):
    v = _randn(g, n, 3) * math.sqrt(KT)
    return v - v.mean(0, keepdim=True) if n > 1 else v


def _system(c, seed):
    """The system of a single-system case (before the library adds its walls)."""
    g = _gen(seed)
    s = _Sys()
    s.seed, s.mask, s.voxel, s.wall_density, s.shell = seed * 7919 + 17, None, 0.5, 6.0, 1.0
    # the sample (image and packed walls) is the case's, the fluid the seed's
    s.wall_seed, s.frozen, s.g = 1001, -1, (c["g"], 0.0, 0.0)
    s.precision, s.xi, s.rho_self = c["precision"], c["xi"], c["rho_self"]
    s.periodic, s.lo = [1, 1, 1 if c["perz"] else 0], [0.0, 0.0, 0.0]
    nt = c["ntypes"]
    if c["shape"] == "bulk":
        s.L = [c["lx"], c["ly"], c["lz"]]
        s.x = _liquid(g, c["n"], s.lo, s.L)
    elif c["shape"] == "slab":
        s.L = [c["lx"], c["ly"], c["lz"]]
        a = 0.5 * (1.0 - c["fill"])
        s.x = _liquid(g, c["n"], (a * s.L[0], 0.0, 0.0), ((1.0 - a) * s.L[0], s.L[1], s.L[2]))
    elif c["shape"] == "slit":
        s.lo, s.L, s.periodic = [0.0, 0.0, -1.0], [c["lx"], c["ly"], c["lz"] + 2.0], [1, 1, 0]
        s.x = _liquid(g, c["n"], (0.0, 0.0, 0.0), (c["lx"], c["ly"], c["lz"]))
        nx, ny, nz = (int(round(v / s.voxel)) for v in s.L)
        z = s.lo[2] + (torch.arange(nz, device=DEV) + 0.5) * s.voxel
        solid = (z < 0.0) | (z >= c["lz"])
        s.mask = solid[:, None, None].expand(nz, ny, nx).to(torch.uint8).contiguous()
    else:
        L = c["nvox"] * s.voxel
        s.L = [L, L, L]
        s.mask = _rock_mask(_gen(c["nvox"]), c["nvox"], c["porosity"])
        pore = (s.mask.reshape(-1) == 0).nonzero().reshape(-1)
        # one particle at a random point of three pore voxels out of four: density 6
        pick = pore[torch.randperm(pore.numel(), generator=g, device=DEV)[: (3 * pore.numel()) // 4]]
        nv = c["nvox"]
        q = torch.stack([pick % nv, pick // nv % nv, pick // (nv * nv)], 1)
        s.x = (q + _rand(g, pick.numel(), 3)) * s.voxel
    n = s.x.shape[0]
    s.v = _velocities(g, n)
    s.t = torch.randint(0, nt, (n,), generator=g, device=DEV, dtype=torch.int32)
    if s.mask is not None:
        s.frozen, nt = nt, nt + 1
    _tables(s, nt, c["A"], c["B"], c["gamma"], c["A_fs"])
    return s


def _tables(s, nt, A, B, gamma, A_fs=-40.0):
    q = np.add.outer(np.arange(8), np.arange(8)).astype(float)
    free = q * (nt > 1) * (s.frozen < 0)
    s.nt, s.A, s.B, s.G = nt, A + 3.0 * free, B - free, gamma + 0.5 * free
    if s.frozen >= 0:
        s.A[s.frozen, :s.frozen] = A_fs
        s.A[:s.frozen, s.frozen] = A_fs


def _params(s):
    p = I.MDPDParams(box_lo=tuple(s.lo), box=tuple(s.L), periodic=tuple(s.periodic), rc=RC, rd=RD,
                     dt=DT, kT=KT, ntypes=s.nt, g=tuple(s.g),
                     frozen_types=(s.frozen,) if s.frozen >= 0 else (), precision=s.precision,
                     xi_dist=s.xi, rho_self=s.rho_self)
    p.A[:], p.B[:], p.gamma[:] = s.A, s.B, s.G
    return p


class _Handle:
    """A program's system made from device arrays (freed with the object)."""

    def __init__(self, s, stream):
        torch.cuda.current_stream().synchronize()
        self.h = None
        self.h = M.mdpd_create_dev(_params(s), s.x.contiguous(), s.v.contiguous(), s.t, s.seed, stream)
        if s.mask is not None:
            M.mdpd_set_walls(self.h, s.mask.cpu().numpy(), s.voxel, s.lo, s.wall_density, s.shell,
                             s.frozen, s.wall_seed)
        self.n = M.mdpd_num_particles(self.h)

    def __del__(self):
        if self.h is not None:
            M.mdpd_destroy(self.h)
            self.h = None


def _replicas(c, seed):
    """Uneven liquid slabs, each with parameters of its own (as for sweeps and fits)."""
    r = np.random.default_rng(c["nrep"])      # sizes and parameters are the case's
    g = _gen(seed)
    out = []
    for k in range(c["nrep"]):
        n = int(r.integers(c["n_min"], c["n_max"] + 1))
        s = _Sys()
        e = (n / 6.0) ** (1.0 / 3.0)
        s.lo, s.L, s.periodic, s.frozen, s.g = [0.0] * 3, [3 * e, e, e], [1, 1, 1], -1, (0.0,) * 3
        s.precision, s.xi, s.rho_self, s.mask, s.seed = c["precision"], 0, 0, None, seed + k
        s.x = _liquid(g, n, (e, 0.0, 0.0), (2 * e, e, e))
        s.v = _velocities(g, n)
        s.t = torch.zeros(n, dtype=torch.int32, device=DEV)
        _tables(s, 1, float(r.uniform(-50.0, -30.0)), float(r.uniform(15.0, 35.0)), 4.5)
        out.append(s)
    return out


def _empty(*shape):
    return torch.empty(*shape, dtype=torch.float64, device=DEV)


def prepare(case, seed):
    c = dict(_DEFAULT, **case)
    st = {"c": c, "stream": torch.cuda.Stream()}
    kind = c["kind"]
    if kind in ("batch", "window"):
        reps = _replicas(c, seed)
        x, v = torch.cat([s.x for s in reps]), torch.cat([s.v for s in reps])
        st["ps"] = [_params(s) for s in reps]
        b = M.Batch(st["ps"], [s.x.shape[0] for s in reps], x.cpu().numpy(), v.cpu().numpy(),
                    torch.cat([s.t for s in reps]).cpu().numpy(), [s.seed for s in reps], st["stream"])
        st["b"], n = b, b.n
        if kind == "window":
            st["leaves"] = [t.requires_grad_(True) for t in
                            [x, v] + [torch.tensor(np.stack([getattr(s, k) for s in reps]), device=DEV)
                                      for k in ("A", "B", "G")]]
            st["cot"] = _window_cotangents(c, seed, n)
            return st
        if c["tune"]:
            b.autotune()
        st["out"] = [_empty(n, 3), _empty(n, 3), _empty(n)]
        return st
    s = _system(c, seed)
    if kind == "density":
        st["p"], st["x"] = _params(s), s.x.contiguous()
        return st
    h = _Handle(s, st["stream"])
    st["h"], n = h, h.n
    if c["phi"]:
        M.mdpd_set_option(h.h, M.OPT_WALL_DENSITY, 1)
    if c["tune"]:
        M.mdpd_autotune(h.h)
    if kind == "step":
        st["out"] = [_empty(n, 3), _empty(n, 3), _empty(n)]
    elif kind == "eval":
        st["x"], st["v"] = _moved(s, seed)
        st["out"] = [_empty(n, 3), _empty(n)]
    elif kind == "vjp":
        st["cot"] = _vjp_cotangents(seed, n)
    elif kind == "host":
        # the state the program holds, in page-locked memory
        host = [torch.empty(n, 3, dtype=torch.float64).pin_memory() for _ in range(3)]
        st["host"] = [t.numpy() for t in host]
        st["keep"] = host
        M.mdpd_get_state(h.h, st["host"][0], st["host"][1], want_type=False, want_rho=False)
        M.mdpd_get_accel(h.h, st["host"][2])
    return st


def _moved(s, seed):
    """Positions and velocities that a host program asks the forces for."""
    g = _gen(seed + 5)
    x = s.x + 0.05 * (_rand(g, *s.x.shape) - 0.5)
    lo = torch.tensor(s.lo, device=DEV, dtype=torch.float64)
    L = torch.tensor(s.L, device=DEV, dtype=torch.float64)
    return torch.minimum(torch.maximum(x, lo), lo + L * (1 - 1e-9)).contiguous(), _randn(g, *s.v.shape)


def _vjp_cotangents(seed, n):
    g = _gen(seed + 6)
    return _randn(g, n, 3), _randn(g, 1, 6) * 1e-2, _randn(g, n)


def _window_cotangents(c, seed, n):
    g = _gen(seed + 7)
    return _randn(g, n, 3), _randn(g, n, 3), _randn(g, n), _randn(g, c["nrep"], 6) * 1e-2


# ---- one pass --------------------------------------------------------------------

def _typed(c, v):
    """A frame in the type that the run's pair arithmetic determines it to."""
    if c["precision"] == 0:
        return v
    return v.float() if isinstance(v, torch.Tensor) else v.astype(np.float32)


def run(st):
    c = st["c"]
    kind = c["kind"]
    with torch.cuda.stream(st["stream"]):
        if kind == "step":
            h, o = st["h"].h, st["out"]
            M.mdpd_step(h, c["steps"])
            M.mdpd_get_state_dev(h, o[0], o[1], None, o[2])
            got = {"x": o[0], "v": o[1], "rho": o[2], "obs": M.mdpd_observables(h)}
            if c["phi"]:
                got["phi"] = M.mdpd_get_wall_density(h)
            return {k: _typed(c, v) for k, v in got.items()}
        if kind == "batch":
            b, o = st["b"], st["out"]
            b.step(c["steps"])
            M.mdpd_get_state_dev(b.h, o[0], o[1], None, o[2])
            return {"x": _typed(c, o[0]), "v": _typed(c, o[1]), "rho": _typed(c, o[2]),
                    "obs": _typed(c, b.observables())}
        if kind == "eval":
            h, o = st["h"].h, st["out"]
            M.mdpd_set_state_dev(h, st["x"], st["v"])
            M.mdpd_forces_dev(h, o[0], o[1])
            return {"force": _typed(c, o[0]), "rho": _typed(c, o[1])}
        if kind == "host":
            h, (x, v, a) = st["h"].h, st["host"]
            M.mdpd_set_state_accel(h, x, v, a)
            M.mdpd_step(h, 1)
            M.mdpd_get_state(h, x, v, want_type=False, want_rho=False)
            M.mdpd_get_accel(h, a)
            return {"x": _typed(c, x), "v": _typed(c, v), "a": _typed(c, a)}
        if kind == "density":
            rho = _empty(st["x"].shape[0])
            M.mdpd_density_noalloc(st["p"], st["x"], rho, st["stream"])
            return {"rho": _typed(c, rho)}
        if kind == "vjp":
            xb, ub, tb = AD.eval_vjp(st["h"], *st["cot"])
            return {"xbar": _typed(c, xb), "ubar": _typed(c, ub), "theta": _typed(c, tb)}
        xk, vk, rho, W = AD.window(st["b"], st["ps"], *st["leaves"], c["steps"], step0=0,
                                   observables=True)
        grads = torch.autograd.grad((xk, vk, rho, W), st["leaves"], st["cot"])
        names = ("x", "v", "rho", "W", "gx", "gv", "gA", "gB", "gG")
        return {k: _typed(c, t.detach()) for k, t in zip(names, (xk, vk, rho, W) + grads)}


# ---- the work a pass cannot do without ---------------------------------------------

#: floating operations of one directed pair (Eq. 1 with its virial), of one density term
#: and of its random draw's integer arithmetic counted as operations
PAIR_OPS, DENSITY_OPS, VJP_OPS = 100.0, 12.0, 160.0


def _counts(c):
    """(mobile particles, all particles, partners within r_c of a mobile one), estimated."""
    k = 4.0 / 3.0 * math.pi * 6.0
    if c["kind"] in ("batch", "window"):
        n = c["nrep"] * 0.5 * (c["n_min"] + c["n_max"])
        return n, n, k
    if c["shape"] == "slit":
        return c["n"], c["n"] + 12.0 * c["lx"] * c["ly"], k
    if c["shape"] == "rock":
        vol = (0.5 * c["nvox"]) ** 3
        m = 6.0 * c["porosity"] * vol
        return m, m + 6.0 * vol * 1.3 * c["porosity"], k
    return c["n"], c["n"], k


def work(case):
    c = dict(_DEFAULT, **case)
    m, n, k = _counts(c)
    w = 8.0 if c["precision"] == 0 else 4.0
    step_flops = m * k * (PAIR_OPS + DENSITY_OPS)
    # a step reads and writes the mobile state (x, v in FP64) and reads the walls' positions
    step_bytes = 96.0 * m + 24.0 * (n - m)
    kind = c["kind"]
    if kind in ("step", "batch"):
        return {"bytes": c["steps"] * step_bytes + 7.0 * w * n, "flops": c["steps"] * step_flops}
    if kind == "host":
        return {"bytes": step_bytes + 2 * 72.0 * n, "flops": step_flops}
    if kind == "eval":
        return {"bytes": (48.0 + 4.0 * w) * n, "flops": step_flops}
    if kind == "density":
        return {"bytes": (24.0 + w) * n, "flops": n * k * DENSITY_OPS}
    if kind == "vjp":
        return {"bytes": (48.0 + 32.0 + 6.0 * w) * n, "flops": n * k * (VJP_OPS + 2 * DENSITY_OPS)}
    K = c["steps"]
    return {"bytes": (K * (48.0 + 96.0) + 200.0) * n,
            "flops": n * k * (K + 1) * (PAIR_OPS + VJP_OPS + 4 * DENSITY_OPS)}


# ---- the same in 64 bits -------------------------------------------------------------

_LOW = 0xFFFFFFFF


def _mulhilo(a, b):
    """High and low words of a * b (a a Python constant, b an int64 tensor below 2^32)."""
    hi = (a * (b >> 16) + ((a * (b & 0xFFFF)) >> 16)) >> 16
    return hi, (a * b) & _LOW


def _philox(c, key):
    """Philox-4x32-10 (Salmon et al. 2011) on int64 tensors holding 32-bit words."""
    k0, k1 = key
    for r in range(10):
        h0, l0 = _mulhilo(0xD2511F53, c[0])
        h1, l1 = _mulhilo(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & _LOW, (k1 + 0xBB67AE85) & _LOW
    return c


def _words(seed):
    return seed & _LOW, (seed >> 32) & _LOW


def _draws(s, i, j, step):
    """xi_ij of the pairs for one step."""
    lo, hi = torch.minimum(i, j), torch.maximum(i, j)
    s0, s1 = _words(step)
    w = _philox([lo, hi, torch.full_like(lo, s0), torch.full_like(lo, s1)], _words(s.seed))
    if s.xi == 0:
        return math.sqrt(3.0) * (2 * (w[0] >> 8) + 1 - 2 ** 24).double() * 2.0 ** -24
    u1, u2 = ((w[0] >> 8).double() + 0.5) * 2.0 ** -24, ((w[1] >> 8).double() + 0.5) * 2.0 ** -24
    return torch.sqrt(-2.0 * torch.log(u1)) * torch.cos(2.0 * math.pi * u2)


def _place_walls(s):
    """Wall particles of the voxel image: solid voxels within `shell` of a pore
    voxel (centre to centre, periodic axes wrapped) get floor(rho h^3 + u)
    particles at uniform points, drawn by voxel id."""
    m = s.mask != 0
    R, R2 = int(s.shell / s.voxel + 1e-9), int((s.shell / s.voxel) ** 2 + 1e-9)
    near = torch.zeros_like(m)
    for dz in range(-R, R + 1):
        for dy in range(-R, R + 1):
            for dx in range(-R, R + 1):
                if dx * dx + dy * dy + dz * dz > R2:
                    continue
                p = ~m
                for axis, d, per in ((0, dz, s.periodic[2]), (1, dy, s.periodic[1]), (2, dx, s.periodic[0])):
                    if d == 0:
                        continue
                    p = torch.roll(p, -d, axis)
                    if not per:
                        idx = [slice(None)] * 3
                        idx[axis] = slice(-d, None) if d > 0 else slice(0, -d)
                        p = p.clone()
                        p[tuple(idx)] = False
                near |= p
    vid = (m & near).reshape(-1).nonzero().reshape(-1)
    zero = torch.zeros_like(vid)
    tag = torch.full_like(vid, 0x57414C4C)
    key = _words(s.wall_seed)
    u = (_philox([vid, zero, tag, zero], key)[0].double() + 0.5) * 2.0 ** -32
    cnt = torch.floor(s.wall_density * s.voxel ** 3 + u).long()
    rep = torch.repeat_interleave(vid, cnt)
    first = torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
    k = torch.arange(rep.numel(), device=DEV) - first
    w = _philox([rep, k + 1, torch.full_like(rep, 0x57414C4C), torch.zeros_like(rep)], key)
    nz, ny, nx = s.mask.shape
    q = (rep % nx, rep // nx % ny, rep // (nx * ny))
    return torch.stack([s.lo[a] + (q[a].double() + (w[a].double() + 0.5) * 2.0 ** -32) * s.voxel
                        for a in range(3)], 1)


class _Exact:
    """One system in 64-bit torch: pairs by cells, Eq. 1, velocity Verlet."""

    def __init__(self, s):
        self.s = s
        x, v, t = s.x, s.v, s.t.long()
        if s.mask is not None:
            wx = _place_walls(s)
            x, v = torch.cat([x, wx]), torch.cat([v, torch.zeros_like(wx)])
            t = torch.cat([t, torch.full((wx.shape[0],), s.frozen, device=DEV)])
        self.t, self.n = t, x.shape[0]
        self.mob = t != s.frozen
        self.lo = torch.tensor(s.lo, device=DEV, dtype=torch.float64)
        self.L = torch.tensor(s.L, device=DEV, dtype=torch.float64)
        self.per = [bool(p) for p in s.periodic]
        self.g = torch.tensor(s.g, device=DEV, dtype=torch.float64)
        self.x, self.v, self.step = x.clone(), v.clone(), 0
        self.A, self.B, self.G = (torch.tensor(np.array(k), device=DEV) for k in (s.A, s.B, s.G))

    def pairs(self, x):
        """Directed pairs (i, j) with 0 < r < r_c."""
        x = x.detach()
        nc = [max(1, int(math.floor(l / RC))) for l in self.s.L]
        h = self.L / torch.tensor(nc, device=DEV, dtype=torch.float64)
        q = [torch.clamp(torch.floor((x[:, k] - self.lo[k]) / h[k]).long(), 0, nc[k] - 1) for k in range(3)]
        cell = q[0] + nc[0] * (q[1] + nc[1] * q[2])
        order = torch.argsort(cell)
        count = torch.bincount(cell, minlength=nc[0] * nc[1] * nc[2])
        start = torch.cumsum(count, 0) - count
        oi, oj = [], []
        me = torch.arange(self.n, device=DEV)
        offs = torch.tensor([(o % 3 - 1, o // 3 % 3 - 1, o // 9 - 1) for o in range(27)], device=DEV)
        for off in offs.split(27 if self.n <= 100_000 else 1):      # neighbour cells at once
            ok = torch.ones(off.shape[0], self.n, dtype=torch.bool, device=DEV)
            z = []
            for k in range(3):
                w = q[k] + off[:, k, None]
                if self.per[k]:
                    w = w % nc[k]
                else:
                    ok &= (w >= 0) & (w < nc[k])
                z.append(w)
            nb = (z[0] + nc[0] * (z[1] + nc[1] * z[2]))[ok]
            own = me.expand_as(ok)[ok]
            c = count[nb]
            i = torch.repeat_interleave(own, c)
            first = torch.repeat_interleave(torch.cumsum(c, 0) - c, c)
            j = order[torch.repeat_interleave(start[nb], c) + torch.arange(i.numel(), device=DEV) - first]
            r2 = (self.sep(x, i, j) ** 2).sum(1)
            keep = (r2 < RC * RC) & (r2 > 0)
            oi.append(i[keep])
            oj.append(j[keep])
        return torch.cat(oi), torch.cat(oj)

    def sep(self, x, i, j):
        d = x[i] - x[j]
        return torch.stack([d[:, k] - self.L[k] * torch.round(d[:, k].detach() / self.L[k])
                            if self.per[k] else d[:, k] for k in range(3)], 1)

    def density(self, x, i, j):
        d = self.sep(x, i, j)
        r = torch.sqrt((d * d).sum(1))
        cw = 15.0 / (2.0 * math.pi * RD ** 3)
        w = cw * torch.clamp(1.0 - r / RD, min=0.0) ** 2
        rho = torch.zeros(self.n, device=DEV, dtype=torch.float64).index_add(0, i, w)
        return rho + cw if self.s.rho_self else rho

    def evaluate(self, x, u, step, grad=False, pairs=None):
        """(a, W, rho) at positions x and velocities u with the draws of `step`."""
        i, j = self.pairs(x) if pairs is None else pairs
        rho = self.density(x, i, j)
        m = self.mob[i]
        fi, fj = i[m], j[m]
        a = torch.zeros_like(x)
        W = torch.zeros(6, device=DEV, dtype=torch.float64)
        size = fi.numel() if grad else 12_000_000
        for b in range(0, max(1, fi.numel()), max(1, size)):
            p, q = fi[b:b + size], fj[b:b + size]
            d = self.sep(x, p, q)
            r = torch.sqrt((d * d).sum(1))
            e = d / r[:, None]
            wc = 1.0 - r / RC
            wd = torch.clamp(1.0 - r / RD, min=0.0)
            A, B, G = self.A[self.t[p], self.t[q]], self.B[self.t[p], self.t[q]], self.G[self.t[p], self.t[q]]
            fc = A * wc + B * (rho[p] + rho[q]) * wd
            ev = (e * (u[p] - u[q])).sum(1)
            f = fc - G * wc * wc * ev + torch.sqrt(2.0 * G * KT) * wc * _draws(self.s, p, q, step) / math.sqrt(DT)
            a = a.index_add(0, p, f[:, None] * e)
            h = 0.5 * fc / r
            W = W + torch.stack([(h * d[:, s] * d[:, t]).sum() for s, t in
                                 ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))])
        return a + self.g * self.mob[:, None], W, rho

    def drift(self, x, v):
        s = self.s
        y = x + DT * v
        blocked = torch.zeros(self.n, dtype=torch.bool, device=DEV)
        cols = []
        for k in range(3):
            lo, hi = s.lo[k], s.lo[k] + s.L[k]
            w = y[:, k]
            if self.per[k]:
                w = torch.where(w >= hi, w - s.L[k], torch.where(w < lo, w + s.L[k], w))
            else:
                blocked |= (w < lo) | (w >= hi)
            cols.append(w)
        y = torch.stack(cols, 1)
        if s.mask is not None:
            nz, ny, nx = s.mask.shape
            q = torch.floor((y.detach() - self.lo) / s.voxel).long()
            inside = ((q >= 0) & (q < torch.tensor([nx, ny, nz], device=DEV))).all(1) & ~blocked
            vid = torch.where(inside, q[:, 0] + nx * (q[:, 1] + ny * q[:, 2]), torch.zeros_like(q[:, 0]))
            blocked |= inside & (s.mask.reshape(-1)[vid] != 0)
        stay = (blocked | ~self.mob)[:, None]
        return torch.where(stay, x, y), torch.where(blocked[:, None] & self.mob[:, None], -v, v)

    def run(self, steps, grad=False):
        """Velocity Verlet from (self.x, self.v); returns (x, v, rho, W, a)."""
        x, v, m = self.x, self.v, self.mob[:, None]
        a, W, rho = self.evaluate(x, v, self.step, grad)
        for _ in range(steps):
            v = v + torch.where(m, 0.5 * DT * a, torch.zeros_like(a))
            x, v = self.drift(x, v)
            self.step += 1
            a, W, rho = self.evaluate(x, v, self.step, grad)
            v = v + torch.where(m, 0.5 * DT * a, torch.zeros_like(a))
        return x, v, rho, W, a

    def observables(self, v, W):
        m = self.mob
        p, s2, nm = v[m].sum(0), (v[m] ** 2).sum(0), float(m.sum())
        ke = 0.5 * s2.sum()
        kT = 2.0 * ke / (3.0 * (nm - 1.0)) if nm > 1 else torch.zeros_like(ke)
        return torch.cat([p, ke[None], kT[None], W, s2,
                          torch.tensor([nm, float(self.step)], device=DEV, dtype=torch.float64)])

    def phi(self, x):
        """Wall density of the mobile particles (Sec. 3.2)."""
        i, j = self.pairs(x)
        m = self.mob[i] & ~self.mob[j]
        i, j = i[m], j[m]
        r = torch.sqrt((self.sep(x, i, j) ** 2).sum(1))
        w = 15.0 / (2.0 * math.pi * RC ** 3) * (1.0 - r / RC) ** 2
        return torch.zeros(self.n, device=DEV, dtype=torch.float64).index_add(0, i, w)


def exact(case, seed):
    c = dict(_DEFAULT, **case)
    kind = c["kind"]
    if kind in ("step", "eval", "host", "density"):
        with torch.no_grad():
            s = _system(c, seed)
            if kind == "density":
                e = _Exact(s)
                return {"rho": e.density(e.x, *e.pairs(e.x))}
            if kind == "eval":
                s.x, s.v = _moved(s, seed)
                e = _Exact(s)
                a, W, rho = e.evaluate(e.x, e.v, 0)
                return {"force": a, "rho": rho}
            e = _Exact(s)
            x, v, rho, W, a = e.run(1 if kind == "host" else c["steps"])
            if kind == "host":
                return {"x": x, "v": v, "a": a}
            got = {"x": x, "v": v, "rho": rho, "obs": e.observables(v, W)}
            if c["phi"]:
                got["phi"] = e.phi(x)
            return got
    if kind == "batch":
        with torch.no_grad():
            got = {"x": [], "v": [], "rho": [], "obs": []}
            for s in _replicas(c, seed):
                e = _Exact(s)
                x, v, rho, W, _ = e.run(c["steps"])
                for k, t in zip(got, (x, v, rho, e.observables(v, W)[None])):
                    got[k].append(t)
            return {k: torch.cat(t) for k, t in got.items()}
    if kind == "vjp":
        s = _system(c, seed)
        e = _Exact(s)
        ab, cw, rb = _vjp_cotangents(seed, e.n)
        leaves = [t.requires_grad_(True) for t in (e.x, e.v, e.A, e.B, e.G)]
        a, W, rho = e.evaluate(e.x, e.v, 0, grad=True)
        gx, gu, *gt = torch.autograd.grad([a, W, rho], leaves, [ab, cw[0], rb])
        # the gradient with respect to the entries of symmetric tables
        th = [t + t.T - torch.diag(torch.diag(t)) for t in gt]
        return {"xbar": gx, "ubar": gu, "theta": torch.stack(th)}
    reps = _replicas(c, seed)
    n = sum(s.x.shape[0] for s in reps)
    xb, vb, rb, wb = _window_cotangents(c, seed, n)
    got = {k: [] for k in ("x", "v", "rho", "W", "gx", "gv", "gA", "gB", "gG")}
    at = 0
    for r, s in enumerate(reps):
        e = _Exact(s)
        leaves = [t.requires_grad_(True) for t in (e.x, e.v, e.A, e.B, e.G)]
        x, v, rho, W, _ = e.run(c["steps"], grad=True)
        k = slice(at, at + e.n)
        at += e.n
        gr = torch.autograd.grad([x, v, rho, W], leaves, [xb[k], vb[k], rb[k], wb[r]])
        for name, t in zip(got, (x, v, rho, W[None]) + gr[:2] +
                           tuple((t + t.T - torch.diag(torch.diag(t)))[None] for t in gr[2:])):
            got[name].append(t.detach())
    return {k: torch.cat(t) for k, t in got.items()}
