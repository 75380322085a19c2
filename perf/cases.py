"""What this framework's speed is measured on: the calls a user of the particle
cycle makes, from the smallest discharge to the largest, each through the public
entry points of ``paper_1801_00972_gb300``.

A case is a dict of plain values.  ``kind`` says which calls a pass makes:

  step      a run advanced by ``steps`` full time steps (``Run.step``), then the grain
            charges and the potential read, as a monitoring loop does;
  ensemble  independent runs of uneven size stepped side by side (``Batch.step``), the
            grain charges and potential of each read;
  advance   tracer particles in an imposed potential: ``set_phi``, then ``steps``
            particle half steps (``Run.advance``) and the charge density read;
  solve     the field solve alone from a zero potential (``set_phi``, ``Run.solve``);
  noalloc   the allocation-free field solve on device buffers (``pic_solve_noalloc``);
  start     a new run from host particle arrays (``Run(...)``: upload, grain tables, first
            deposit and field), its charge density, potential and grain tables read.

Meshes, densities and options are the package's own workloads (``inputs.workload``,
``inputs.ensemble``), the benchmark's legs and the tests' small and uneven meshes, and
sizes between them.  The drive's phase is kept away from its zero crossing, where the
potential would be particle noise alone.
"""
from __future__ import annotations

import ctypes
import dataclasses
import math

import numpy as np
import torch

import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import inputs as I

EPS0 = 8.8541878128e-12
DX = 0.2e-3


def _step(name, nx, ny, nz, n, grains, steps, prec="mixed", sort_every=5, v_dc=0.0, v_rf=100.0, phase=1.2,
          pressure=2.0, coulomb=False, diagnostics=False):
    return dict(name=name, kind="step", nx=nx, ny=ny, nz=nz, n=n, grains=grains, steps=steps, prec=prec,
                sort_every=sort_every, v_dc=v_dc, v_rf=v_rf, phase=phase, pressure=pressure, coulomb=coulomb,
                diagnostics=diagnostics)


def listed():
    return [
        # the small DC sheath with one grain (workload 0), with a Run's own defaults: latency and launches
        _step("dc_32x32x64_2e5", 32, 32, 64, 200_000, 1, 4, sort_every=20, v_dc=-50.0, v_rf=0.0),
        # the rf sheath with the 7-grain cluster (workload 1), the everyday run
        _step("rf_64x64x256_1e7", 64, 64, 256, 10_000_000, 7, 5),
        # the paper-scale 50-grain cluster (workload 2)
        _step("rf_128x128x512_2e8", 128, 128, 512, 200_000_000, 50, 3),
        # the largest workload (workload 4, the benchmark's headline)
        _step("rf_256x256x1024_5e8", 256, 256, 1024, 500_000_000, 100, 2),
        # the reference precision on the everyday run
        _step("fp64_64x64x256_1e7", 64, 64, 256, 10_000_000, 7, 2, prec="fp64"),
        # the everyday run with Coulomb collisions
        _step("coulomb_64x64x256_1e7", 64, 64, 256, 10_000_000, 7, 3, coulomb=True),
        # the data-taking phase of a run: phase-resolved moments and the energy histogram every step
        _step("diag_64x64x128_4e6", 64, 64, 128, 4_000_001, 19, 3, diagnostics=True),
        # an uneven mesh and odd particle count at higher pressure
        _step("rf_80x48x100_3e6", 80, 48, 100, 2_999_999, 11, 4, v_dc=-20.0, pressure=6.0, sort_every=10),
        # a parameter study: independent runs side by side (the ensemble workload, fewer of its runs)
        dict(name="ensemble_12", kind="ensemble", runs=12, study=3, n_lo=100_000, n_hi=2_000_000, steps=2, prec="mixed",
             sort_every=5),
        # tracers in an imposed potential: the particle half alone
        dict(name="advance_64x64x64_4e6", kind="advance", nx=64, ny=64, nz=64, n=4_000_000, steps=4, prec="mixed",
             sort_every=5, phase=1.2, pressure=2.0),
        # the field solve from a zero potential
        dict(name="solve_64x64x256", kind="solve", nx=64, ny=64, nz=256, n=2_000_000, prec="mixed", v_dc=-50.0),
        # a run's start from host particles
        dict(name="start_64x64x128_2e6", kind="start", nx=64, ny=64, nz=128, n=2_000_000, grains=7, prec="mixed",
             v_dc=-50.0, v_rf=100.0, phase=1.2),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _coarsens(nx, ny, nz):
    """Whether halving takes the mesh to a small one whose sides are multiples of 4: other meshes the
    library refuses, or solves with many sweeps, and no workload has them."""
    small = False
    while nx % 4 == 0 and ny % 4 == 0 and nz % 2 == 0 and nz >= 4:
        nx, ny, nz = nx // 2, ny // 2, nz // 2
        small = small or (nx * ny * (nz + 1) <= 32000 and nx % 4 == 0 and ny % 4 == 0 and nz >= 4)
    return small and nx * ny * (nz + 1) <= 12000


def _mesh(rng, most):
    """Even and uneven edges as the workloads' and between them, up to ``most`` cells."""
    while True:
        nx = rng.choice((16, 24, 32, 32, 40, 48, 64, 64, 64, 80, 96, 112, 128, 128, 256))
        ny = rng.choice((16, 24, 32, 32, 40, 48, 64, 64, 64, 80, 96, 112, 128, 128, 256))
        nz = 4 * int(round(_log(rng, 32, 1024) / 4))
        if max(nx, ny) <= 4 * min(nx, ny) and nx * ny * nz <= most and _coarsens(nx, ny, nz):
            return nx, ny, nz


def draw(rng):
    kind = rng.choice(("step",) * 6 + ("ensemble", "advance", "solve", "noalloc", "start"))
    phase = round(rng.uniform(0.6, 2.4), 3)
    if kind == "step":
        prec = "fp64" if rng.random() < 0.2 else "mixed"
        extra = rng.random()
        plain = extra < 0.7
        nx, ny, nz = _mesh(rng, 2.0e7 if prec == "mixed" and plain else 2.0e6)
        n = int(min(nx * ny * nz * _log(rng, 3.0, 25.0), 3.0e8 if prec == "mixed" and plain else 1.5e7))
        c = _step("", nx, ny, nz, n, rng.randrange(1, 20), rng.randrange(2, 5), prec=prec,
                  sort_every=rng.choice((5, 5, 8, 10, 20)), v_dc=round(rng.uniform(-60.0, -10.0), 2),
                  v_rf=rng.choice((0.0, 80.0, 100.0)), phase=phase, pressure=round(_log(rng, 1.0, 6.0), 3),
                  coulomb=0.7 <= extra < 0.85, diagnostics=extra >= 0.85)
    elif kind == "ensemble":
        c = dict(kind=kind, runs=rng.randrange(3, 16), study=rng.randrange(1000), n_lo=100_000, n_hi=int(_log(rng, 3.0e5, 2.0e6)),
                 steps=rng.randrange(1, 4), prec=rng.choice(("mixed", "mixed", "fp64")), sort_every=rng.choice((5, 10)))
    elif kind == "advance":
        nx, ny, nz = _mesh(rng, 2.0e6)
        c = dict(kind=kind, nx=nx, ny=ny, nz=nz, n=int(min(nx * ny * nz * _log(rng, 3.0, 25.0), 1.5e7)),
                 steps=rng.randrange(1, 6), prec=rng.choice(("mixed", "mixed", "fp64")), sort_every=rng.choice((5, 10)),
                 phase=phase, pressure=round(_log(rng, 1.0, 6.0), 3))
    elif kind == "solve":
        nx, ny, nz = _mesh(rng, 4.0e6)
        c = dict(kind=kind, nx=nx, ny=ny, nz=nz, n=int(min(nx * ny * nz * 2, 2.0e6)),
                 prec=rng.choice(("mixed", "mixed", "fp64")), v_dc=round(rng.uniform(-60.0, -10.0), 2))
    elif kind == "noalloc":
        nx, ny, nz = rng.choice(((8, 8, 16), (16, 16, 32), (32, 16, 64), (32, 32, 64), (12, 12, 24), (32, 32, 120)))
        c = dict(kind=kind, nx=nx, ny=ny, nz=nz, density=round(rng.uniform(3.0, 25.0), 2),
                 prec=rng.choice(("mixed", "fp64")), v_dc=round(rng.uniform(-60.0, -10.0), 2))
    else:
        nx, ny, nz = _mesh(rng, 1.0e6)
        c = dict(kind=kind, nx=nx, ny=ny, nz=nz, n=int(min(nx * ny * nz * _log(rng, 1.0, 6.0), 3.0e6)),
                 grains=rng.randrange(1, 12), prec=rng.choice(("mixed", "mixed", "fp64")),
                 v_dc=round(rng.uniform(-60.0, -10.0), 2), v_rf=rng.choice((0.0, 100.0)), phase=phase)
    c.pop("name", None)
    return c


# ----------------------------------------------------------------- inputs
def _prec(case):
    return P.PIC_FP64 if case["prec"] == "fp64" else P.PIC_MIXED


def _workload(case, seed):
    """A discharge of the package's kind on the case's mesh, its grains placed from the seed."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    base = I.small(n_e=1, n_i=1, grains=0, pressure=case.get("pressure", 2.0))
    n = case["n"]
    n_e = n // 2
    lx, ly, lz = nx * DX, ny * DX, nz * DX
    ng = case.get("grains", 0)
    if ng:
        radius = min(1.5e-3, 0.3 * lx, 0.3 * ly, 0.3 * lz)
        pos, r = I.sphere_cluster(ng, radius, (lx / 2, ly / 2, min(5.6e-3, lz / 2)), 4e-6, 5e-6, DX, (nx, ny, nz), seed)
    else:
        pos, r = np.zeros((0, 3)), np.zeros(0)
    return dataclasses.replace(base, name="case", nx=nx, ny=ny, nz=nz, dx=DX, weight=1e15 * lx * ly * lz / n_e,
                               v_dc=case.get("v_dc", 0.0), v_rf=case.get("v_rf", 0.0), f_rf=13.56e6,
                               phase=case.get("phase", 0.0), grain_pos=pos, grain_r=r, seed=I.BASE_SEED + seed,
                               n_e=n_e, n_i=n - n_e)


def _room(wl):
    """Particle slots per species for a long run: ionization adds particles."""
    return tuple(int(1.5 * n) + 65536 for n in (wl.n_e, wl.n_i))


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _host(n):
    """A caller's own page-locked buffer of n doubles for the potential."""
    return torch.empty(n, dtype=torch.float64, pin_memory=True)


def _read_phi(ctx, buf):
    if P.load().pic_get_phi(ctx, ctypes.cast(buf.data_ptr(), ctypes.POINTER(ctypes.c_double)), buf.numel()) != P.PIC_OK:
        raise RuntimeError(P.pic_last_error(ctx))
    return buf


def prepare(case, seed):
    kind = case["kind"]
    if kind == "noalloc":
        rho = _charge(case, seed)
        return dict(case=case, rho=torch.from_numpy(rho).cuda(), phi=torch.zeros(rho.size, dtype=torch.float64, device="cuda"))
    if kind == "ensemble":
        wls = []
        for w in I.ensemble(case["runs"], seed=I.BASE_SEED + case["study"]):
            k = case["n_hi"] / 2.0e6   # the package's ensemble draws up to 2e6 particles a run
            n = max(case["n_lo"] // 2, int(w.n_e * k))
            gas = I.small(n_e=1, n_i=1, grains=0, pressure=1.0 + 3.0 * w.phase / (2 * math.pi))   # 1 to 4 Pa
            wls.append(dataclasses.replace(w, n_e=n, n_i=n, weight=w.weight * w.n_e / n, seed=w.seed + seed, n_gas=gas.n_gas, nu_max_e=gas.nu_max_e,
                                           nu_max_i=gas.nu_max_i, phase=0.6 + 1.8 * (w.phase / (2 * math.pi))))
        cap = case["n_hi"] + 65536   # a species' slots, for every run: at least twice its particles
        batch = P.Batch(wls, [I.sample_particles(w) for w in wls], prec=_prec(case), sort_every=case["sort_every"], capacity=(cap, cap))
        return dict(case=case, batch=batch, ng=[len(w.grain_r) for w in wls], out=[_host(w.nodes) for w in wls])
    wl = _workload(case, seed)
    if kind == "start":
        return dict(case=case, wl=wl, parts=I.sample_particles(wl))
    if kind == "solve":
        return dict(case=case, run=P.Run(wl, _particles(case, seed), prec=_prec(case), stream=_stream()), zero=np.zeros(wl.nodes), out=_host(wl.nodes))
    if kind == "advance":
        run = P.Run(wl, None, prec=_prec(case), stream=_stream(), sort_every=case["sort_every"], capacity=_room(wl))
        return dict(case=case, run=run, phi=_imposed(case, seed))
    flags = P.PIC_F_COULOMB if case["coulomb"] else 0
    more = {}
    if case["diagnostics"]:
        flags |= P.PIC_F_MOMENTS
        more = dict(mom_phases=16, eepf_bins=200, eepf_de_ev=0.1)
    run = P.Run(wl, None, prec=_prec(case), flags=flags, stream=_stream(), sort_every=case["sort_every"], capacity=_room(wl),
                **more)
    return dict(case=case, run=run, out=_host(wl.nodes))


# ----------------------------------------------------------------- one pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        r = state["run"]
        r.step(case["steps"])
        n_abs, q = r.grains()
        out = {"n_abs": n_abs, "q": q, "phi": _read_phi(r.ctx, state["out"])}
        if case["diagnostics"]:
            out["oml"] = r.oml_charges()
        return out
    if kind == "ensemble":
        b = state["batch"]
        b.step(case["steps"])
        return [{"q": P.pic_grain_charges(c, ng)[1], "phi": _read_phi(c, o)}
                for c, ng, o in zip(b.runs, state["ng"], state["out"])]
    if kind == "advance":
        r = state["run"]
        r.set_phi(state["phi"])
        for _ in range(case["steps"]):
            r.advance()
        return {"rho": r.rho()}
    if kind == "solve":
        r = state["run"]
        r.set_phi(state["zero"])
        r.solve()
        return {"phi": _read_phi(r.ctx, state["out"])}
    if kind == "noalloc":
        state["phi"].zero_()
        P.pic_solve_noalloc(case["nx"], case["ny"], case["nz"], DX, state["rho"].data_ptr(), _scale(case), case["v_dc"], 0.0,
                            state["phi"].data_ptr(), _prec(case), 1e-10, 60, _stream())
        return {"phi": state["phi"]}
    r = P.Run(state["wl"], state["parts"], prec=_prec(case), stream=_stream())
    out = {"rho": r.rho(), "phi": r.phi(), "tables": r.gtab()}
    r.close()
    return out


def work(case):
    """Bytes and operations a pass cannot do without: every particle record read and written and the
    charge and potential of every node, once per step; about 200 operations a particle and 60 a node."""
    kind = case["kind"]
    rec = 128 if case["prec"] == "fp64" else 64
    if kind == "ensemble":
        n = case["runs"] * 6.0e5 * case["n_hi"] / 2.0e6   # the ensemble's mean run
        nodes = case["runs"] * 2.0e5
        s = case["steps"]
        return {"bytes": s * (rec * n + 24.0 * nodes), "flops": s * (200.0 * n + 60.0 * nodes)}
    nodes = case["nx"] * case["ny"] * (case["nz"] + 1)
    if kind in ("solve", "noalloc"):
        return {"bytes": 16.0 * nodes, "flops": 60.0 * nodes}
    if kind == "start":
        return {"bytes": (52 + rec // 2) * case["n"] + 16.0 * nodes, "flops": 50.0 * case["n"] + 60.0 * nodes}
    s = case["steps"]
    return {"bytes": s * (rec * case["n"] + 24.0 * nodes), "flops": s * (200.0 * case["n"] + 60.0 * nodes)}


# ----------------------------------------------------------------- inputs written out here, and 64-bit results
def _weight(case):
    vol = case["nx"] * case["ny"] * case["nz"] * DX ** 3
    return 1e15 * vol / (case["n"] // 2) if "n" in case else 1e15 * DX ** 3 / case["density"]


def _scale(case):
    """From fixed-point charge (units e W 2^-42) to rho / eps0."""
    return 1.602176634e-19 * _weight(case) / DX ** 3 * 2.0 ** -42 / EPS0


def _particles(case, seed):
    """A quiet plasma with a depleted sheath: positions in the box, thermal velocities."""
    rng = np.random.default_rng(1000 + seed)
    ln = np.array([case["nx"], case["ny"], case["nz"]])
    out, base = [], 0
    for n, v in ((case["n"] // 2, 7.3e5), (case["n"] - case["n"] // 2, 269.0)):
        x = rng.random((n, 3)) * ln
        if base == 0:
            x[:, 2] = ln[2] * (0.1 + 0.9 * x[:, 2] / ln[2])
        x = np.minimum(x, ln - 1e-3) * DX
        out.append((x, rng.standard_normal((n, 3)) * v, np.arange(base, base + n, dtype=np.uint32)))
        base += n
    return out


def _deposit(case, particles):
    """Fixed-point charge of the particles on the nodes (14-bit weights per axis)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    rho = np.zeros(nx * ny * (nz + 1), np.int64)
    for sign, (x, _, _) in zip((-1, 1), particles):
        c = np.minimum(np.floor(x / DX).astype(np.int64), np.array([nx - 1, ny - 1, nz - 1]))
        f = x / DX - c
        if case["prec"] == "mixed":
            f = np.minimum(f.astype(np.float32), np.float32(0.99999994)).astype(np.float64)
        a = np.rint(f * 16384.0).astype(np.int64)
        for corner in range(8):
            d = np.array([corner & 1, (corner >> 1) & 1, corner >> 2])
            w = np.where(d == 1, a, 16384 - a).prod(axis=1)
            q = c + d
            np.add.at(rho, (q[:, 2] * ny + q[:, 1] % ny) * nx + q[:, 0] % nx, sign * w)
    return rho


def _charge(case, seed):
    """Fixed-point charge of a plasma with the case's particles per cell and species."""
    rng = np.random.default_rng(2000 + seed)
    n = case["nx"] * case["ny"] * (case["nz"] + 1)
    k = case["density"]
    return np.rint((rng.standard_normal(n) * math.sqrt(2 * k) * 0.3 + 0.1 * k * rng.random(n)) * 2.0 ** 42).astype(np.int64)


def _imposed(case, seed):
    """A sheath potential with a smooth lateral ripple, V per node."""
    rng = np.random.default_rng(3000 + seed)
    x = np.arange(case["nx"]) * (2 * math.pi / case["nx"])
    y = np.arange(case["ny"]) * (2 * math.pi / case["ny"])
    z = np.arange(case["nz"] + 1) / case["nz"]
    a, b = rng.uniform(0.0, 2 * math.pi, 2)
    v = -100.0 * math.sin(case["phase"])
    ramp = v * np.exp(-25.0 * z) + 8.0 * z * (1.0 - z)
    ripple = 0.5 * np.cos(x + a)[None, None, :] + 0.5 * np.cos(2 * y + b)[None, :, None]
    return (ramp[:, None, None] + ripple * np.sin(math.pi * z)[:, None, None]).reshape(-1)


def _poisson(case, rho):
    """-lap(phi) = rho / eps0 on the nodes, periodic in x and y, v_dc and 0 on the electrode planes."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    f = (rho.astype(np.float64) * _scale(case) * DX ** 2).reshape(nz + 1, ny, nx)[1:nz].copy()
    f[0] += case["v_dc"]
    g = np.fft.rfft2(f, axes=(1, 2))
    lam = (2 - 2 * np.cos(2 * math.pi * np.arange(ny) / ny))[:, None] + (2 - 2 * np.cos(2 * math.pi * np.arange(g.shape[2]) / nx))[None, :]
    p = np.zeros((nz - 1,) + lam.shape)
    for k in range(nz - 1):
        p[k] = 1.0 / (2.0 + lam - (p[k - 1] if k else 0.0))
        g[k] = p[k] * (g[k] + (g[k - 1] if k else 0.0))
    for k in range(nz - 3, -1, -1):
        g[k] += p[k] * g[k + 1]
    phi = np.zeros((nz + 1, ny, nx))
    phi[0] = case["v_dc"]
    phi[1:nz] = np.fft.irfft2(g, s=(ny, nx), axes=(1, 2))
    return phi.reshape(-1)


def exact(case, seed):
    if case["kind"] == "noalloc":
        return {"phi": _poisson(case, _charge(case, seed))}
    if case["kind"] == "solve":
        return {"phi": _poisson(case, _deposit(case, _particles(case, seed)))}
    return None
