"""The workloads that the speed of this library is measured on.

Every case goes through the package's public entry points, as a program that
couples a fluid solver to a particle solver calls them:

* ``step``     one eager ``cfdem_coupling_step`` (void fraction, projection,
               forces, fluid source) on one bed;
* ``replay``   the same step through ``cfdem_batch_coupling_step``, one or many
               beds, replayed as a CUDA graph from the second call on;
* ``host``     a replayed step whose inputs and results live in page-locked
               host memory (a fluid solver on the host cores);
* ``grad``     a loss of the step and its gradients, through
               ``paper_2211_01185_gb300.autograd`` (mixed) or the C entry
               points ``cfdem_adjoint`` and ``cfdem_mass_apply`` (FP64);
* ``dem``      the particle side: ten Velocity Verlet sub-steps with contacts;
* ``mapped``   location on a curved mesh and interpolation of the velocity.

The projection starts from zero in every pass, so that each pass does the
whole solve.  Results of the mixed path carry FP32 accuracy (forces and void
fraction good to 1e-5 by the library's contract): the program keeps them in
FP32, as one cast of the results' buffer at the end of the pass.  DEM
positions stay in FP64 on both paths.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2211_01185_gb300 import autograd as ag
from paper_2211_01185_gb300 import cfdem as cf
from paper_2211_01185_gb300 import synth

DEV = "cuda:0"
F64 = torch.float64
RHO_F, MU_F, RHO_P, G = 1.2, 1.8e-5, 2500.0, 9.81
#: DEM sub-steps of one pass and their length (the coupling frequency of the benchmark)
NSUB, DT = 10, 5e-6

# closures (drag_model)
DI_FELICE, RONG, KOCH_HILL, BEETSTRA = 0, 2, 3, 5


# ------------------------------------------------------------------ the cases

def _bed(name, path, k, ne, h, n, d, phi, precision, drag=DI_FELICE, model=0, shear=0,
         fluid_drag=0, conserve=0, shuffled=0):
    """One bed: k and ne the mesh, h the element edge [m], n spheres with
    diameters uniform in d [m] on a jittered lattice of solid fraction phi,
    numbered by the lattice or at random (a bed that has mixed)."""
    return {"name": name, "path": path, "k": k, "nx": ne[0], "ny": ne[1], "nz": ne[2], "h": h,
            "n": n, "d_lo": d[0], "d_hi": d[1], "phi": phi, "precision": precision,
            "drag": drag, "model": model, "shear": shear, "fluid_drag": fluid_drag,
            "conserve": conserve, "shuffled": shuffled}


def listed():
    return [
        # the smallest call: a laboratory-scale bed stepped eagerly, launches and latency only
        _bed("step_q1_2k", "step", 1, (8, 8, 32), 2.5e-3, 2000, (1e-3, 1e-3), 0.065,
             "mixed"),
        # the headline: the benchmark's bed, one graph replay per fluid step
        _bed("replay_q2_100k", "replay", 2, (32, 32, 128), 3.125e-3, 100_000, (2e-3, 2.8e-3),
             0.72, "mixed"),
        # the same bed in FP64 (the library's default precision), host to host
        _bed("host_q2_100k_fp64", "host", 2, (32, 32, 128), 3.125e-3, 100_000, (2e-3, 2.8e-3),
             0.72, "fp64"),
        # the largest: high-order elements six particle diameters wide, a settled bed
        _bed("replay_q3_1m", "replay", 3, (24, 24, 96), 6e-3, 1_000_000, (1e-3, 1e-3), 0.6,
             "mixed"),
        # every option of the forces, on a ragged Q3 mesh with a mixed-up bed, FP64
        _bed("step_q3_options_fp64", "step", 3, (11, 13, 31), 5e-3, 23_457, (1e-3, 2.5e-3),
             0.6, "fp64", drag=RONG, model=1, shear=1, fluid_drag=1, shuffled=1),
        # volume-conserving void fraction and another closure on a ragged Q2 mesh, mixed
        _bed("step_q2_conserve", "step", 2, (17, 23, 61), 4e-3, 61_111, (1.5e-3, 2.5e-3), 0.65,
             "mixed", drag=BEETSTRA, conserve=1, shuffled=1),
        # a parameter study: independent beds of uneven mesh, degree and size in one replay
        {"name": "ensemble_12", "path": "ensemble", "beds": 12, "layout": 4, "n_lo": 3000,
         "n_hi": 60_000, "ne_hi": 24, "precision": "mixed"},
        # gradients of a loss for calibration, through torch.autograd
        _bed("grad_q2_150k", "grad", 2, (24, 24, 96), 4e-3, 150_000, (2e-3, 2e-3), 0.5, "mixed"),
        # gradients on a small odd mesh through the C entry points, FP64
        _bed("grad_q1_9k_fp64", "grad", 1, (15, 13, 37), 3e-3, 9001, (1e-3, 2e-3), 0.5, "fp64",
             shuffled=1),
        # the particle side of one fluid step of the headline bed
        {"name": "dem_100k", "path": "dem", "n": 100_000, "side": 40, "d": 2.5e-3,
         "precision": "mixed", "shuffled": 0},
        # the same in FP64 (the default) for a small bed
        {"name": "dem_5k_fp64", "path": "dem", "n": 5003, "side": 13, "d": 2e-3,
         "precision": "fp64", "shuffled": 1},
        # a fluidised bed's cylinder: particles located on the curved mesh every fluid step
        {"name": "mapped_q2_120k", "path": "mapped", "k": 2, "n": 120_000, "n_core": 6,
         "n_ring": 4, "n_z": 40, "ncomp": 3},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ones' ranges."""
    path = rng.choice(["step", "step", "replay", "replay", "host", "grad", "dem", "mapped",
                       "ensemble"])
    precision = rng.choice(["mixed", "fp64"])
    if path == "dem":
        return {"path": path, "n": _log(rng, 1000, 100_000 if precision == "mixed" else 40_000),
                "side": rng.randint(9, 40),
                "d": rng.uniform(1e-3, 3e-3), "precision": precision,
                "shuffled": rng.randint(0, 1)}
    if path == "mapped":
        return {"path": path, "k": rng.randint(1, 3), "n": _log(rng, 1000, 120_000),
                "n_core": rng.randint(2, 6), "n_ring": rng.randint(1, 4),
                "n_z": rng.randint(5, 30), "ncomp": rng.choice([1, 3, 4])}
    if path == "ensemble":
        return {"path": path, "beds": rng.randint(2, 10), "layout": rng.randint(0, 10 ** 6),
                "n_lo": 1000, "n_hi": _log(rng, 5000, 50_000), "ne_hi": rng.randint(9, 22),
                "precision": "mixed"}
    k = rng.randint(1, 3)
    fp64, grad = precision == "fp64", path == "grad"
    n = _log(rng, 1500, 40_000 if fp64 or grad else 300_000)
    top = 96 // k if not (fp64 or grad) else 48 // k
    ne = (rng.randint(6, top // 2), rng.randint(6, top // 2), _log(rng, 8, top))
    d_hi = rng.uniform(1e-3, 3e-3)
    d_lo = d_hi * rng.uniform(0.5, 1.0)
    # elements such that the spheres take about a fifth of the box, one to six diameters wide
    v = n * math.pi / 6 * d_hi ** 3
    h = (v / (0.2 * ne[0] * ne[1] * ne[2])) ** (1.0 / 3.0)
    h = max(h, 1.0 * d_hi)
    if h > 6.0 * d_hi:
        d_hi, d_lo = h / 6.0, d_lo / d_hi * h / 6.0
    opt = not grad and rng.random() < 0.4
    c = _bed("", path, k, ne, h, n, (d_lo, d_hi), rng.uniform(0.4, 0.55), precision,
             drag=rng.choice([DI_FELICE, DI_FELICE, RONG, KOCH_HILL, BEETSTRA]),
             model=rng.randint(0, 1) if opt else 0, shear=int(opt and rng.random() < 0.5),
             fluid_drag=int(opt and rng.random() < 0.5), conserve=int(opt and rng.random() < 0.3),
             shuffled=rng.randint(0, 1))
    del c["name"]
    return c


def _ensemble_beds(case):
    """The beds of an ensemble: their sizes come from the case, the inputs from the seed."""
    rng = random.Random(case["layout"])
    beds = []
    for _ in range(case["beds"]):
        ne = (rng.randint(8, case["ne_hi"]), rng.randint(8, case["ne_hi"]),
              rng.randint(8, 2 * case["ne_hi"]))
        n = _log(rng, case["n_lo"], case["n_hi"])
        d = rng.uniform(1e-3, 3e-3)
        h = (n * math.pi / 6 * d ** 3 / (0.25 * ne[0] * ne[1] * ne[2])) ** (1.0 / 3.0)
        beds.append(_bed("", "replay", rng.randint(1, 3), ne, h, n, (d, d), 0.55,
                         case["precision"]))
    return beds


# ------------------------------------------------------------------ inputs

def _lattice(n, a_nn, ncx, ncy):
    """The first n sites of an FCC lattice of nearest-neighbour distance a_nn,
    ncx x ncy cells wide, by layers from the floor up."""
    a = a_nn * math.sqrt(2.0)
    j = torch.arange(n, device=DEV)
    layer, rest = j // (2 * ncx * ncy), j % (2 * ncx * ncy)
    cell, half, up = rest // 2, rest % 2, layer % 2
    ix, iy = cell % ncx, cell // ncx
    x = ix + torch.where(half == 1, 0.5, 0.0).to(F64)
    y = iy + torch.where((half == 1) != (up == 1), 0.5, 0.0).to(F64)
    z = 0.5 * layer.to(F64)
    return a * (torch.stack([x, y, z], dim=1) + 0.25)


def _rand(gen, *shape):
    return torch.rand(shape, generator=gen, device=DEV, dtype=F64)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFFFFFF)


def _geometry(c):
    ne = (c["nx"], c["ny"], c["nz"])
    return ne, tuple(c["h"] * v for v in ne)


def _radius(c):
    """The averaging radius: of the element's volume, at least the largest particle's."""
    return max((3.0 / (4.0 * math.pi)) ** (1.0 / 3.0) * c["h"], 0.5 * c["d_hi"])


def _inputs(c, gen):
    """Particles and nodal fields of one bed."""
    ne, L = _geometry(c)
    k, n = c["k"], c["n"]
    kp = max(1, k - 1)
    a_nn = c["d_hi"] * (0.74048 / c["phi"]) ** (1.0 / 3.0)
    cells = [max(1, int(L[a] / (a_nn * math.sqrt(2.0)) + 1e-9)) for a in (0, 1)]
    x = _lattice(n, a_nn, *cells)
    x = x + 0.5 * (a_nn - c["d_hi"]) * (_rand(gen, n, 3) - 0.5)
    top = torch.tensor(L, device=DEV, dtype=F64)
    x = torch.minimum(torch.clamp(x, min=0.0), top * (1 - 1e-9))
    r = 0.5 * (c["d_lo"] + (c["d_hi"] - c["d_lo"]) * _rand(gen, n))
    if c["shuffled"]:
        p = torch.randperm(n, generator=gen, device=DEV)
        x, r = x[p], r[p]
    nn = [v * k + 1 for v in ne]
    u = 0.05 * (2.0 * _rand(gen, nn[0] * nn[1] * nn[2], 3) - 1.0)
    u[:, 2] += 1.0
    zp = torch.tensor(_GLL[kp], device=DEV, dtype=F64)
    pz = (torch.arange(ne[2], device=DEV)[:, None] + zp[None, :-1]).reshape(-1)
    pz = torch.cat([pz, torch.full((1,), float(ne[2]), device=DEV, dtype=F64)]) * c["h"]
    grad_p = c["phi"] * (RHO_P - RHO_F) * G
    p = (grad_p * (L[2] - pz)).repeat_interleave((ne[0] * kp + 1) * (ne[1] * kp + 1))
    u_p = 0.1 * _rand(gen, n, 3) - 0.05
    return {"x": x.contiguous(), "r": r.contiguous(), "u_p": u_p, "u": u, "p": p}


def _params(c):
    mixed = c["precision"] == "mixed"
    d = 0.5 * (c["d_lo"] + c["d_hi"])
    return cf.make_params(rho_f=RHO_F, mu_f=MU_F, g=(0.0, 0.0, -G), qcm_radius=_radius(c),
                          l2_smoothing=4.0 * d * d, drag_model=c["drag"],
                          vans_model=c["model"], shear_force=c["shear"],
                          fluid_drag=c["fluid_drag"], qcm_conserve=c["conserve"],
                          precision=1 if mixed else 0, cg_rtol=1e-12 if mixed else 1e-13,
                          max_radius=0.5 * c["d_hi"])


class _Results:
    """The results of one or more beds in one buffer: the projected void
    fractions first (cleared in one go), then the forces and the sources."""

    def __init__(self, beds):
        sizes = []
        for c in beds:
            ne, _ = _geometry(c)
            sizes.append(math.prod(v * c["k"] + 1 for v in ne))
        self.n_eps = sum(sizes)
        for c in beds:
            ne, _ = _geometry(c)
            e = math.prod(ne)
            sizes += [3 * c["n"], 3 * e] + ([3 * e * (c["k"] + 1) ** 3] if c["fluid_drag"] else [])
        self.sizes = sizes
        self.buf = torch.zeros(sum(sizes), device=DEV, dtype=F64)
        self.eps_all = self.buf[:self.n_eps]
        parts = self.buf.split(sizes)
        self.eps = parts[:len(beds)]
        rest, self.f, self.F_e, self.F_q = iter(parts[len(beds):]), [], [], []
        for c in beds:
            self.f.append(next(rest))
            self.F_e.append(next(rest))
            self.F_q.append(next(rest) if c["fluid_drag"] else None)

    def outputs(self, mixed):
        return list((self.buf.float() if mixed else self.buf).split(self.sizes))


class _Batch:
    """A batch handle and what its beds point at; freed with the state."""

    def __init__(self, n_beds):
        self.h = cf.cfdem_batch_create(n_beds, 0, torch.cuda.current_stream().cuda_stream)

    def __del__(self):
        cf.cfdem_batch_destroy(self.h)


class _Owner:
    """A handle without a destructor of its own, closed with the state."""

    def __init__(self, obj):
        self.obj = obj

    def __del__(self):
        self.obj.close()


def _grad_seed(c):
    """dJ/df_D of the loss: the drag along z."""
    g = torch.zeros(c["n"], 3, device=DEV, dtype=F64)
    g[:, 2] = 1.0
    return g


def _dem_inputs(case, gen):
    """A bed of spheres on an FCC lattice, a little over half of the
    neighbours in contact with small overlaps, on the floor of an open box."""
    n, d, m = case["n"], case["d"], case["side"]
    x = _lattice(n, d, m, m) + 2e-3 * d * (_rand(gen, n, 3) - 0.5)
    r = 0.5 * d * (0.985 + 0.025 * _rand(gen, n))
    if case["shuffled"]:
        p = torch.randperm(n, generator=gen, device=DEV)
        x, r = x[p], r[p]
    a = d * math.sqrt(2.0)
    lo = [0.25 * a - 0.503 * d] * 3
    hi = [lo[0] + a * (m - 0.5) + 1.006 * d] * 2
    layers = -(-n // (2 * m * m))
    hi.append(lo[2] + 1.5 * (0.5 * a * layers + d))
    v = 0.1 * _rand(gen, n, 3) - 0.05
    w = 2.0 * _rand(gen, n, 3) - 1.0
    mass = RHO_P * 4.0 / 3.0 * math.pi * r ** 3
    f = 0.1 * G * mass[:, None] * (2.0 * _rand(gen, n, 3) - 1.0)
    f[:, 2] += 0.5 * G * mass
    return {"x": x.contiguous(), "r": r.contiguous(), "v": v, "w": w, "f": f, "lo": lo, "hi": hi}


#: contact parameters of particles and walls (glass beads, softened as is usual)
_CONTACT = {"youngs": 1e7, "poisson": 0.3, "restitution": 0.9, "friction": 0.3,
            "rolling_friction": 0.01}


def _mapped_inputs(case, gen):
    """Particles inside the elements of a subdivided cylinder, and a velocity field."""
    mesh = synth.make_cylinder_mesh(0.05, 0.2, case["n_core"], case["n_ring"], case["n_z"],
                                    case["k"])
    conn = torch.as_tensor(mesh["conn"], device=DEV, dtype=torch.int64)
    nodes = torch.as_tensor(mesh["nodes"], device=DEV, dtype=F64)
    n = case["n"]
    elem = torch.randint(conn.shape[0], (n,), generator=gen, device=DEV)
    xi = 0.02 + 0.96 * _rand(gen, n, 3)
    x = _on_nodes(case["k"], conn, nodes, elem, xi)
    field = 2.0 * _rand(gen, nodes.shape[0], case["ncomp"]) - 1.0
    return mesh, conn, nodes, elem, xi, x.contiguous(), field


def prepare(case, seed):
    gen = _gen(seed)
    path = case["path"]
    if path == "dem":
        s = _dem_inputs(case, gen)
        s["vw"] = torch.stack([s.pop("v"), s.pop("w")])
        wall = {"wall_" + k: v for k, v in _CONTACT.items() if k != "youngs"}
        s["own"] = _Owner(cf.Dem(dict(_CONTACT, **wall, wall_youngs=1e7, rho_p=RHO_P,
                                      g=(0.0, 0.0, -G), lo=s["lo"], hi=s["hi"],
                                      max_radius=0.505 * case["d"], capacity=24,
                                      precision=int(case["precision"] == "mixed"))))
        return {"case": case, **s}
    if path == "mapped":
        mesh, _, _, _, _, x, field = _mapped_inputs(case, gen)
        n = case["n"]
        return {"case": case, "x": x, "field": field,
                "own": _Owner(cf.MappedMesh(case["k"], mesh["conn"], mesh["nodes"])),
                "elem": torch.empty(n, device=DEV, dtype=torch.int32),
                "xi": torch.empty(n, 3, device=DEV, dtype=F64),
                "out": torch.empty(n, case["ncomp"], device=DEV, dtype=F64)}
    beds = _ensemble_beds(case) if path == "ensemble" else [case]
    ins = [_inputs(c, gen) for c in beds]
    s = {"case": case, "in": ins}
    if path == "grad" and case["precision"] == "mixed":
        ne, L = _geometry(case)
        s["ctx"] = cf.Context((0.0, 0.0, 0.0), L, ne, case["k"], _params(case))
        ins[0]["x"].requires_grad_(True)
        ins[0]["u"].requires_grad_(True)
        return s
    s["res"] = res = _Results(beds)
    if path in ("step", "grad"):
        ne, L = _geometry(case)
        s["ctx"] = cf.Context((0.0, 0.0, 0.0), L, ne, case["k"], _params(case))
        if path == "grad":
            s["g_fd"] = _grad_seed(case)
            s["fd"], s["dx"] = torch.empty_like(ins[0]["x"]), torch.empty_like(ins[0]["x"])
            s["du"], s["Me"] = torch.empty_like(ins[0]["u"]), torch.empty_like(res.eps[0])
        return s
    s["batch"] = b = _Batch(len(beds))
    s["io"] = []
    for i, (c, w) in enumerate(zip(beds, ins)):
        ne, L = _geometry(c)
        bed = cf.cfdem_batch_bed(b.h, i)
        cf.cfdem_set_mesh(bed, (0.0, 0.0, 0.0), L, ne, c["k"])
        cf.cfdem_set_params(bed, _params(c))
        host = None
        if path == "host":
            s["host"] = host = {"x": w["x"], "r": w["r"], "u_p": w["u_p"], "u_nodal": w["u"],
                                "p_nodal": w["p"], "f": res.f[i], "F_elem": res.F_e[i]}
            for key in host:
                host[key] = host[key].cpu().pin_memory()
        s["io"].append(cf.bed_io(c["n"], w["x"], w["r"], w["u_p"], w["u"], w["p"], res.eps[i],
                                 res.f[i], None, res.F_e[i], res.F_q[i], host))
    return s


# ------------------------------------------------------------------ one pass

def run(s):
    case = s["case"]
    path, mixed = case["path"], case.get("precision") == "mixed"
    if path == "dem":
        s["own"].obj.step(s["x"], s["vw"][0], s["vw"][1], s["r"], s["f"], DT, NSUB)
        vw = s["vw"].float() if mixed else s["vw"]
        return {"x": s["x"], "v": vw[0], "w": vw[1]}
    if path == "mapped":
        m, n = s["own"].obj, case["n"]
        m.locate(n, s["x"], s["elem"], s["xi"])
        m.interpolate(n, s["elem"], s["xi"], case["ncomp"], s["field"], s["out"])
        return {"elem": s["elem"], "xi": s["xi"], "u": s["out"]}
    if path == "grad" and mixed:
        w = s["in"][0]
        w["x"].grad = w["u"].grad = None
        f, fd, eps, F_e = ag.coupling_step(s["ctx"], w["x"], w["r"], w["u_p"], w["u"], w["p"])
        (fd[:, 2].sum() + ag.mass_norm(s["ctx"], eps)).backward()
        return [t.detach().float() for t in (eps, fd, w["x"].grad, w["u"].grad)]
    res = s["res"]
    res.eps_all.zero_()
    if path in ("step", "grad"):
        w, h, n = s["in"][0], s["ctx"].h, case["n"]
        if path == "step":
            cf.cfdem_coupling_step(h, n, w["x"], w["r"], w["u_p"], w["u"], w["p"], res.eps[0],
                                   res.f[0], None, res.F_e[0], res.F_q[0])
            return res.outputs(mixed)
        eps = res.eps[0]
        cf.cfdem_coupling_step(h, n, w["x"], w["r"], w["u_p"], w["u"], w["p"], eps, res.f[0],
                               s["fd"])
        cf.cfdem_mass_apply(h, eps, s["Me"])
        g_eps = s["Me"] / torch.sqrt(torch.dot(eps, s["Me"]))
        cf.cfdem_adjoint(h, n, w["x"], w["r"], w["u_p"], w["u"], w["p"], eps, None, s["g_fd"],
                         g_eps, s["dx"], s["du"])
        return [eps, s["fd"], s["dx"], s["du"]]
    if cf.cfdem_batch_coupling_step(s["batch"].h, s["io"]) != cf.OK:
        raise RuntimeError(cf.cfdem_batch_last_error(s["batch"].h))
    if path == "host":
        if cf.cfdem_batch_synchronize(s["batch"].h)[0] != cf.OK:
            raise RuntimeError("the step failed")
        return [res.eps[0], s["host"]["f"], s["host"]["F_elem"]]
    return res.outputs(mixed)


# ------------------------------------------------------------------ what a pass cannot do without

def _bed_work(c):
    ne, _ = _geometry(c)
    k, n, E = c["k"], c["n"], math.prod(ne)
    kp, nq = max(1, k - 1), (k + 1) ** 3
    nn = [v * k + 1 for v in ne]
    nodes, pnodes = math.prod(nn), math.prod(v * kp + 1 for v in ne)
    b = 8.0 * (7 * n + 3 * nodes + pnodes)                       # x, r, u_p, u, p
    b += 8.0 * (nodes + 3 * n + 3 * E + (3 * E * nq if c["fluid_drag"] else 0))
    if c["path"] == "grad":
        b += 8.0 * (3 * n + 3 * nodes)
    # lens volumes of the (Gauss point, particle) pairs within R + r: 8 to test, 25 to evaluate
    cut = _radius(c) + 0.25 * (c["d_lo"] + c["d_hi"])
    fl = 33.0 * n * nq * 4.0 / 3.0 * math.pi * (cut / c["h"]) ** 3
    fl += 2.0 * 3 * E * (k + 1) ** 4                             # right-hand side
    # a direct solve by fast diagonalisation: x and y there and back (by parity), z banded
    solve = nodes * (2.0 * (nn[0] + nn[1]) + 8.0 * k + 2.0)
    fl += solve
    fl += n * (8.0 * nq + 9.0 * 2 * (kp + 1) ** 3 + 120.0)       # interpolation and closure
    if c["path"] == "grad":
        fl += solve + 33.0 * n * nq * 4.0 / 3.0 * math.pi * (cut / c["h"]) ** 3 + n * 16.0 * nq
    return b, fl


def work(case):
    path = case["path"]
    if path == "dem":
        # state in and out, radii and f_ext in; per sub-step ~6 contacts of ~150 operations
        return {"bytes": 8.0 * 22 * case["n"], "flops": float(NSUB) * case["n"] * (6 * 150 + 40)}
    if path == "mapped":
        E = (case["n_core"] ** 2 + 4 * case["n_core"] * case["n_ring"]) * case["n_z"]
        nodes, nq = E * case["k"] ** 3, (case["k"] + 1) ** 3
        return {"bytes": case["n"] * (8.0 * (6 + case["ncomp"]) + 4)
                + nodes * 8.0 * (3 + case["ncomp"]) + 4.0 * E * nq,
                # four Newton steps on the map and its Jacobian, then the interpolation
                "flops": case["n"] * nq * (4 * 24.0 + 2.0 * case["ncomp"])}
    beds = _ensemble_beds(case) if path == "ensemble" else [case]
    got = [_bed_work(c) for c in beds]
    return {"bytes": sum(g[0] for g in got), "flops": sum(g[1] for g in got)}


# ------------------------------------------------------------------ the results in 64 bits

_GLL = {1: [0.0, 1.0], 2: [0.0, 0.5, 1.0],
        3: [0.0, 0.5 - 0.5 / math.sqrt(5.0), 0.5 + 0.5 / math.sqrt(5.0), 1.0]}


def _lagrange(k, t, deriv=0):
    """Values (or derivatives) of the Lagrange basis on the GLL nodes at t: [..., k + 1]."""
    z = _GLL[k]
    out = []
    for a in range(k + 1):
        c = np.poly([z[b] for b in range(k + 1) if b != a])
        c = c / np.polyval(c, z[a])
        for _ in range(deriv):
            c = np.polyder(c) if len(c) > 1 else np.zeros(1)
        v = torch.full_like(t, float(c[0]))
        for ci in c[1:]:
            v = v * t + float(ci)
        out.append(v)
    return torch.stack(out, dim=-1)


def _gauss(nq):
    s, w = np.polynomial.legendre.leggauss(nq)
    return (torch.tensor(0.5 * (s + 1.0), device=DEV), torch.tensor(0.5 * w, device=DEV))


def _on_nodes(k, conn, values, elem, xi):
    """The Q_k interpolant of nodal values on an unstructured mesh at (elem, xi)."""
    l = [_lagrange(k, xi[:, a]) for a in range(3)]
    out = []
    for i in range(0, xi.shape[0], 20_000):
        c = slice(i, i + 20_000)
        phi = (l[2][c][:, :, None, None] * l[1][c][:, None, :, None] * l[0][c][:, None, None, :])
        out.append((phi.reshape(phi.shape[0], -1, 1) * values[conn[elem[c]]]).sum(1))
    return torch.cat(out)


class _Exact:
    """One bed's coupling step and its gradients in plain torch, 64 bits."""

    def __init__(self, c, w):
        self.c, self.w = c, w
        self.ne, self.L = _geometry(c)
        self.k, self.h = c["k"], c["h"]
        self.kp = max(1, self.k - 1)
        self.nn = [v * self.k + 1 for v in self.ne]
        self.E, self.nq = math.prod(self.ne), self.k + 1
        self.R = _radius(c)
        self.VR = 4.0 / 3.0 * math.pi * self.R ** 3
        self.g, self.gw = _gauss(self.nq)
        d = 0.5 * (c["d_lo"] + c["d_hi"])
        self.L2 = 4.0 * d * d
        B = _lagrange(self.k, self.g)
        D = _lagrange(self.k, self.g, 1)
        self.B = B
        self.mass = torch.einsum("q,qa,qb->ab", self.gw, B, B) * self.h
        self.stiff = torch.einsum("q,qa,qb->ab", self.gw, D, D) / self.h
        self.eig = []
        for a in range(3):
            M, K = self._assemble(self.mass, a), self._assemble(self.stiff, a)
            C = torch.linalg.cholesky(M)
            S = torch.linalg.solve_triangular(C, K, upper=False)
            S = torch.linalg.solve_triangular(C, S.T.contiguous(), upper=False)
            lam, V = torch.linalg.eigh(0.5 * (S + S.T))
            self.eig.append((lam, torch.linalg.solve_triangular(C.T.contiguous(), V, upper=True),
                             M))
        x = w["x"].detach()
        self.ie = torch.stack([torch.clamp(torch.floor(x[:, a] / self.h), 0, self.ne[a] - 1)
                               for a in range(3)], dim=1).to(torch.int64)

    def _assemble(self, m, a):
        n, k = self.nn[a], self.k
        A = torch.zeros(n, n, device=DEV, dtype=F64)
        for e in range(self.ne[a]):
            A[e * k:e * k + k + 1, e * k:e * k + k + 1] += m
        return A

    def _pairs(self):
        """(particles, element, d [n, nq^3], x - x_q) block by block over the
        elements that an averaging sphere's reach covers."""
        x, r = self.w["x"].detach(), self.w["r"]
        reach = int(math.ceil((self.R + 0.5 * self.c["d_hi"]) / self.h)) + 1
        ne = torch.tensor(self.ne, device=DEV)
        for i in range(0, x.shape[0], 100_000):
            sl = slice(i, i + 100_000)
            xs, rs, ie = x[sl], r[sl], self.ie[sl]
            for oz in range(-reach, reach + 1):
                for oy in range(-reach, reach + 1):
                    for ox in range(-reach, reach + 1):
                        e = ie + torch.tensor([ox, oy, oz], device=DEV)
                        # the box of the element's Gauss points against the reach
                        lo = (e + self.g[0]) * self.h
                        hi = (e + self.g[-1]) * self.h
                        gap = torch.clamp(torch.maximum(lo - xs, xs - hi), min=0.0)
                        ok = ((e >= 0) & (e < ne)).all(1)
                        ok &= (gap * gap).sum(1) < (self.R + rs) ** 2
                        at = torch.nonzero(ok)[:, 0]
                        if at.numel() == 0:
                            continue
                        xa, ea = xs[at], e[at]
                        dd = [xa[:, a:a + 1] - (ea[:, a:a + 1] + self.g[None, :]) * self.h
                              for a in range(3)]
                        d2 = ((dd[2] ** 2)[:, :, None, None] + (dd[1] ** 2)[:, None, :, None]
                              + (dd[0] ** 2)[:, None, None, :])
                        el = ea[:, 0] + self.ne[0] * (ea[:, 1] + self.ne[1] * ea[:, 2])
                        yield i + at, el, rs[at], torch.sqrt(d2), dd

    def _lens(self, r, d):
        """Volume of a particle of radius r inside the averaging sphere at distance d."""
        R, r = self.R, r[:, None, None, None]
        V = (math.pi * (R + r - d) ** 2 * (d * d + 2.0 * d * (R + r) - 3.0 * (R - r) ** 2)
             / (12.0 * d.clamp(min=1e-300)))
        V = torch.where(d <= (R - r).abs(), 4.0 / 3.0 * math.pi * r.clamp(max=R) ** 3, V)
        return torch.where(d < R + r, V, torch.zeros_like(V))

    def void_fraction(self):
        n, Q = self.c["n"], self.nq ** 3
        scale = torch.ones(n, device=DEV, dtype=F64)
        w3 = (self.gw[:, None, None] * self.gw[:, None] * self.gw) * self.h ** 3
        if self.c["conserve"]:
            S = torch.zeros(n, device=DEV, dtype=F64)
            for at, _, r, d, _ in self._pairs():
                S.index_add_(0, at, (self._lens(r, d) * w3).sum((1, 2, 3)) / self.VR)
            V = 4.0 / 3.0 * math.pi * self.w["r"] ** 3
            scale = torch.where(S > 0, V / S.clamp(min=1e-300), scale)
        sums = torch.zeros(self.E, Q, device=DEV, dtype=F64)
        for at, el, r, d, _ in self._pairs():
            V = self._lens(r, d) * scale[at][:, None, None, None]
            sums.index_add_(0, el, V.reshape(-1, Q))
        return 1.0 - sums / self.VR

    def _element_sum(self, v):
        """Scatter of element-local nodal values [ez, ey, ex, c, b, a] to the nodes."""
        k = self.k
        out = torch.zeros(self.nn[2], self.nn[1], self.nn[0], device=DEV, dtype=F64)
        for c in range(k + 1):
            for b in range(k + 1):
                for a in range(k + 1):
                    out[c:c + k * self.ne[2]:k, b:b + k * self.ne[1]:k,
                        a:a + k * self.ne[0]:k] += v[:, :, :, c, b, a]
        return out

    def rhs(self, eps_q):
        v = eps_q.reshape(self.ne[2], self.ne[1], self.ne[0], self.nq, self.nq, self.nq)
        Bw = self.B * self.gw[:, None]
        for ax in (3, 4, 5):
            v = torch.movedim(torch.tensordot(v, Bw, dims=([ax], [0])), -1, ax)
        return self._element_sum(v) * self.h ** 3

    def solve(self, b):
        """(M + L^2 K)^-1 b through the generalised eigenvectors of each axis."""
        (lx, Vx, _), (ly, Vy, _), (lz, Vz, _) = self.eig
        t = torch.tensordot(b, Vx, ([2], [0]))
        t = torch.tensordot(t, Vy, ([1], [0]))
        t = torch.tensordot(t, Vz, ([0], [0]))          # [kx, ky, kz]
        den = 1.0 + self.L2 * (lx[:, None, None] + ly[None, :, None] + lz[None, None, :])
        t = t / den
        t = torch.tensordot(t, Vz, ([2], [1]))          # [kx, ky, z]
        t = torch.tensordot(t, Vy, ([1], [1]))          # [kx, z, y]
        return torch.tensordot(t, Vx, ([0], [1]))       # [z, y, x]

    def mass_apply(self, v):
        (_, _, Mx), (_, _, My), (_, _, Mz) = self.eig
        t = torch.tensordot(v, Mx, ([2], [0]))
        t = torch.tensordot(t, My, ([1], [0]))
        t = torch.tensordot(t, Mz, ([0], [0]))          # [x, y, z]
        return t.permute(2, 1, 0)

    def _nodes(self, ie, k):
        nn = [v * k + 1 for v in self.ne]
        o = torch.arange(k + 1, device=DEV)
        idx = [ie[:, a:a + 1] * k + o for a in range(3)]
        return (idx[0][:, None, None, :]
                + nn[0] * (idx[1][:, None, :, None] + nn[1] * idx[2][:, :, None, None]))

    def drag(self, eps, U, r):
        c = self.c
        speed = torch.sqrt((U * U).sum(1))
        d, e_p = 2.0 * r, 1.0 - eps
        Re = RHO_F * eps * speed * d / MU_F
        V = 4.0 / 3.0 * math.pi * r ** 3
        bell = torch.exp(-0.5 * (1.5 - torch.log10(Re)) ** 2)
        if c["drag"] in (DI_FELICE, RONG):
            cd = (0.63 * torch.sqrt(speed) + 4.8 * torch.sqrt(MU_F / (RHO_F * eps * d))) ** 2
            chi = (3.7 - 0.65 * bell if c["drag"] == DI_FELICE else
                   2.65 * (eps + 1.0) - (5.3 - 3.5 * eps) * eps ** 2 * bell)
            return 0.5 * RHO_F * cd * eps ** (2.0 - chi) * math.pi * r ** 2
        if c["drag"] == KOCH_HILL:
            s = e_p.clamp(min=1e-300)
            f0 = torch.where(e_p >= 0.4, 10.0 * e_p / eps ** 3,
                             (1.0 + 3.0 * torch.sqrt(s / 2.0) + 135.0 / 64.0 * s * torch.log(s)
                              + 16.14 * e_p)
                             / (1.0 + 0.681 * e_p - 8.48 * e_p ** 2 + 8.14 * e_p ** 3))
            f3 = 0.0673 + 0.212 * e_p + 0.0232 / eps ** 5
            return 18.0 * MU_F * eps ** 2 / d ** 2 * (f0 + 0.5 * f3 * Re) * V
        F = (10.0 * e_p / eps ** 2 + eps ** 2 * (1.0 + 1.5 * torch.sqrt(e_p))
             + 0.413 * Re / (24.0 * eps ** 2)
             * (1.0 / eps + 3.0 * e_p * eps + 8.4 * Re ** -0.343)
             / (1.0 + 10.0 ** (3.0 * e_p) * Re ** (-0.5 * (1.0 + 4.0 * e_p))))
        return 3.0 * math.pi * MU_F * d * eps * F

    def forces(self, x, u, eps_h, sl):
        """(f, f_D, drag coefficient, pressure and shear part) of the particles in sl."""
        c, w, k, kp, h = self.c, self.w, self.k, self.kp, self.h
        ie, x, r, u_p = self.ie[sl], x[sl], w["r"][sl], w["u_p"][sl]
        xi = x / h - ie
        l = [_lagrange(k, xi[:, a]) for a in range(3)]
        idx = self._nodes(ie, k)
        un = u[idx]

        def at(bz, by, bx, v):
            return torch.einsum("nc,nb,na,ncba...->n...", bz, by, bx, v)

        uf = at(l[2], l[1], l[0], un)
        eps = at(l[2], l[1], l[0], eps_h.reshape(-1)[idx])
        q = [_lagrange(kp, xi[:, a]) for a in range(3)]
        dq = [_lagrange(kp, xi[:, a], 1) / h for a in range(3)]
        pn = w["p"][self._nodes(ie, kp)]
        gp = torch.stack([at(q[2], q[1], dq[0], pn - pn[:, :, :, :1]),
                          at(q[2], dq[1], q[0], pn - pn[:, :, :1, :]),
                          at(dq[2], q[1], q[0], pn - pn[:, :1, :, :])], dim=1)
        V = 4.0 / 3.0 * math.pi * r ** 3
        beta = self.drag(torch.clamp(eps, 0.05, 1.0), uf - u_p, r)
        fd = beta[:, None] * (uf - u_p)
        other = -V[:, None] * gp
        if c["shear"]:
            dl = [_lagrange(k, xi[:, a], 1) / h for a in range(3)]
            d2 = [_lagrange(k, xi[:, a], 2) / h ** 2 for a in range(3)]
            lap = (at(l[2], l[1], d2[0], un) + at(l[2], d2[1], l[0], un)
                   + at(d2[2], l[1], l[0], un))
            xx, yy, zz = (at(l[2], l[1], d2[0], un[..., 0]), at(l[2], d2[1], l[0], un[..., 1]),
                          at(d2[2], l[1], l[0], un[..., 2]))
            xy = [at(l[2], dl[1], dl[0], un[..., j]) for j in (0, 1)]
            xz = [at(dl[2], l[1], dl[0], un[..., j]) for j in (0, 2)]
            yz = [at(dl[2], dl[1], l[0], un[..., j]) for j in (1, 2)]
            gdiv = torch.stack([xx + xy[1] + xz[1], xy[0] + yy + yz[1], xz[0] + yz[0] + zz],
                               dim=1)
            other = other - V[:, None] * MU_F * (lap + gdiv / 3.0)
        buoy = torch.zeros_like(fd)
        buoy[:, 2] = RHO_F * V * G
        return fd + other + buoy, fd, beta, other

    def step(self):
        c, w = self.c, self.w
        n, E, k = c["n"], self.E, self.k
        eps_h = self.solve(self.rhs(self.void_fraction()))
        f = torch.empty(n, 3, device=DEV, dtype=F64)
        el = self.ie[:, 0] + self.ne[0] * (self.ie[:, 1] + self.ne[1] * self.ie[:, 2])
        S = torch.zeros(E, 3, device=DEV, dtype=F64)
        beta_e, count = torch.zeros(E, device=DEV, dtype=F64), torch.zeros(E, device=DEV, dtype=F64)
        up_e = torch.zeros(E, 3, device=DEV, dtype=F64)
        for i in range(0, n, 50_000):
            sl = slice(i, i + 50_000)
            f[sl], fd, beta, other = self.forces(w["x"], w["u"], eps_h, sl)
            if not c["fluid_drag"]:
                S.index_add_(0, el[sl], fd)
            if c["model"]:
                S.index_add_(0, el[sl], other)
            beta_e.index_add_(0, el[sl], beta)
            count.index_add_(0, el[sl], torch.ones_like(beta))
            up_e.index_add_(0, el[sl], w["u_p"][sl])
        F_e = -S / self.h ** 3
        out = [eps_h.reshape(-1), f.reshape(-1)]
        if not c["fluid_drag"]:
            return out + [F_e.reshape(-1)]
        beta_e, up_e = beta_e / self.h ** 3, up_e / count.clamp(min=1.0)[:, None]
        e = torch.arange(E, device=DEV)
        ie = torch.stack([e % self.ne[0], e // self.ne[0] % self.ne[1],
                          e // (self.ne[0] * self.ne[1])], dim=1)
        uq = w["u"][self._nodes(ie, k)]                                  # [E, c, b, a, 3]
        for ax in (1, 2, 3):
            uq = torch.movedim(torch.tensordot(uq, self.B, dims=([ax], [1])), -1, ax)
        F_q = (F_e[:, None, None, None, :]
               - beta_e[:, None, None, None, None] * (uq - up_e[:, None, None, None, :]))
        F_e = torch.einsum("z,y,x,ezyxa->ea", self.gw, self.gw, self.gw, F_q)
        return out + [F_e.reshape(-1), F_q.reshape(-1)]

    def gradients(self):
        """eps_h, f_D and dJ/dx, dJ/du of J = sum_i f_D,i . e_z + ||eps_h||_M."""
        c, w = self.c, self.w
        n = c["n"]
        eps_h = self.solve(self.rhs(self.void_fraction()))
        Me = self.mass_apply(eps_h)
        g_eps = (Me / torch.sqrt((eps_h * Me).sum())).reshape(-1).clone()
        fd, dx = torch.empty(n, 3, device=DEV, dtype=F64), torch.empty(n, 3, device=DEV, dtype=F64)
        du = torch.zeros_like(w["u"])
        for i in range(0, n, 50_000):
            sl = slice(i, i + 50_000)
            x = w["x"].detach().clone().requires_grad_(True)
            u = w["u"].detach().clone().requires_grad_(True)
            e = eps_h.detach().reshape(-1).clone().requires_grad_(True)
            with torch.enable_grad():
                _, d, _, _ = self.forces(x, u, e, sl)
                gx, gu, ge = torch.autograd.grad(d[:, 2].sum(), (x, u, e))
            fd[sl], dx[sl] = d.detach(), gx[sl]
            du += gu
            g_eps += ge
        lam = self.solve(g_eps.reshape(eps_h.shape))
        # through the quadrature: dJ/deps_q = w_q |J| lam(x_q)
        e = torch.arange(self.E, device=DEV)
        ie = torch.stack([e % self.ne[0], e // self.ne[0] % self.ne[1],
                          e // (self.ne[0] * self.ne[1])], dim=1)
        lq = lam.reshape(-1)[self._nodes(ie, self.k)]
        for ax in (1, 2, 3):
            lq = torch.movedim(torch.tensordot(lq, self.B, dims=([ax], [1])), -1, ax)
        gq = lq * (self.gw[:, None, None] * self.gw[:, None] * self.gw) * self.h ** 3
        for at, el, r, d, dd in self._pairs():
            R, r = self.R, r[:, None, None, None]
            a2 = R * R - ((d * d - r * r + R * R) / (2.0 * d)) ** 2
            on = (d < R + r) & (d > (R - r).abs())
            s = torch.where(on, gq[el] * math.pi * a2 / self.VR / d, torch.zeros_like(d))
            dx.index_add_(0, at, torch.stack([(s * dd[0][:, None, None, :]).sum((1, 2, 3)),
                                              (s * dd[1][:, None, :, None]).sum((1, 2, 3)),
                                              (s * dd[2][:, :, None, None]).sum((1, 2, 3))], 1))
        return eps_h.reshape(-1), fd, dx, du


def _cross(a, b):
    return torch.linalg.cross(a, b)


def _contact(nrm, dn, vrel, wrel, r, me, Re, hist, dt):
    """Force and torque on the first partner of each contact, and its new tangential
    displacement (particles and walls have the same material)."""
    p = _CONTACT
    Ye = 1.0 / (2.0 * (1.0 - p["poisson"] ** 2) / p["youngs"])
    Ge = 1.0 / (4.0 * (2.0 - p["poisson"]) * (1.0 + p["poisson"]) / p["youngs"])
    le = math.log(p["restitution"])
    damp = -2.0 * math.sqrt(5.0 / 6.0) * le / math.sqrt(le * le + math.pi ** 2)
    on = dn > 0
    sq = torch.sqrt(Re * dn.clamp(min=0.0))
    kn, kt = 4.0 / 3.0 * Ye * sq, 8.0 * Ge * sq
    en, et = damp * torch.sqrt(2.0 * Ye * sq * me), damp * torch.sqrt(8.0 * Ge * sq * me)
    vrn = (vrel * nrm).sum(1, keepdim=True) * nrm
    vrt = vrel - vrn
    hist = hist - (hist * nrm).sum(1, keepdim=True) * nrm + vrt * dt
    fn = -(kn * dn)[:, None] * nrm - en[:, None] * vrn
    ft = -kt[:, None] * hist - et[:, None] * vrt
    fnm, ftm = fn.norm(dim=1), ft.norm(dim=1)
    slip = ftm > p["friction"] * fnm
    ft = torch.where(slip[:, None], ft * (p["friction"] * fnm / ftm.clamp(min=1e-300))[:, None], ft)
    hist = torch.where(slip[:, None], -(ft + et[:, None] * vrt) / kt.clamp(min=1e-300)[:, None],
                       hist)
    wm = wrel.norm(dim=1)
    T = _cross(r[:, None] * nrm, ft)
    T = T - (p["rolling_friction"] * Re * fnm / wm.clamp(min=1e-300))[:, None] * wrel
    z = torch.zeros_like(fn)
    o = on[:, None]
    return torch.where(o, fn + ft, z), torch.where(o, T, z), torch.where(o, hist, z)


def _exact_dem(case, s):
    x, v, w, r, f_ext = (s[k].clone() for k in ("x", "v", "w", "r", "f"))
    n = x.shape[0]
    near = []
    for i in range(0, n, 2000):          # pairs that can touch within the pass
        c = torch.cdist(x[i:i + 2000], x)
        c = torch.nonzero(c < (r[i:i + 2000, None] + r[None, :]) + 0.02 * case["d"])
        near.append(c + torch.tensor([i, 0], device=DEV))
    near = torch.cat(near)
    I, J = near[near[:, 0] != near[:, 1]].T
    m = RHO_P * 4.0 / 3.0 * math.pi * r ** 3
    inertia = 0.4 * m * r * r
    me, Re = 1.0 / (1.0 / m[I] + 1.0 / m[J]), 1.0 / (1.0 / r[I] + 1.0 / r[J])
    hist = torch.zeros(I.shape[0], 3, device=DEV, dtype=F64)
    whist = [torch.zeros(n, 3, device=DEV, dtype=F64) for _ in range(6)]
    grav = torch.tensor([0.0, 0.0, -G], device=DEV, dtype=F64)

    def accelerations(dt):
        nonlocal hist
        d = x[J] - x[I]
        dist = d.norm(dim=1)
        nrm = d / dist[:, None]
        vrel = v[I] - v[J] + _cross(r[I, None] * w[I] + r[J, None] * w[J], nrm)
        fc, tc, hist = _contact(nrm, r[I] + r[J] - dist, vrel, w[I] - w[J], r[I], me, Re, hist, dt)
        F, T = torch.zeros_like(x), torch.zeros_like(x)
        F.index_add_(0, I, fc)
        T.index_add_(0, I, tc)
        for wl in range(6):
            ax, nrm = wl // 2, torch.zeros_like(x)
            nrm[:, ax] = 1.0 if wl % 2 else -1.0
            dn = r - ((s["hi"][ax] - x[:, ax]) if wl % 2 else (x[:, ax] - s["lo"][ax]))
            fc, tc, whist[wl] = _contact(nrm, dn, v + _cross(r[:, None] * w, nrm), w, r, m, r,
                                         whist[wl], dt)
            F, T = F + fc, T + tc
        return (F + m[:, None] * grav + f_ext) / m[:, None], T / inertia[:, None]

    a, al = accelerations(0.0)
    for _ in range(NSUB):
        v, w = v + 0.5 * DT * a, w + 0.5 * DT * al
        x = x + DT * v
        a, al = accelerations(DT)
        v, w = v + 0.5 * DT * a, w + 0.5 * DT * al
    return {"x": x, "v": v, "w": w}


def exact(case, seed):
    gen = _gen(seed)
    path = case["path"]
    if path == "dem":
        return _exact_dem(case, _dem_inputs(case, gen))
    if path == "mapped":
        _, conn, _, elem, xi, _, field = _mapped_inputs(case, gen)
        return {"elem": elem.to(torch.int32), "xi": xi,
                "u": _on_nodes(case["k"], conn, field, elem, xi)}
    if path == "grad":
        return list(_Exact(case, _inputs(case, gen)).gradients())
    beds = _ensemble_beds(case) if path == "ensemble" else [case]
    ins = [_inputs(c, gen) for c in beds]
    got = [_Exact(c, w).step() for c, w in zip(beds, ins)]
    if path == "host":
        return got[0][:3]
    return [g[0] for g in got] + [t for g in got for t in g[1:]]
