"""Performance cases: the work a program has this library do, through its public entry points.

A case is one of four kinds.

  step      a time-stepping call on one bed, as a solver run makes it: the initial PDFs (rest, or
            a developed field), K steps, the mass and flux of the last one, the fields rho and u,
            and the PDFs.
  assemble  the sparse representation of a new geometry from its voxel flags: cells, adjacency,
            inverse, as a program that runs many geometries pays for each of them.
  adjoint   one gradient: the mean flux after K steps and its gradients with respect to the body
            force and the damping field, as each iteration of an optimisation takes it.
  batch     many beds of uneven size stepped together, each with its own force.

The geometries are the library's seeded packed beds.  ``exact`` restates the method in plain
FP64 torch (links, collision, autograd) and shares no code with the library.
"""
import dataclasses
import math
import random

import numpy as np
import torch

from paper_1111_1129_gb300 import (Adjoint, BatchedState, LBMFlux, LBMState, SparseLattice,
                                   deviation_bound, inputs, omega_minus, shifted_scale_exp)

FORCE = 1e-6
STORAGE = {"f64": 8, "f64x": 8, "f32": 4, "f32s": 4, "f16s": 2, "bf16s": 2}
FLOPS = 200          # floating-point operations of one TRT update
FLOPS_REVERSE = 400  # and of one reverse step


def _step(name, box, axis, radius, order, form, steps, damped=False, start="rest", block=8,
          omega=1.25):
    return {"name": name, "kind": "step", "nx": box[0], "ny": box[1], "nz": box[2], "axis": axis,
            "radius": radius, "order": order, "block": block, "form": form, "steps": steps,
            "damped": damped, "start": start, "omega": omega}


def listed():
    small, medium, large = (32, 32, 64), (256, 128, 128), (1024, 256, 256)
    return [
        # one step and its sums on a small bed: a loop that looks at the flow after every step
        _step("monitor_small_f64x", small, 2, 4.0, "lex", "f64x", 1, start="flow"),
        # a small bed run towards steady state in one call
        _step("run_small_f32s", small, 2, 4.0, "lex", "f32s", 1000),
        # the default form, IEEE FP64 arithmetic, as a checking run uses it
        _step("run_medium_f64", medium, 0, 8.0, "lex", "f64", 10),
        # odd box along a space-filling curve, with a Brinkman field, resumed from a developed flow
        _step("resume_odd_f32s_damped", (251, 127, 125), 0, 8.0, "hilbert", "f32s", 50,
              damped=True, start="flow"),
        # the benchmark's bed in its default form: FP64 storage, lexicographic order
        _step("run_large_f64x", large, 0, 8.0, "lex", "f64x", 30),
        # the same bed in the most compact storage, blocked order
        _step("run_large_f16s", large, 0, 8.0, "blocked", "f16s", 50),
        # a bed between the two sizes, FP32 storage, a relaxation rate of its own
        _step("run_wide_f32s", (500, 230, 210), 0, 8.0, "lex", "f32s", 40, omega=1.6),
        # a new large geometry in the benchmark's order; a medium one along the Hilbert curve
        {"name": "assemble_large_lex", "kind": "assemble", "nx": 1024, "ny": 256, "nz": 256,
         "axis": 0, "radius": 8.0, "order": "lex", "block": 8},
        {"name": "assemble_medium_hilbert", "kind": "assemble", "nx": 256, "ny": 128, "nz": 128,
         "axis": 0, "radius": 8.0, "order": "hilbert", "block": 8},
        # gradients of the damped 128^3 bed in FP32, and of a smaller odd bed in FP64 storage
        {"name": "gradient_cube_f32s", "kind": "adjoint", "nx": 128, "ny": 128, "nz": 128,
         "axis": 2, "radius": 6.0, "order": "lex", "block": 8, "form": "f32s", "steps": 200,
         "damped": True, "omega": 1.25},
        {"name": "gradient_odd_f64x", "kind": "adjoint", "nx": 91, "ny": 83, "nz": 117, "axis": 2,
         "radius": 5.0, "order": "morton1", "block": 8, "form": "f64x", "steps": 60,
         "damped": True, "omega": 1.25},
        # many beds of uneven size, the library's batch workload with fewer beds
        {"name": "batch_beds_f32s", "kind": "batch", "beds": 40, "form": "f32s", "steps": 100,
         "omega": 1.25},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["assemble", "adjoint", "adjoint", "batch"])
    omega = rng.choice([1.25, 1.25, 1.0, 1.5, round(rng.uniform(0.7, 1.9), 3)])
    if kind == "batch":
        return {"kind": kind, "beds": int(_log(rng, 2, 48)), "omega": omega,
                "form": rng.choice(["f32s", "f32s", "f16s", "bf16s", "f32"]),
                "steps": int(_log(rng, 2, 300))}
    order = rng.choice(["lex", "lex", "blocked", "blocked", "morton1", "morton2", "hilbert"])
    axis = rng.randrange(3)
    cells = _log(rng, 2.5e4, {"step": 2.4e7, "assemble": 3e7, "adjoint": 1.5e6}[kind])
    # a tube: one long axis, a square or slightly flattened section
    long = rng.uniform(1.0, 5.0)
    flat = rng.uniform(0.8, 1.25)
    d = (cells / long) ** (1.0 / 3.0)
    dims = [0, 0, 0]
    dims[axis] = max(16, int(d * long))
    dims[(axis + 1) % 3] = max(16, int(d * math.sqrt(flat)))
    dims[(axis + 2) % 3] = max(16, int(d / math.sqrt(flat)))
    case = {"kind": kind, "nx": dims[0], "ny": dims[1], "nz": dims[2], "axis": axis,
            "radius": round(rng.uniform(3.0, 8.0), 2), "order": order,
            "block": rng.choice([4, 8, 16, 32])}
    if kind == "assemble":
        return case
    n = dims[0] * dims[1] * dims[2]
    case["form"] = rng.choice(["f64", "f64x", "f64x", "f32", "f32s", "f32s", "f16s", "f16s",
                               "bf16s"] if kind == "step" else ["f32s", "f32s", "f64x", "f64"])
    case["omega"] = omega
    if kind == "adjoint":
        case["steps"] = int(_log(rng, 4, max(8, min(400, (6e7 if case["form"] == "f64" else 1.4e8) / n))))
        case["damped"] = rng.random() < 0.6
        return case
    case["steps"] = int(_log(rng, 1, max(4, min(1000, (2.5e8 if case["form"] == "f64" else 4e8) / n))))
    case["damped"] = rng.random() < 0.25
    case["start"] = rng.choice(["rest", "flow"])
    return case


# ---- inputs -------------------------------------------------------------------

C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
              (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)])
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
OPP = [0] + [q + 1 if q % 2 else q - 1 for q in range(1, 19)]


def _turned(bed, seed):
    """The bed moved along its periodic axis and mirrored, by the seed: another geometry with
    the same number of fluid cells."""
    rng = random.Random(seed)
    at = 2 - bed.axis
    flags = np.roll(bed.flags, rng.randrange(bed.flags.shape[at]), at)
    flags = np.flip(flags, [a for a in range(3) if rng.random() < 0.5])
    return dataclasses.replace(bed, flags=np.ascontiguousarray(flags))


def _bed(case, seed):
    dims = (case["nx"], case["ny"], case["nz"])
    across = [d for a, d in enumerate(dims) if a != case["axis"]]
    return _turned(inputs.packed_bed(dims, case["axis"], min(across) - 2.0, case["radius"], 0.40,
                                     0, max_rejects=2000), seed)


def _flags(bed):
    return torch.from_numpy(bed.flags).cuda()


def _force(case, seed):
    size = FORCE * random.Random(seed + 17).uniform(0.5, 1.0)
    return tuple(size if a == case["axis"] else 0.0 for a in range(3))


def _scale_exp(case):
    if case["form"] not in ("f16s", "bf16s"):
        return 0
    across = [d for a, d in enumerate((case["nx"], case["ny"], case["nz"])) if a != case["axis"]]
    return shifted_scale_exp(deviation_bound(FORCE, 0.5 * min(across) - 1.0, case["omega"]))


def _uniform(n, seed, lo, hi):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return torch.rand(n, generator=g, dtype=torch.float64, device="cuda") * (hi - lo) + lo


def _flow_deviation(n, case, seed):
    """Deviations f - w of a developed flow of the case's scale: a velocity along the axis, a
    little across, density and non-equilibrium parts, [19, n]."""
    across = [d for a, d in enumerate((case["nx"], case["ny"], case["nz"])) if a != case["axis"]]
    nu = (1.0 / case["omega"] - 0.5) / 3.0
    top = min(1e-2, 0.2 * FORCE * (0.5 * min(across)) ** 2 / (4.0 * nu))
    u = [_uniform(n, 3 * seed + a, -0.1 * top, top if a == case["axis"] else 0.1 * top)
         for a in range(3)]
    rho = _uniform(n, 3 * seed + 5, -0.05 * top, 0.05 * top)
    usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    h = torch.empty((19, n), dtype=torch.float64, device="cuda")
    for q in range(19):
        cu = sum(float(C[q][a]) * u[a] for a in range(3))
        noise = _uniform(n, 7919 * seed + q, -0.02 * top, 0.02 * top)
        h[q] = float(W[q]) * (rho + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq + noise)
    return h


def _alpha(n, seed):
    return _uniform(n, seed + 101, 0.0, 0.05)


def _lattice(case, bed):
    return SparseLattice(_flags(bed), case["order"], (case["block"],) * 3, bed.periodic)


def _batch(case, seed):
    sides, radii, _ = inputs.batch_params(case["beds"], 0)
    forces = inputs.batch_params(case["beds"], seed)[2]
    beds = [_turned(inputs.packed_bed((int(s),) * 3, 2, float(s - 2), float(r), 0.0, b,
                                      max_rejects=2000), seed + b)
            for b, (s, r) in enumerate(zip(sides, radii))]
    return beds, [(0.0, 0.0, float(f)) for f in forces]


def _batch_scale_exp(case):
    if case["form"] not in ("f16s", "bf16s"):
        return 0
    return shifted_scale_exp(deviation_bound(1e-5, 47.0, case["omega"]))


def prepare(case, seed):
    state = {"kind": case["kind"], "case": case}
    if case["kind"] == "batch":
        beds, forces = _batch(case, seed)
        lats = [SparseLattice(_flags(b), "lex", periodic=b.periodic) for b in beds]
        state["batch"] = BatchedState(lats, case["form"], _batch_scale_exp(case))
        state["forces"] = forces
        return state
    bed = _bed(case, seed)
    if case["kind"] == "assemble":
        state["flags"], state["periodic"] = _flags(bed), bed.periodic
        return state
    lat = _lattice(case, bed)
    st = LBMState(lat, case["form"], _scale_exp(case))
    state["lattice"], state["state"], state["body_force"] = lat, st, _force(case, seed)
    if case["kind"] == "adjoint":
        state["adjoint"] = Adjoint(st, case["steps"])
        state["force"] = torch.tensor(state["body_force"], dtype=torch.float64,
                                      requires_grad=True)
        state["alpha"] = (_alpha(lat.n, seed).requires_grad_() if case["damped"] else None)
        return state
    if case["damped"]:
        st.set_damping(_alpha(lat.n, seed))
    if case["start"] == "flow":
        w = torch.from_numpy(W).cuda()[:, None]
        state["f0"] = _flow_deviation(lat.n, case, seed) + w
    return state


# ---- one pass -------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = state["kind"]
    if kind == "assemble":
        lat = SparseLattice(state["flags"], case["order"], (case["block"],) * 3,
                            state["periodic"])
        out = {"cells": lat.cells(), "adjacency": lat.adjacency(), "inverse": lat.inverse()}
        lat.close()
        return out
    wp = case["omega"]
    wm = omega_minus(wp)
    if kind == "batch":
        b = state["batch"]
        b.reset()
        b.step(case["steps"], wp, wm, state["forces"])
        mass, flux = b.reduce_flux(2)
        return {"mass": np.array(mass), "flux": np.array(flux), "f": b.get_pdfs()}
    if kind == "adjoint":
        force, alpha = state["force"], state["alpha"]
        force.grad = None
        if alpha is not None:
            alpha.grad = None
        J = LBMFlux.apply(force, alpha, state["adjoint"], wp, wm, case["axis"])
        J.backward()
        out = {"J": J.detach(), "force": force.grad}
        if alpha is not None:
            out["alpha"] = alpha.grad
        return out
    st = state["state"]
    if case["start"] == "flow":
        st.set_pdfs(state["f0"])
    else:
        st.reset()
    st.step(case["steps"], wp, wm, state["body_force"])
    mass, flux = st.reduce_flux(case["axis"])
    rho, u = st.moments()
    return {"mass": mass, "flux": flux, "rho": rho, "u": u, "f": st.get_pdfs()}


# ---- what a pass cannot do without --------------------------------------------------

def _fluid(case):
    """Fluid cells of a bed, from its box: a tube of solid fraction ~0.34."""
    return 0.5 * case["nx"] * case["ny"] * case["nz"]


def work(case):
    if case["kind"] == "assemble":
        box = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": box * (1 + 4) + _fluid(case) * (4 + 72), "flops": 0.0}
    if case["kind"] == "batch":
        n = case["beds"] * 0.45 * 65.0 ** 3
        return {"bytes": n * (72 + 152), "flops": n * case["steps"] * FLOPS}
    n = _fluid(case)
    if case["kind"] == "adjoint":
        # links and initial PDFs in, the damping field and its gradient
        return {"bytes": n * (72 + 19 * STORAGE[case["form"]] + (16 if case["damped"] else 0)),
                "flops": n * case["steps"] * (FLOPS + FLOPS_REVERSE)}
    # links (and the given PDFs and damping) in; rho, u and the PDFs out
    read = 72 + (152 if case["start"] == "flow" else 0) + (8 if case["damped"] else 0)
    return {"bytes": n * (read + 32 + 152), "flops": n * case["steps"] * FLOPS}


# ---- the same in plain FP64 torch ---------------------------------------------------

def _spread(v, step):
    """Bits of v moved `step` apart."""
    out = torch.zeros_like(v)
    for b in range(11):
        out |= ((v >> b) & 1) << (step * b)
    return out


def _hilbert(x, y, z, bits):
    """Hilbert curve key of each cell (Skilling 2004)."""
    X = [x.clone(), y.clone(), z.clone()]
    q = 1 << (bits - 1)
    while q > 1:
        p = q - 1
        for i in range(3):
            hit = (X[i] & q) != 0
            t = (X[0] ^ X[i]) & p
            X[0] = torch.where(hit, X[0] ^ p, X[0] ^ t)
            if i:
                X[i] = torch.where(hit, X[i], X[i] ^ t)
        q >>= 1
    X[1] ^= X[0]
    X[2] ^= X[1]
    t = torch.zeros_like(x)
    q = 1 << (bits - 1)
    while q > 1:
        t = torch.where((X[2] & q) != 0, t ^ (q - 1), t)
        q >>= 1
    X = [v ^ t for v in X]
    key = torch.zeros_like(x)
    for lvl in range(bits - 1, -1, -1):
        for v in X:
            key = (key << 1) | ((v >> lvl) & 1)
    return key


def _order_key(case, x, y, z):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["order"] == "lex":
        return x + nx * (y + ny * z)
    if case["order"] == "blocked":
        b = case["block"]
        nbx, nby = -(-nx // b), -(-ny // b)
        blk = x // b + nbx * (y // b + nby * (z // b))
        return blk * b ** 3 + x % b + b * (y % b + b * (z % b))
    if case["order"] == "morton1":
        return _spread(x, 3) | (_spread(y, 3) << 1) | (_spread(z, 3) << 2)
    if case["order"] == "morton2":
        key = torch.zeros_like(x)
        for g in range(6):
            for a, v in enumerate((x, y, z)):
                key |= ((v >> (2 * g)) & 3) << (6 * g + 2 * a)
        return key
    bits = max(1, (max(nx, ny, nz) - 1).bit_length())
    return _hilbert(x, y, z, bits)


def _links(case, bed):
    """Source slot of each pulled PDF, [18 n] flat, in the case's cell order."""
    flags = _flags(bed)
    nz, ny, nx = flags.shape
    cell = torch.nonzero(flags.reshape(-1) == 0).reshape(-1)
    x, y, z = cell % nx, (cell // nx) % ny, cell // (nx * ny)
    order = torch.argsort(_order_key(case, x, y, z))
    x, y, z, cell = x[order], y[order], z[order], cell[order]
    n = cell.numel()
    rank = torch.full((nx * ny * nz,), -1, dtype=torch.int64, device="cuda")
    rank[cell] = torch.arange(n, device="cuda")
    here = torch.arange(n, device="cuda")
    rows = []
    for q in range(1, 19):
        s = [v - int(C[q][a]) for a, v in enumerate((x, y, z))]
        inside = torch.ones(n, dtype=torch.bool, device="cuda")
        for a, d in enumerate((nx, ny, nz)):
            if (bed.periodic >> a) & 1:
                s[a] = s[a] % d
            else:
                inside &= (s[a] >= 0) & (s[a] < d)
                s[a] = s[a].clamp(0, d - 1)
        m = rank[s[0] + nx * (s[1] + ny * s[2])]
        rows.append(torch.where(inside & (m >= 0), q * n + m, OPP[q] * n + here))
    return torch.cat(rows), n


class _Stream(torch.autograd.Function):
    """g = f pulled through the links; the links permute the slots, so the transpose is the
    inverse permutation."""

    @staticmethod
    def forward(ctx, f, src, inv):
        ctx.inv = inv
        return torch.cat([f[:1], f.reshape(-1)[src].reshape(18, -1)])

    @staticmethod
    def backward(ctx, g):
        return torch.cat([g[:1], g[1:].reshape(-1)[ctx.inv].reshape(18, -1)]), None, None


def _moments(g, F, alpha):
    """rho - 1 and u of pulled deviations g."""
    rho = g.sum(0)
    u = []
    for a in range(3):
        j = sum(float(C[q][a]) * g[q] for q in range(1, 19) if C[q][a])
        u.append((j + 0.5 * F[a]) / (1.0 if alpha is None else 1.0 + 0.5 * alpha))
    return rho, u


def _collide(g, F, alpha, wp, wm):
    rho, u = _moments(g, F, alpha)
    Fn = [F[a] if alpha is None else F[a] - alpha * u[a] for a in range(3)]
    usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    out = [g[0] - wp * (g[0] - (rho - 1.5 * usq) / 3.0)]
    for p in range(1, 19, 2):
        a, b, w = g[p], g[p + 1], float(W[p])
        axes = [k for k in range(3) if C[p][k]]
        cu = sum(float(C[p][k]) * u[k] for k in axes)
        cF = sum(float(C[p][k]) * Fn[k] for k in axes)
        even = wp * (0.5 * (a + b) - w * (rho + 4.5 * cu * cu - 1.5 * usq))
        odd = wm * (0.5 * (a - b) - w * 3.0 * cu) - (1.0 - 0.5 * wm) * 3.0 * w * cF
        out += [a - even - odd, b - even + odd]
    return torch.stack(out), rho, u


def _exact_step(case, seed):
    bed = _bed(case, seed)
    src, n = _links(case, bed)
    alpha = _alpha(n, seed) if case["damped"] else None
    h = (_flow_deviation(n, case, seed) if case["start"] == "flow"
         else torch.zeros((19, n), dtype=torch.float64, device="cuda"))
    wp, F = case["omega"], _force(case, seed)
    rho = u = None
    for _ in range(case["steps"]):
        g = _Stream.apply(h, src, None)
        h, rho, u = _collide(g, F, alpha, wp, omega_minus_of(wp))
    u = torch.stack(u)
    w = torch.from_numpy(W).cuda()[:, None]
    return {"mass": n + float(rho.sum()), "flux": float(u[case["axis"]].mean()), "rho": 1.0 + rho,
            "u": u, "f": h + w}


def omega_minus_of(wp):
    """The odd rate of Lambda = 3/16."""
    return 1.0 / (0.5 + 0.1875 / (1.0 / wp - 0.5))


def _exact_adjoint(case, seed):
    from torch.utils.checkpoint import checkpoint
    bed = _bed(case, seed)
    src, n = _links(case, bed)
    inv = torch.empty(18 * n, dtype=torch.int64, device="cuda")
    inv[src - n] = torch.arange(18 * n, device="cuda")
    force = torch.tensor(_force(case, seed), dtype=torch.float64, device="cuda",
                         requires_grad=True)
    alpha = _alpha(n, seed).requires_grad_() if case["damped"] else None
    wp, wm = case["omega"], omega_minus_of(case["omega"])

    def advance(h, F, al, steps):
        for _ in range(steps):
            h = _collide(_Stream.apply(h, src, inv), F, al, wp, wm)[0]
        return h

    h = torch.zeros((19, n), dtype=torch.float64, device="cuda")
    left, stride = case["steps"] - 1, max(1, math.isqrt(case["steps"]))
    while left > 0:
        k = min(stride, left)
        h = checkpoint(advance, h, force, alpha, k, use_reentrant=False)
        left -= k
    J = _moments(_Stream.apply(h, src, inv), force, alpha)[1][case["axis"]].mean()
    J.backward()
    out = {"J": J.detach().cpu(), "force": force.grad.cpu()}
    if alpha is not None:
        out["alpha"] = alpha.grad
    return out


def exact(case, seed):
    if case["kind"] == "assemble":
        return None
    if case["kind"] == "batch":
        return None
    if case["kind"] == "adjoint":
        return (_exact_adjoint(case, seed)
                if _fluid(case) * case["steps"] < 2.5e8 else None)
    return _exact_step(case, seed) if _fluid(case) * case["steps"] < 4e9 else None
