"""Performance cases of the thermonoise library: the calls a user of it makes,
through the Python binding's public entry points, over the sizes the
repository's workloads and tests use.

  listed()             the cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  the context (mesh, materials, preconditioner factors)
                       and the seeded fields a program holds before the call
  run(state)           one pass
  work(case)           bytes and operations one pass cannot do without
  exact(case, seed)    the outputs in 64 bits from plain torch / numpy

A case is a dict: "op" (what is called), "prec" (f32 / f64 vectors) and the
mirror: "mesh" = "box" (nx x nx columns, `slabs` slabs) or "cylinder" (9 k^2
columns, `layers` coating layers of thickness `thick` on `slabs` substrate
slabs) with the polynomial degree "p", or "sweep" (a batch of `count` mirrors
of uneven degree, layer count and thickness).
"""
import math

import numpy as np
import torch

from paper_2111_06893_gb300 import thermonoise as tn

GPA = 1.0e9
SILICA = {"kind": "iso", "Y": 72 * GPA, "nu": 0.17}
HIGH = {"kind": "iso", "Y": 140 * GPA, "nu": 0.23}
CUBIC_A = {"kind": "cubic", "c11": 119.9 * GPA, "c12": 53.8 * GPA, "c44": 59.4 * GPA}
CUBIC_B = {"kind": "cubic", "c11": 120.5 * GPA, "c12": 57.0 * GPA, "c44": 58.9 * GPA}


# ------------------------------------------------------------------- cases

def listed():
    return [
        # operator applies: a user's own iteration, a residual, a data-driven model
        # the 12 288-unknown box of the plain method: launch latency counts
        {"name": "apply_f32_box_p3", "op": "apply", "prec": "f32", "mesh": "box", "p": 3, "nx": 4, "slabs": 4},
        # the single-coating mirror (2.0 M unknowns, p = 6)
        {"name": "apply_f32_cyl_p6", "op": "apply", "prec": "f32", "mesh": "cylinder", "p": 6, "k": 3, "layers": 1,
         "thick": 0.02, "slabs": 23, "R": 10.0},
        # the large mirror (59 M unknowns, p = 8): fields larger than L2
        {"name": "apply_f32_cyl_p8", "op": "apply", "prec": "f32", "mesh": "cylinder", "p": 8, "k": 10, "layers": 20,
         "thick": 1e-3, "slabs": 10, "R": 20.0},
        # FP64 residuals of the crystalline stack (8.0 M unknowns, p = 5)
        {"name": "apply_f64_cyl_p5", "op": "apply", "prec": "f64", "mesh": "cylinder", "p": 5, "k": 5, "layers": 40,
         "thick": 4e-4, "slabs": 15, "R": 10.0},
        # a design sweep held as one batch: degrees 4 to 8, uneven element counts
        {"name": "apply_f32_sweep", "op": "apply", "prec": "f32", "mesh": "sweep", "count": 24, "first": 0},
        # the grouped-line preconditioner (every Krylov iteration of a solve)
        {"name": "precond_f32_cyl_p6", "op": "precond", "prec": "f32", "mesh": "cylinder", "p": 6, "k": 3, "layers": 1,
         "thick": 0.02, "slabs": 23, "R": 10.0},
        {"name": "precond_f64_cyl_p7", "op": "precond", "prec": "f64", "mesh": "cylinder", "p": 7, "k": 2, "layers": 2,
         "thick": 0.05, "slabs": 9, "R": 10.0},
        {"name": "precond_f32_sweep", "op": "precond", "prec": "f32", "mesh": "sweep", "count": 24, "first": 0},
        # layer energies of a solved field (the crystalline stack's 41 layers)
        {"name": "energies_cyl_p5", "op": "energies", "prec": "f64", "mesh": "cylinder", "p": 5, "k": 5, "layers": 40,
         "thick": 4e-4, "slabs": 15, "R": 10.0},
        # plain FP64 solve of the small box, mesh and factors kept, a new beam width each time
        {"name": "solve_f64_box_p3", "op": "solve_f64", "prec": "f64", "mesh": "box", "p": 3, "nx": 4, "slabs": 4},
        # one step of a design study: a new mirror (mesh, materials, factors),
        # the mixed-precision solve and the layer energies
        {"name": "design_mixed_cyl_p6", "op": "design_mixed", "prec": "f64", "mesh": "cylinder", "p": 6, "k": 3,
         "layers": 1, "thick": 0.02, "slabs": 23, "R": 10.0},
        # energies and their gradient in every thickness, modulus and the beam
        # width through autograd: forward, adjoint solve, contractions
        {"name": "gradient_box_p4", "op": "gradient", "prec": "f64", "mesh": "box", "p": 4, "nx": 6, "slabs": 8},
    ]


def draw(rng):
    def logu(a, b):
        return math.exp(rng.uniform(math.log(a), math.log(b)))

    op = rng.choice(["apply", "apply", "apply", "precond", "precond", "energies", "solve_f64", "design_mixed",
                     "gradient"])
    prec = rng.choice(["f32", "f64"]) if op in ("apply", "precond") else "f64"
    if op in ("apply", "precond") and rng.random() < 0.25:
        # the mixed solves of a sweep apply its factors in FP32
        return {"op": op, "prec": prec if op == "apply" else "f32", "mesh": "sweep", "count": int(round(logu(2, 24))),
                "first": rng.randrange(1, 4096)}
    if op == "gradient":  # gradients of layered boxes: residual floor far below the solver's tolerance
        return {"op": op, "prec": prec, "mesh": "box", "p": rng.randint(3, 5), "nx": rng.randint(3, 6),
                "slabs": rng.randint(4, 8)}
    if op == "solve_f64":
        return {"op": op, "prec": prec, "mesh": "box", "p": rng.randint(3, 7), "nx": rng.randint(2, 5),
                "slabs": rng.randint(2, 7)}
    if op in ("apply", "precond", "energies") and rng.random() < 0.3:
        return {"op": op, "prec": prec, "mesh": "box", "p": rng.randint(2, 8), "nx": int(round(logu(1, 24))),
                "slabs": int(round(logu(1, 24)))}
    # cylinders, sized by their unknowns
    top = {"apply": 59e6 if prec == "f32" else 8e6, "precond": 8e6 if prec == "f32" else 2e6, "energies": 8e6,
           "design_mixed": 1.5e6}[op]
    p = rng.randint(4 if op == "design_mixed" else 2, 7 if op == "design_mixed" else 8)
    layers, slabs = int(round(logu(1, 40 if op != "design_mixed" else 4))), rng.randint(2, 23)
    per = 3 * (p + 1) ** 3 * 9 * (layers + slabs)  # unknowns at k = 1
    k = int(max(1, min(10, math.sqrt(logu(min(per, 0.9 * top), top) / per))))
    thin = {"design_mixed": 0.02, "precond": 4e-4 if prec == "f32" else 5e-3}.get(op, 4e-4)
    thick = logu(thin, 0.05)
    return {"op": op, "prec": prec, "mesh": "cylinder", "p": p, "k": k, "layers": layers,
            "thick": round(thick, 6), "slabs": slabs, "R": rng.choice([10.0, 20.0])}


# ----------------------------------------------------------------- mirrors

def _cylinder(R, thick, mats, k, p, n_sub, r0):
    """Coating layers (one linear slab each) on a substrate of n_sub slabs
    geometric in depth (logarithmic map inside), free mantle, fixed bottom."""
    depth = [0.0]
    for t in thick:
        depth.append(depth[-1] + t)
    d = depth[-1]
    depth += [d * (R / d) ** (i / n_sub) for i in range(1, n_sub + 1)]
    nl = len(thick)
    return {"kind": "cylinder", "degree": p, "R": R, "a": R / 5.0, "R1": R / 2.0, "k": k,
            "slab_z": [-z for z in depth], "slab_layer": list(range(nl)) + [nl] * n_sub,
            "slab_log": [0] * nl + [1] * n_sub, "materials": mats, "penalty_C": 100.0, "bc_side": "free",
            "bc_bottom": "fixed", "beam": {"r0": r0, "F0": 1.0}}


def _box(nx, slabs, p, r0, layered, rng):
    """[-10, 10]^2 x [-20, 0] in equal elements, fixed on all faces but the
    top; `layered`: a [-2, 2]^2 x [-2.5, 0] box of coating layers on silica."""
    if not layered:
        br = [-10.0 + 20.0 * i / nx for i in range(nx + 1)]
        return {"kind": "box", "degree": p, "x_breaks": br, "y_breaks": br,
                "slab_z": [-20.0 * i / slabs for i in range(slabs + 1)], "slab_layer": [0] * slabs,
                "slab_log": [0] * slabs, "materials": [SILICA], "penalty_C": 1.5, "bc_side": "fixed",
                "bc_bottom": "fixed", "beam": {"r0": r0, "F0": 1.0}}
    br = [-2.0 + 4.0 * i / nx for i in range(nx + 1)]
    nl = slabs // 2  # layers of unlike thickness over substrate slabs
    depth = [0.0]
    for i in range(nl):
        depth.append(depth[-1] + rng.uniform(0.08, 0.2))
    d = depth[-1]
    depth += [d + (2.5 - d) * ((i + 1) / (slabs - nl)) ** 1.5 for i in range(slabs - nl)]
    mats = [dict((CUBIC_A, HIGH, CUBIC_B, SILICA)[i % 4]) for i in range(nl)] + [SILICA]
    return {"kind": "box", "degree": p, "x_breaks": br, "y_breaks": br, "slab_z": [-z for z in depth],
            "slab_layer": list(range(nl)) + [nl] * (slabs - nl), "slab_log": [0] * slabs, "materials": mats,
            "penalty_C": 3.0, "bc_side": "fixed", "bc_bottom": "free", "beam": {"r0": r0, "F0": 1.0}}


def _sweep_mirror(seed):
    """One mirror of the design sweep: 1 to 20 layers, thicknesses log-uniform
    in [1e-4, 5e-2], beam width in [0.5, 2], degree 4 to 8, four substrate slabs."""
    rng = np.random.default_rng(seed)
    n = int(rng.integers(1, 21))
    th = np.exp(rng.uniform(math.log(1e-4), math.log(5e-2), size=n))
    r0, p = float(rng.uniform(0.5, 2.0)), int(rng.integers(4, 9))
    return _cylinder(10.0, [float(t) for t in th], [HIGH if i % 2 == 0 else SILICA for i in range(n)] + [SILICA], 1,
                     p, 4, r0)


def _descs(case, seed):
    """The mirror(s) of a case; the seed moves thicknesses and the beam width
    of the cases that solve, and the fields of the others."""
    rng = np.random.default_rng([7, seed])
    vary = case["op"] in ("solve_f64", "design_mixed", "gradient")
    r0 = float(rng.uniform(0.9, 1.1)) if vary else 1.0
    if case["mesh"] == "sweep":
        return [_sweep_mirror(case["first"] + i) for i in range(case["count"])]
    if case["mesh"] == "box":
        return [_box(case["nx"], case["slabs"], case["p"], r0, case["op"] == "gradient", rng)]
    n = case["layers"]
    th = [case["thick"] * (float(rng.uniform(0.95, 1.05)) if vary else 1.0) for _ in range(n)]
    if n >= 40:
        mats = [CUBIC_A if i % 2 == 0 else CUBIC_B for i in range(n)]
    else:
        mats = [HIGH if i % 2 == 0 else SILICA for i in range(n)]
    return [_cylinder(case["R"], th, mats + [SILICA], case["k"], case["p"], case["slabs"], r0)]


def _columns(d):
    return (len(d["x_breaks"]) - 1) * (len(d["y_breaks"]) - 1) if d["kind"] == "box" else 9 * d["k"] ** 2


def _ndof(d):
    return 3 * (d["degree"] + 1) ** 3 * _columns(d) * (len(d["slab_z"]) - 1)


def _field(n, seed, dtype):
    """Nodal values uniform in [-1, 1]."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 17)
    return torch.rand(n, dtype=torch.float64, device="cuda", generator=g).mul_(2).sub_(1).to(dtype)


# ------------------------------------------------------------- prepare, run

def prepare(case, seed):
    descs = _descs(case, seed)
    op = case["op"]
    dtype = torch.float32 if case["prec"] == "f32" else torch.float64
    if op == "gradient":
        d = descs[0]
        mod = [tn.iso_moduli(m["Y"], m["nu"]) if m["kind"] == "iso" else (m["c11"], m["c12"], m["c44"])
               for m in d["materials"]]
        return {"op": op, "desc": d, "z": torch.tensor(d["slab_z"], dtype=torch.float64),
                "r0": torch.tensor(d["beam"]["r0"], dtype=torch.float64),
                "mod": torch.tensor(mod, dtype=torch.float64),
                "w": torch.tensor(np.random.default_rng(seed).uniform(0.5, 2.0, len(mod)))}
    if op == "design_mixed":
        return {"op": op, "desc": descs[0], "ctx": tn.Context()}
    if case["mesh"] == "sweep":
        ctx = tn.Context().build_batch(descs)
    else:
        ctx = tn.setup(descs[0])
    if op == "solve_f64":
        ctx.precond_factor_bytes()  # builds the factors: a program that solves for many beams keeps them
        return {"op": op, "ctx": ctx}
    u = _field(ctx.ndof, seed, dtype)
    if op == "precond":
        ctx.precond_factor_bytes()
    return {"op": op, "ctx": ctx, "u": u, "y": torch.empty_like(u)}


def run(state):
    op = state["op"]
    if op == "apply":
        return state["ctx"].apply_operator(state["u"], state["y"])
    if op == "precond":
        return state["ctx"].precond_apply(state["u"], state["y"], "zgroup")
    if op == "energies":
        return state["ctx"].layer_energies(state["u"])
    if op == "solve_f64":
        ctx = state["ctx"]
        u, _ = ctx.solve(mode="f64", rtol=1e-12)
        return {"u": u, "U": ctx.layer_energies(u)}
    if op == "design_mixed":
        ctx, d = state["ctx"], state["desc"]
        ctx.build_mesh(d).set_materials(d["materials"]).set_beam(d["beam"]["r0"], d["beam"]["F0"])
        u, _ = ctx.solve(mode="mixed", rtol=1e-13, energy_rtol=1e-12)
        return {"u": u, "U": ctx.layer_energies(u)}
    z, r0, mod = (state[k].clone().requires_grad_(True) for k in ("z", "r0", "mod"))
    U = tn.energy_fn().apply(z, r0, mod, state["desc"], {"mode": "mixed", "rtol": 1e-12})
    (U * state["w"]).sum().backward()
    return {"U": U.detach(), "z": z.grad, "r0": r0.grad, "moduli": mod.grad}


# --------------------------------------------------------------------- work

def _apply_flops(d):
    """Sum-factorised gradient and divergence (36 N per node), strain, stress
    and fluxes per node, traction, jump and penalty per face node."""
    N = d["degree"] + 1
    return _columns(d) * (len(d["slab_z"]) - 1) * (N ** 3 * (36 * N + 80) + 6 * N * N * 130)


def _factor_entries(d):
    """Entries of the inverse Schur complements (symmetric) and of the slab
    couplings (6 numbers per row) of every group of lines through one point
    of the cross-section."""
    N = d["degree"] + 1
    pts = np.round(_cross_section(d)[0].reshape(-1, 2), 6) + 0.0
    sizes = np.unique(pts, axis=0, return_counts=True)[1]
    M = 3 * N * sizes.astype(np.float64)
    return (len(d["slab_z"]) - 1) * float(np.sum(M * (M + 1) / 2 + 6 * M))


def work(case):
    descs = _descs(case, 0)
    es = 4 if case["prec"] == "f32" else 8
    n, fl = sum(_ndof(d) for d in descs), sum(_apply_flops(d) for d in descs)
    if case["op"] == "apply":
        return {"bytes": 2 * n * es, "flops": fl}
    fac = sum(_factor_entries(d) for d in descs)
    if case["op"] == "precond":
        return {"bytes": fac * es + 2 * n * es, "flops": 4 * fac}
    if case["op"] == "energies":
        return {"bytes": n * es, "flops": fl // 2}
    # solves: iterations taken at the stated tolerances, each an operator
    # apply, a factor pass and the vector updates
    its, es = {"solve_f64": (80, 8), "design_mixed": (800, 4), "gradient": (250, 4)}[case["op"]]
    return {"bytes": its * (fac * es + 12 * n * es), "flops": its * (fl + 4 * fac)}


# --------------------------------------------------- 64-bit reference (torch)

def _lgl(N):
    c = np.zeros(N)
    c[-1] = 1.0
    P = np.polynomial.legendre.Legendre(c)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    w = 2.0 / (N * (N - 1) * P(x) ** 2)
    D = np.zeros((N, N))
    for a in range(N):
        for b in range(N):
            if a != b:
                D[a, b] = P(x[a]) / (P(x[b]) * (x[a] - x[b]))
    D[0, 0], D[-1, -1] = -N * (N - 1) / 4.0, N * (N - 1) / 4.0
    return x, w, D


def _map_xy(d, c, xi, eta):
    if d["kind"] == "box":
        xb, yb = d["x_breaks"], d["y_breaks"]
        i, j = c % (len(xb) - 1), c // (len(xb) - 1)
        return xb[i] + 0.5 * (1 + xi) * (xb[i + 1] - xb[i]), yb[j] + 0.5 * (1 + eta) * (yb[j + 1] - yb[j])
    k, a, R1, R = d["k"], d["a"], d["R1"], d["R"]
    blk, cl = divmod(c, k * k)
    s, t = -1.0 + (2.0 * (cl % k) + 1.0 + xi) / k, -1.0 + (2.0 * (cl // k) + 1.0 + eta) / k
    if blk == 0:
        return a * s, a * t
    th = math.pi * t / 4.0
    if blk <= 4:
        x = 0.5 * (1 - s) * a + 0.5 * (1 + s) * R1 * np.cos(th)
        y = 0.5 * (1 - s) * a * t + 0.5 * (1 + s) * R1 * np.sin(th)
    else:
        rad = 0.5 * (1 - s) * R1 + 0.5 * (1 + s) * R
        x, y = rad * np.cos(th), rad * np.sin(th)
    return ((x, y), (-y, x), (-x, -y), (y, -x))[(blk - 1) % 4]


def _cross_section(d):
    """Node positions [col, N^2, 2] (node j N + i) and Jacobians [col, N^2, 2, 2]."""
    x = _lgl(d["degree"] + 1)[0]
    eta, xi = (v.ravel() for v in np.meshgrid(x, x, indexing="ij"))
    h = 1e-30
    pos, jac = [], []
    for c in range(_columns(d)):
        X, Y = _map_xy(d, c, xi + 1j * h, eta + 0j)
        X2, Y2 = _map_xy(d, c, xi + 0j, eta + 1j * h)
        pos.append(np.stack([np.real(X), np.real(Y)], -1))
        jac.append(np.stack([np.stack([X.imag, X2.imag], -1), np.stack([Y.imag, Y2.imag], -1)], -2) / h)
    return np.array(pos), np.array(jac)


class _Reference:
    """The discontinuous-Galerkin operator on [..., slab, col, 3, k, N^2] fields."""

    def __init__(self, d):
        def dev(v):
            return torch.as_tensor(np.ascontiguousarray(v), device="cuda")

        N = self.N = d["degree"] + 1
        x, w, D = _lgl(N)
        pos, J = _cross_section(d)
        self.nc, self.ns = len(pos), len(d["slab_z"]) - 1
        det2, inv = np.linalg.det(J), np.linalg.inv(J)  # inv[c, q, m, a] = d xi^m / d x^a
        zt, zb = np.array(d["slab_z"][:-1])[:, None], np.array(d["slab_z"][1:])[:, None]
        a, b = 0.5 * (1 + x), 0.5 * (1 - x)
        log = np.array(d["slab_log"])[:, None] > 0
        top, bot = np.where(log, -zt, 1.0), np.where(log, -zb, 2.0)
        dz = np.where(log, 0.5 * np.exp(a * np.log(top) + b * np.log(bot)) * np.log(bot / top), 0.5 * (zt - zb))
        self.D, self.w1 = dev(D), dev(w)
        self.inv, self.det2, self.dz = dev(inv), dev(det2), dev(dz)
        w2 = np.outer(w, w).ravel()
        self.wJ = dev(w2)[None, None, None] * self.det2[None, :, None] * (self.w1 * self.dz)[:, None, :, None]
        mats = [tuple(_lame(m)) for m in d["materials"]]
        self.c = [dev([mats[L][q] for L in d["slab_layer"]]) for q in range(3)]
        self.layer = dev(np.array(d["slab_layer"]))
        self.nl = len(mats)
        self.pen = d["penalty_C"] * N * N
        self.fixed_side, self.fixed_bottom = d["bc_side"] == "fixed", d["bc_bottom"] == "fixed"
        # lateral edges: own nodes, and the matching nodes of the column across
        r = np.arange(N)
        self.edge = [r * N, r * N + N - 1, r, (N - 1) * N + r]
        ends, where = {}, {}
        for c in range(self.nc):
            for f in range(4):
                key = tuple(np.round(pos[c, self.edge[f]].mean(0), 6) + 0.0)
                ends.setdefault(key, []).append((c, f))
        self.nb = []
        for f in range(4):
            nbc, nbq = np.zeros(self.nc, int), np.zeros((self.nc, N), int)
            inner, mag2 = np.zeros(self.nc, bool), np.zeros((self.nc, N))
            for c in range(self.nc):
                key = tuple(np.round(pos[c, self.edge[f]].mean(0), 6) + 0.0)
                nbc[c], nbq[c] = c, self.edge[f]
                for c2, f2 in ends[key]:
                    if (c2, f2) != (c, f):
                        q = self.edge[f2]
                        dist = np.abs(pos[c, self.edge[f]][:, None] - pos[c2, q][None]).sum(-1)
                        nbc[c], nbq[c], inner[c] = c2, q[dist.argmin(1)], True
                        mag2[c] = np.linalg.norm(inv[c2, nbq[c], f2 // 2], axis=-1)
            q = self.edge[f]
            row = inv[:, q, f // 2] * (1.0 if f & 1 else -1.0)
            mag = np.linalg.norm(row, axis=-1)
            # h = 2 / mag; W = tangential weights * det * mag
            W = dev((w * det2[:, q] * mag)[None, :, None, :]) * (self.w1 * self.dz)[:, None, :, None]
            self.nb.append((dev(nbc), dev(nbq), dev(inner), dev(row / mag[..., None]), W,
                            dev(0.5 * np.maximum(mag, mag2))))
        self.w2 = dev(w2)

    def stress(self, S, c=None):
        """S, result: six fields (xx, yy, zz, xy, xz, yz); c: moduli per slab."""
        c11, c12, c44 = (v.view(-1, 1, 1, 1) for v in (c or self.c))
        tr, df = c12 * (S[0] + S[1] + S[2]), c11 - c12
        return [df * S[0] + tr, df * S[1] + tr, df * S[2] + tr, 2 * c44 * S[3], 2 * c44 * S[4], 2 * c44 * S[5]]

    def strain(self, u):
        N, D = self.N, self.D
        v = u.unflatten(-1, (N, N))
        dx = (v @ D.T).flatten(-2)
        dy = torch.einsum("jm,...mi->...ji", D, v).flatten(-2)
        dzt = torch.einsum("km,...mq->...kq", D, u) / self.dz[:, None, None, :, None]
        i = self.inv[:, None, None]
        g = [i[..., 0, 0] * dx + i[..., 1, 0] * dy, i[..., 0, 1] * dx + i[..., 1, 1] * dy, dzt]
        G = [[g[a][..., l, :, :] for l in range(3)] for a in range(3)]
        return [G[0][0], G[1][1], G[2][2], 0.5 * (G[0][1] + G[1][0]), 0.5 * (G[0][2] + G[2][0]),
                0.5 * (G[1][2] + G[2][1])]

    @staticmethod
    def dot_n(s, n):
        return torch.stack([n[0] * s[0] + n[1] * s[3] + n[2] * s[4], n[0] * s[3] + n[1] * s[1] + n[2] * s[5],
                            n[0] * s[4] + n[1] * s[5] + n[2] * s[2]])

    @staticmethod
    def outer(n, v):
        return [n[0] * v[0], n[1] * v[1], n[2] * v[2], 0.5 * (n[0] * v[1] + n[1] * v[0]),
                0.5 * (n[0] * v[2] + n[2] * v[0]), 0.5 * (n[1] * v[2] + n[2] * v[1])]

    def energies(self, u):
        u = u.view(self.ns, self.nc, 3, self.N, -1)
        S = self.strain(u)
        s = self.stress(S)
        e = S[0] * s[0] + S[1] * s[1] + S[2] * s[2] + 2 * (S[3] * s[3] + S[4] * s[4] + S[5] * s[5])
        e = (0.5 * self.wJ * e).sum((1, 2, 3))
        return torch.zeros(self.nl, dtype=e.dtype, device=e.device).index_add_(0, self.layer, e)

    def apply(self, u):
        N, ns, nc = self.N, self.ns, self.nc
        u = u.view(-1, ns, nc, 3, N, N * N) if u.dim() > 1 else u.view(ns, nc, 3, N, N * N)
        y = torch.zeros_like(u)
        S = self.strain(u)
        sig = self.stress(S)
        wJ = self.wJ
        eff = [wJ * v for v in S]
        del S
        uc = [u[..., l, :, :] for l in range(3)]
        one = torch.ones(1, dtype=u.dtype, device=u.device)
        for f in range(4):
            nbc, nbq, inner, n, W, hinv = self.nb[f]
            q = torch.as_tensor(self.edge[f], device=u.device)
            n3 = [n[:, None, :, 0], n[:, None, :, 1], 0 * one]  # [col, 1, t]
            across = [v[..., nbc[:, None], :, nbq].movedim((0, 1), (-3, -1)) for v in uc + sig]
            own, inn = [v[..., q] for v in uc], inner.view(-1, 1, 1)
            so = [v[..., q] for v in sig]
            on = inn | torch.tensor(self.fixed_side, device=u.device)
            jump = [torch.where(inn, a - b, 2 * a) * on for a, b in zip(own, across[:3])]
            trac = 0.5 * self.dot_n([a + torch.where(inn, b, a) for a, b in zip(so, across[3:])], n3)
            E = self.outer(n3, jump)
            pen = self.dot_n(self.stress(E), n3) * (self.pen * hinv[:, None, :])  # one slab: one material
            for l in range(3):
                y[..., l, :, :][..., q] -= W[:, :, :] * on * (trac[l] - pen[l])
            for l in range(6):
                eff[l][..., q] += -0.5 * W * E[l]
        for k, sgn, sh in ((0, -1.0, -1), (N - 1, 1.0, 1)):  # bottom, top of every slab
            ko = N - 1 - k
            dim = u.dim() - 5
            idx = torch.arange(ns, device=u.device)
            nbi = (idx + 1 if sgn < 0 else idx - 1)
            inner = ((nbi >= 0) & (nbi < ns)).view(-1, 1, 1)
            nbi = nbi.clamp(0, ns - 1)
            on = inner.clone()
            if sgn < 0 and self.fixed_bottom:
                on[:] = True
            n3 = [0 * one, 0 * one, sgn * one]
            own, so = [v[..., k, :] for v in uc], [v[..., k, :] for v in sig]
            ext = [v[..., ko, :].index_select(dim, nbi) for v in uc + sig]
            jump = [torch.where(inner, a - b, 2 * a) * on for a, b in zip(own, ext[:3])]
            trac = 0.5 * self.dot_n([a + torch.where(inner, b, a) for a, b in zip(so, ext[3:])], n3)
            E = self.outer(n3, jump)
            m = inner.flatten()
            cs = [torch.where(m, 0.5 * (v + v[nbi]), v) for v in self.c]
            h = torch.where(m, torch.minimum(self.dz[:, k], self.dz[nbi, ko]), self.dz[:, k]) * 2
            sE = [v.squeeze(-2) for v in self.stress([e.unsqueeze(-2) for e in E], cs)]
            pen = self.dot_n(sE, n3) * (self.pen / h).view(-1, 1, 1)
            W = (self.w2 * self.det2)[None]
            for l in range(3):
                y[..., l, k, :] -= W * on * (trac[l] - pen[l])
            for l in range(6):
                eff[l][..., k, :] += -0.5 * W * E[l]
        del sig
        s = self.stress(eff)
        rows = [[s[0], s[3], s[4]], [s[3], s[1], s[5]], [s[4], s[5], s[2]]]
        i = self.inv[:, None, :]  # [col, 1, q, m, a]
        for l in range(3):
            Fx, Fy = (i[..., m, 0] * rows[0][l] + i[..., m, 1] * rows[1][l] for m in range(2))
            Fz = rows[2][l] / self.dz[:, None, :, None]
            Fx, Fy = Fx.unflatten(-1, (N, N)), Fy.unflatten(-1, (N, N))
            y[..., l, :, :] += (Fx @ self.D).flatten(-2) + torch.einsum("mj,...mi->...ji", self.D, Fy).flatten(-2) \
                + torch.einsum("mk,...mq->...kq", self.D, Fz)
        return y

    def load(self, d):
        """The Gaussian beam pressure on the top surface, as a right-hand side."""
        r0, F0 = d["beam"]["r0"], d["beam"]["F0"]
        r2 = torch.as_tensor((_cross_section(d)[0] ** 2).sum(-1), device="cuda")
        b = torch.zeros(self.ns, self.nc, 3, self.N, self.N ** 2, dtype=torch.float64, device="cuda")
        b[0, :, 2, self.N - 1] = -self.w2 * self.det2 * F0 * torch.exp(-r2 / r0 ** 2) / (math.pi * r0 ** 2)
        return b.flatten()


def _lame(m):
    if m["kind"] == "cubic":
        return m["c11"], m["c12"], m["c44"]
    mu = m["Y"] / (2 * (1 + m["nu"]))
    lam = m["Y"] * m["nu"] / ((1 + m["nu"]) * (1 - 2 * m["nu"]))
    return lam + 2 * mu, lam, mu


def exact(case, seed):
    op = case["op"]
    if op not in ("apply", "energies", "solve_f64"):
        return None  # factorised blocks, thin-layer solves and adjoints: minutes as plain dense algebra
    descs = _descs(case, seed)
    dtype = torch.float32 if case["prec"] == "f32" else torch.float64
    if op == "solve_f64":
        d = descs[0]
        n = _ndof(d)
        if n > 13000:
            return None  # dense factorisation too large
        ref = _Reference(d)
        A = torch.empty(n, n, dtype=torch.float64, device="cuda")
        for c in range(0, n, 1024):
            m = min(1024, n - c)
            e = torch.zeros(m, n, dtype=torch.float64, device="cuda")
            e[torch.arange(m), c + torch.arange(m)] = 1.0
            A[c:c + m] = ref.apply(e).reshape(m, n)
        L = torch.linalg.cholesky(0.5 * (A + A.T))
        b = ref.load(d)
        u = torch.cholesky_solve(b[:, None], L)[:, 0]
        u += torch.cholesky_solve((b - A @ u)[:, None], L)[:, 0]
        return {"u": u, "U": ref.energies(u).cpu().numpy()}
    u = _field(sum(_ndof(d) for d in descs), seed, dtype).double()
    out, at = [], 0
    for d in descs:
        ref, n = _Reference(d), _ndof(d)
        ui = u[at:at + n]
        out.append(ref.apply(ui).reshape(-1) if op == "apply" else ref.energies(ui))
        at += n
    out = torch.cat(out)
    return out if op == "apply" else out.cpu().numpy()
