"""The measured cases: the work that users of this library have it do, through the Python entry points.

Kinds of pass (every array is made on the GPU from the seed alone):
  demag     one mm_demag_field call: the demagnetisation field of a state, alone
  field     one mm_effective_field call: demag + exchange + anisotropy + Zeeman (+ DMI)
  relax     mm_relax (adaptive RKF45) to a fixed simulated time: the dynamics run of an example script, cut short
  rk4       mm_rk4_trajectory: fixed-step dynamics
  minimize  mm_minimize_bb: a fixed number of Barzilai-Borwein iterations towards a ground state
  gradient  mm_rk4_trajectory, then mm_rk4_trajectory_vjp: one gradient of an inverse-design loop over the cell-wise Ms
  energy    mm_energy and mm_max_torque: the read-out of a state
Meshes, cells and materials are those of this repository's workloads, tests and benchmark, or generic ones between them.
"""
import functools
import math

import numpy as np
import torch

import paper_2606_01114_gb300 as mm

MU0 = 4e-7 * math.pi
GAMMA = 2.2127615e5
TARGET = (0.0, 0.0, 1.0)      # the gradient cases pull the final state towards this direction


def _case(name, kind, n, d, prec, **more):
    c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "dx": d[0], "dy": d[1], "dz": d[2], "prec": prec,
         "Ms": 8e5, "A": 1.3e-11, "alpha": 0.02, "Ku": 0.0, "D": 0.0, "ms_map": "uniform", "state": "smooth"}
    c.update(more)
    return c if name is None else {"name": name, **c}


def listed():
    nm = 1e-9
    return [
        # one field of the standard-problem-4 film: the smallest call, all latency
        _case("field_sp4_f32", "field", (100, 25, 1), (5 * nm, 5 * nm, 3 * nm), "f32"),
        # the standard-problem-4 film moved on in double precision: a small dynamics run, host and launches count
        _case("relax_sp4_f64", "relax", (100, 25, 1), (5 * nm, 5 * nm, 3 * nm), "f64", t_max=8e-12, steps=24),
        # the small film in fixed RK4 steps
        _case("rk4_film64_f32", "rk4", (64, 64, 4), (2.5 * nm, 2.5 * nm, 3 * nm), "f32", state="random", dt=1e-13, steps=20),
        # demag of one single-layer film: the usual 2-D problem
        _case("demag_film256_f32", "demag", (256, 256, 1), (4 * nm, 4 * nm, 4 * nm), "f32"),
        # a disc cut out of a mesh of no special size, vacuum around it
        _case("field_disc300_f32", "field", (300, 300, 2), (3 * nm, 3 * nm, 3 * nm), "f32", ms_map="disc"),
        # an ordinary mesh whose sides are not powers of two
        _case("field_film350_f32", "field", (350, 350, 4), (3 * nm, 3 * nm, 3 * nm), "f32", Ku=1e5),
        # the ground state of a film with interfacial DMI
        # (in double precision: the step lengths are quotients of differences, which single precision carries to 1e-4 at best)
        _case("minimize_dmi256_ff", "minimize", (256, 256, 1), (2 * nm, 2 * nm, 1 * nm), "ff", Ms=5.8e5, A=1.5e-11, alpha=0.3, Ku=8e5, D=3e-3, steps=20),
        # one gradient with respect to the cell-wise saturation magnetisation
        _case("gradient_design256_f32", "gradient", (256, 256, 4), (3 * nm, 3 * nm, 3 * nm), "f32", ms_map="smooth", dt=1e-13, steps=9),
        # energies and torque of a design in double precision
        _case("energy_design256_f64", "energy", (256, 256, 4), (3 * nm, 3 * nm, 3 * nm), "f64", ms_map="smooth", Ku=1e5),
        # the large film in float-float arithmetic (double-precision context)
        _case("demag_film512_ff", "demag", (512, 512, 16), (2 * nm, 2 * nm, 2 * nm), "ff", state="vortex"),
        # the effective field of the cube: the longest z transforms, the largest mesh
        _case("field_cube256_f32", "field", (256, 256, 256), (1 * nm, 1 * nm, 1 * nm), "f32", Ku=5e5, state="random"),
        # the benchmark film moved on by the adaptive integrator: the headline path
        _case("relax_film512_f32", "relax", (512, 512, 16), (2 * nm, 2 * nm, 2 * nm), "f32", alpha=0.5, state="vortex", t_max=4e-13, steps=10),
    ]


def _side(rng, lo=16, hi=512):
    if rng.random() < 0.5:
        return 2 ** rng.randint(int(math.log2(lo)), int(math.log2(hi)))
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["demag", "field", "field", "relax", "rk4", "minimize", "gradient", "energy"])
    prec = {"demag": rng.choice(["f32", "f32", "ff", "f64"]), "field": rng.choice(["f32", "f32", "f64"]),
            "relax": rng.choice(["f32", "f32", "f64"]), "minimize": rng.choice(["ff", "f64"]), "energy": "f64"}.get(kind, "f32")
    # cell evaluations a pass may cost, by how much dearer the arithmetic is
    most = {"f32": 1.0, "ff": 0.08, "f64": 0.03}[prec] * 1.2e8
    per = {"relax": 6, "rk4": 4, "minimize": 1, "gradient": 20}.get(kind, 1)
    steps = {"relax": rng.randint(4, 20), "rk4": rng.randint(5, 25), "minimize": rng.randint(8, 20), "gradient": rng.randint(4, 9)}.get(kind, 1)
    while True:
        n = (_side(rng), _side(rng), 2 ** rng.randint(0, 5 if kind in ("demag", "field") else 4))
        if prec == "ff" and any(v & (v - 1) for v in n):
            continue
        cells = n[0] * n[1] * n[2]
        dear = 4 if any(v & (v - 1) for v in n) else 1
        if 1000 <= cells <= 512 * 512 * 16 and cells * per * steps * dear <= most:
            break
    h = rng.choice([2e-9, 2.5e-9, 3e-9, 4e-9])
    c = _case(None, kind, n, (h, h, rng.choice([0.75, 1.0, 1.2]) * h), prec, state=rng.choice(["smooth", "vortex", "random"]))
    if kind != "demag":
        c["Ku"] = rng.choice([0.0, 1e5, 5e5])
        c["alpha"] = rng.choice([0.02, 0.1, 0.5])
    if kind in ("field", "energy", "demag", "gradient"):
        c["ms_map"] = "smooth" if kind == "gradient" else rng.choice(["uniform", "smooth", "disc"])
    if kind in ("field", "relax", "minimize") and rng.random() < 0.25:
        c["D"] = 1.5e-3
    if kind in ("rk4", "gradient"):
        c["dt"] = 5e-14 if h < 2.4e-9 else 1e-13
    if kind == "relax":
        c["t_max"] = steps * (8e-14 if h < 2.4e-9 else 1.5e-13)
    if kind in ("relax", "rk4", "minimize", "gradient"):
        c["steps"] = steps
    return c


# ------------------------------------------------------------------ inputs
def _gen(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 13)
    return g


def _coords(case):
    return [((torch.arange(k, device="cuda", dtype=torch.float64) + 0.5) / k - 0.5).reshape([-1 if a == ax else 1 for a in range(3)])
            for ax, k in ((2, case["nx"]), (1, case["ny"]), (0, case["nz"]))]


def _smooth(case, g, waves=6):
    """A sum of a few plane waves of random direction and phase, about 1 in size."""
    x, y, z = _coords(case)
    w = torch.randn((waves, 4), generator=g, device="cuda", dtype=torch.float64).cpu().tolist()
    f = 0.0
    for a, b, c, p in w:
        f = f + torch.cos(2 * math.pi * (2.0 * a * x + 2.0 * b * y + 0.3 * c * z) + 6.0 * p)
    return f.expand(case["nz"], case["ny"], case["nx"]) / math.sqrt(waves / 2)


def _dtype(case):
    return torch.float32 if case["prec"] == "f32" else torch.float64


def _inputs(case, seed):
    """(m, Ms per cell or None) in the context's type."""
    g = _gen(case, seed)
    shape = (3, case["nz"], case["ny"], case["nx"])
    if case["state"] == "random":
        m = torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    elif case["state"] == "vortex":      # vortex in the middle with 5 % noise
        x, y, z = _coords(case)
        X, Y = x * case["nx"] * case["dx"], y * case["ny"] * case["dy"]
        r = torch.sqrt(X * X + Y * Y).clamp_min(1e-12)
        mz = torch.exp(-(r / 10e-9) ** 2)
        ip = torch.sqrt(1 - mz * mz)
        m = torch.stack([(v + 0 * z).expand(shape[1:]) for v in (-Y / r * ip, X / r * ip, mz)])
        m = m + 0.05 * torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    else:
        m = torch.stack([_smooth(case, g) for _ in range(3)]) + 0.02 * torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    m = m / m.norm(dim=0, keepdim=True)
    ms = None
    if case["ms_map"] == "smooth":
        f = _smooth(case, g)
        ms = 4e5 + 5e5 * (f - f.min()) / (f.max() - f.min())
    elif case["ms_map"] == "disc":
        x, y, _ = _coords(case)
        ms = torch.where(x * x + y * y < 0.23, case["Ms"], 0.0).expand(shape[1:])
    t = _dtype(case)
    return m.to(t).contiguous(), None if ms is None else ms.to(t).contiguous()


def prepare(case, seed):
    m0, ms = _inputs(case, seed)
    ctx = mm.mm_init_mesh(case["nx"], case["ny"], case["nz"], case["dx"], case["dy"], case["dz"],
                          precision=mm.MM_F32 if case["prec"] == "f32" else mm.MM_F64)
    mm.mm_set_material(ctx, case["Ms"], case["A"], case["alpha"], case["Ku"])
    if ms is not None:
        mm.mm_set_material_fields(ctx, Ms_cell=ms)
    if case["D"]:
        mm.mm_set_dmi(ctx, case["D"], mm.MM_DMI_INTERFACIAL)
    if case["prec"] == "ff":
        mm.mm_set_fft_mode(ctx, mm.MM_FFT_FF)
    return {"case": case, "ctx": ctx, "m0": m0, "ms": ms, "m": torch.empty_like(m0), "H": torch.empty_like(m0)}


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "demag":
        mm.mm_demag_field(ctx, s["m0"], s["H"])
        return s["H"]
    if kind == "field":
        mm.mm_effective_field(ctx, s["m0"], s["H"])
        return s["H"]
    if kind == "energy":
        return mm.mm_energy(ctx, s["m0"]), mm.mm_max_torque(ctx, s["m0"])
    m = s["m"].copy_(s["m0"])
    if kind == "relax":
        t, _ = mm.mm_relax(ctx, m, case["t_max"], torque_tol=0.0)
        return m, t
    if kind == "rk4":
        mm.mm_rk4_trajectory(ctx, m, case["dt"], case["steps"])
        return m
    if kind == "minimize":
        try:
            mm.mm_minimize_bb(ctx, m, torque_tol=0.0, max_iter=case["steps"])
        except mm.MMError as e:
            if e.code != mm.MM_ERR_NOT_CONVERGED:     # the number of iterations is the limit here
                raise
        return m
    mm.mm_rk4_trajectory(ctx, m, case["dt"], case["steps"])
    lam = m - torch.tensor(TARGET, dtype=m.dtype, device=m.device).reshape(3, 1, 1, 1)
    g = torch.zeros(ctx.shape1, dtype=m.dtype, device=m.device)
    mm.mm_rk4_trajectory_vjp(ctx, s["m0"], case["dt"], case["steps"], lam, g)
    return m, lam, g


def work(case):
    n = (case["nx"], case["ny"], case["nz"])
    cells = n[0] * n[1] * n[2]
    e = 4 if case["prec"] == "f32" else 8
    # one field evaluation: real transforms of three components there and back over the padded grid, the non-zero
    # parts only (3/8 of the first level's lines, half of the second's), the symmetric product, the local terms
    px, py, pz = (2 * v if v > 1 else 1 for v in n)

    def line(p):
        return 5.0 * p * math.log2(p) if p > 1 else 0.0
    flops = 6 * (n[1] * n[2] * line(px) / 2 + (n[0] + 1) * n[2] * line(py) + (n[0] + 1) * py * line(pz)) + 30.0 * (n[0] + 1) * py * pz
    local = {"demag": 0.0, "field": 60.0, "energy": 80.0}.get(case["kind"], 120.0) * cells
    # field evaluations of a pass; each needs the whole state and gives a whole field
    evals = {"demag": 1, "field": 1, "energy": 2, "relax": 6 * case.get("steps", 1) + 1, "rk4": 4 * case.get("steps", 1),
             "minimize": case.get("steps", 1) + 1, "gradient": 12 * case.get("steps", 1)}[case["kind"]]
    fields = {"energy": 1}.get(case["kind"], 2)
    return {"bytes": float(evals * (fields * 3 + (case["ms_map"] != "uniform")) * cells * e), "flops": evals * (flops + local)}


# ------------------------------------------- the same in 64 bits, plain torch
def _newell_f(x, y, z):
    x, y, z = x.abs(), y.abs(), z.abs()
    r = torch.sqrt(x * x + y * y + z * z)
    t = 1e-300

    def part(a, b, c):   # a/2 (c^2 - b^2) asinh(a / sqrt(b^2 + c^2))
        q = torch.sqrt(b * b + c * c)
        return torch.where(q > 0, 0.5 * a * (c * c - b * b) * torch.asinh(a / q.clamp_min(t)), torch.zeros_like(r))
    at = torch.where(x * r > 0, x * y * z * torch.atan(y * z / (x * r).clamp_min(t)), torch.zeros_like(r))
    # f is even in every argument; axes of the two logarithms: y and z against x
    return part(y, x, z) + part(z, x, y) - at + (2 * x * x - y * y - z * z) * r / 6


def _newell_g(x, y, z):
    z = z.abs()
    r = torch.sqrt(x * x + y * y + z * z)
    t = 1e-300

    def lg(a, b, c):
        q = torch.sqrt(b * b + c * c)
        return torch.where(q > 0, torch.asinh(a / q.clamp_min(t)), torch.zeros_like(r))

    def at(num, den):
        return torch.where(den.abs() > 0, torch.atan(num / torch.where(den == 0, torch.ones_like(den), den)), torch.zeros_like(r))
    return (x * y * z * lg(z, x, y) + y / 6 * (3 * z * z - y * y) * lg(x, y, z) + x / 6 * (3 * z * z - x * x) * lg(y, x, z)
            - z ** 3 / 6 * at(x * y, z * r) - z * y * y / 2 * at(x * z, y * r) - z * x * x / 2 * at(y * z, x * r) - x * y * r / 3)


def _near(i, j, k, d):
    """The six components at the given cell offsets from Newell's formulas (second differences, 64 bits)."""
    (dx, dy, dz), V = d, d[0] * d[1] * d[2]

    def diff(fn, perm):
        acc = 0.0
        for a, wa in ((-1, -1.0), (0, 2.0), (1, -1.0)):
            for b, wb in ((-1, -1.0), (0, 2.0), (1, -1.0)):
                for c, wc in ((-1, -1.0), (0, 2.0), (1, -1.0)):
                    r = ((i + a) * dx, (j + b) * dy, (k + c) * dz)
                    acc = acc + wa * wb * wc * fn(*(r[q] for q in perm))
        return acc / (4 * math.pi * V)
    return [diff(_newell_f, (0, 1, 2)), diff(_newell_f, (1, 2, 0)), diff(_newell_f, (2, 0, 1)),
            diff(_newell_g, (0, 1, 2)), diff(_newell_g, (0, 2, 1)), diff(_newell_g, (1, 2, 0))]


def _far(i, j, k, d):
    """The same from the dipole kernel, averaged over both cells: 5-point Gauss rule of the triangular weight per axis."""
    mom = np.zeros(11)      # moments of 1 - |u| on [-1, 1]
    mom[::2] = [2.0 / ((2 * q + 1) * (2 * q + 2)) for q in range(6)]
    hank = np.array([[mom[p + q] for q in range(6)] for p in range(6)])
    L = np.linalg.cholesky(hank)
    R = L.T
    off = [R[q, q + 1] / R[q, q] - (R[q - 1, q] / R[q - 1, q - 1] if q else 0.0) for q in range(5)]
    sub = [R[q + 1, q + 1] / R[q, q] for q in range(4)]
    J = np.diag(off) + np.diag(sub, 1) + np.diag(sub, -1)
    nodes, vec = np.linalg.eigh(J)
    wts = vec[0] ** 2
    (dx, dy, dz), V = d, d[0] * d[1] * d[2]
    out = [torch.zeros_like(i + j + k) for _ in range(6)]
    for a in range(5):
        x = (i + nodes[a]) * dx
        for b_ in range(5):
            y = (j + nodes[b_]) * dy
            xy2 = x * x + y * y
            for c in range(5):
                z = (k + nodes[c]) * dz
                r2 = xy2 + z * z
                w = (wts[a] * wts[b_] * wts[c] * V / (4 * math.pi)) / (r2 * r2 * torch.sqrt(r2))
                out[0] += w * (r2 - 3 * x * x)
                out[1] += w * (r2 - 3 * y * y)
                out[2] += w * (r2 - 3 * z * z)
                out[3] -= 3 * w * (x * y)
                out[4] -= 3 * w * (x * z)
                out[5] -= 3 * w * (y * z)
    return out


@functools.lru_cache(maxsize=1)
def _tensor_hat(n, d):
    nx, ny, nz = n
    scale = max(d)
    d = tuple(v / scale for v in d)
    i, j, k = (torch.arange(v, device="cuda", dtype=torch.float64).reshape([-1 if a == ax else 1 for a in range(3)])
               for ax, v in ((2, nx), (1, ny), (0, nz)))
    comps = _far(i, j, k, d)
    near = ((i * d[0]) ** 2 + (j * d[1]) ** 2 + (k * d[2]) ** 2 < 100.0).nonzero()
    for c, v in zip(comps, _near(*(near[:, q].double() for q in (2, 1, 0)), d)):
        c[near[:, 0], near[:, 1], near[:, 2]] = v
    parity = ((1, 1, 1), (1, 1, 1), (1, 1, 1), (-1, -1, 1), (-1, 1, -1), (1, -1, -1))    # in x, y, z
    hat = []
    for c, p in zip(comps, parity):
        for ax, v, s in ((2, nx, p[0]), (1, ny, p[1]), (0, nz, p[2])):
            if v > 1:       # offsets 0 .. v-1, one unused place, -(v-1) .. -1
                pad = torch.zeros_like(c.narrow(ax, 0, 1))
                c = torch.cat([c, pad, s * c.narrow(ax, 1, v - 1).flip(ax)], dim=ax)
        hat.append(torch.fft.rfftn(c))
    return hat


class _Plain:
    """The fields of a case in float64."""

    def __init__(self, case, ms):
        self.n, self.d = (case["nx"], case["ny"], case["nz"]), (case["dx"], case["dy"], case["dz"])
        self.c = case
        self.Ms = torch.full((case["nz"], case["ny"], case["nx"]), case["Ms"], device="cuda", dtype=torch.float64) if ms is None else ms.double()
        self.hat = _tensor_hat(self.n, self.d)
        self.pad = [2 * v if v > 1 else 1 for v in self.n[::-1]]

    def demag(self, m):
        M = torch.fft.rfftn(self.Ms * m, s=self.pad, dim=(1, 2, 3))
        xx, yy, zz, xy, xz, yz = self.hat
        H = torch.stack([xx * M[0] + xy * M[1] + xz * M[2], xy * M[0] + yy * M[1] + yz * M[2], xz * M[0] + yz * M[1] + zz * M[2]])
        return -torch.fft.irfftn(H, s=self.pad, dim=(1, 2, 3))[:, :self.n[2], :self.n[1], :self.n[0]]

    def local(self, m):
        c, Ms = self.c, self.Ms
        mag = (Ms > 0).double()
        inv = torch.where(Ms > 0, 1 / Ms.clamp_min(1e-30), torch.zeros_like(Ms))
        H = torch.zeros_like(m)
        dmi = ((0, 1, 0), (-1, 0, 0), (0, 0, 0))      # interfacial: e_y, -e_x, none
        for ax, (h, dv) in enumerate(zip(self.d, dmi)):
            dim, v = 3 - ax, self.n[ax]
            if v == 1:
                continue
            lo, hi = m.narrow(dim, 0, v - 1), m.narrow(dim, 1, v - 1)
            bond = mag.narrow(dim - 1, 0, v - 1) * mag.narrow(dim - 1, 1, v - 1)
            step = 2 * c["A"] / MU0 / h ** 2 * bond * (hi - lo)
            H = H + torch.nn.functional.pad(step, [0, 0] * (3 - dim) + [0, 1]) - torch.nn.functional.pad(step, [0, 0] * (3 - dim) + [1, 0])
            if c["D"] and any(dv):
                w = c["D"] / MU0 / h * bond

                def turn(u):
                    return torch.stack([dv[1] * u[2] - dv[2] * u[1], dv[2] * u[0] - dv[0] * u[2], dv[0] * u[1] - dv[1] * u[0]])
                H = H + torch.nn.functional.pad(w * turn(hi), [0, 0] * (3 - dim) + [0, 1]) - torch.nn.functional.pad(w * turn(lo), [0, 0] * (3 - dim) + [1, 0])
        anis = torch.stack([torch.zeros_like(m[2]), torch.zeros_like(m[2]), 2 * c["Ku"] / MU0 * m[2]])
        return H * inv, anis * inv

    def field(self, m):
        h, a = self.local(m)
        return self.demag(m) + h + a

    def rhs(self, m):
        H, a = self.field(m), self.c["alpha"]
        mh = torch.linalg.cross(m, H, dim=0)
        return -GAMMA / (1 + a * a) * (mh + a * torch.linalg.cross(m, mh, dim=0)) * (self.Ms > 0)

    def unit(self, u):
        return torch.where(self.Ms > 0, u / u.norm(dim=0), u)

    def rk4(self, m, dt, steps):
        for _ in range(steps):
            k1 = self.rhs(m)
            k2 = self.rhs(m + dt / 2 * k1)
            k3 = self.rhs(m + dt / 2 * k2)
            k4 = self.rhs(m + dt * k3)
            m = self.unit(m + dt / 6 * (k1 + 2 * k2 + 2 * k3 + k4))
        return m

    def relax(self, m, t_max, tol=1e-5):
        A = ((), (1 / 4,), (3 / 32, 9 / 32), (1932 / 2197, -7200 / 2197, 7296 / 2197), (439 / 216, -8.0, 3680 / 513, -845 / 4104),
             (-8 / 27, 2.0, -3544 / 2565, 1859 / 4104, -11 / 40))
        b4 = (25 / 216, 0.0, 1408 / 2565, 2197 / 4104, -1 / 5, 0.0)
        b5 = (16 / 135, 0.0, 6656 / 12825, 28561 / 56430, -9 / 50, 2 / 55)
        t, dt = 0.0, min(1e-14, t_max)
        while t < t_max:
            k = []
            for row in A:
                k.append(self.rhs(m + dt * sum(a * v for a, v in zip(row, k)) if row else m))
            err = dt * float(sum((q - p) * v for p, q, v in zip(b4, b5, k)).norm(dim=0).max())
            if err <= tol:
                m, t = self.unit(m + dt * sum(p * v for p, v in zip(b4, k))), t + dt
            dt *= 5.0 if err == 0 else min(5.0, max(0.2, 0.9 * (tol / err) ** 0.2))
            dt = min(dt, t_max - t) if t < t_max else dt
        return m

    def minimize(self, m, iters):
        inv = torch.where(self.Ms > 0, 1 / self.Ms.clamp_min(1e-30), torch.zeros_like(self.Ms))
        old = None
        for it in range(iters):
            h = self.field(m) * inv
            g = torch.linalg.cross(m, torch.linalg.cross(m, h, dim=0), dim=0) * (self.Ms > 0)
            tau = 1e-4
            if old is not None:
                s, y = m - old[0], g - old[1]
                ss, sy, yy = (float((p * q).sum()) for p, q in ((s, s), (s, y), (y, y)))
                tau = ss / sy if it % 2 else sy / yy
                tau = tau if math.isfinite(tau) and tau > 0 else 1.0
            old = (m, g)
            m = self.unit(m - tau * g)
        return m


def exact(case, seed):
    m, ms = _inputs(case, seed)
    m = m.double()
    p = _Plain(case, ms)
    kind = case["kind"]
    if kind == "demag":
        return p.demag(m)
    if kind == "field":
        return p.field(m)
    if kind == "relax":
        return p.relax(m, case["t_max"]), case["t_max"]
    if kind == "rk4":
        return p.rk4(m, case["dt"], case["steps"])
    if kind == "minimize":
        return p.minimize(m, case["steps"])
    if kind == "energy":
        V = case["dx"] * case["dy"] * case["dz"]
        Hd, (hx, ha) = p.demag(m), p.local(m)
        e = [-0.5 * MU0 * V * float((p.Ms * (m * h).sum(0)).sum()) for h in (Hd, hx)]
        ea = -case["Ku"] * V * float(((p.Ms > 0) * m[2] ** 2).sum())
        tq = torch.linalg.cross(m, Hd + hx + ha, dim=0).norm(dim=0)
        tq = torch.where(p.Ms > 0, tq / p.Ms.clamp_min(1e-30), torch.zeros_like(tq))
        return np.array([e[0], e[1], ea, 0.0, 0.0]), float(tq.max())
    m.requires_grad_(True)
    p.Ms.requires_grad_(True)
    out = p.rk4(m, case["dt"], case["steps"])
    lam = (out - torch.tensor(TARGET, dtype=out.dtype, device=out.device).reshape(3, 1, 1, 1)).detach()
    gm, gms = torch.autograd.grad(out, (m, p.Ms), lam)
    return out.detach(), gm, gms
