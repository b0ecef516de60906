"""Performance cases of the PRC-LBM library: what its users have it do.

A single solve starts from given macroscopic fields, advances a number of time
steps and hands the fields back, all on the device; a batch advances many
uneven cavities by one chunk, as a solve server does between two looks at its
queue.  Every case goes through the public binding (``paper_2208_03562_gb300.lbm``).

``exact`` states the same runs in FP64 torch operations, from the moment
definitions of arXiv:2208.03562 (Sec. 4.2, Eqs. 12-14, 38-48), without the
library.
"""
import math

import numpy as np
import torch

from paper_2208_03562_gb300 import inputs as I
from paper_2208_03562_gb300 import lbm as L

BC = {"cavity": L.BC_CAVITY, "channel": L.BC_CHANNEL, "periodic": L.BC_PERIODIC}
ELEM = {"f64": 8, "f32": 4, "f16": 2}
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPPOSITE = (0, 3, 4, 1, 2, 7, 8, 5, 6)
FLOPS = 220          # floating-point operations of one node update (an fma counts two)
MAX_NODE_STEPS = 6.5e8


def single(name, dtype, nx, ny, r, gamma, nu, u_lid, calls, steps, bc="cavity", fx=0.0):
    return {"name": name, "kind": "single", "dtype": dtype, "nx": nx, "ny": ny, "r": r, "gamma": gamma, "nu": nu,
            "u_lid": u_lid, "bc": bc, "fx": fx, "calls": calls, "steps": steps}


def listed():
    c1, c2, c3, c3h = (I.square_cavity_64(), I.deep_cavity_128(), I.shallow_cavity_8192x2048("f32"),
                       I.shallow_cavity_8192x2048("f16"))
    deep = I.Cavity(100, 150, 4.0 / 3.0, 1.0, 1000.0, 0.06 * I.CS_STAR)
    u02 = 0.06 * 0.2 * I.CS_STAR
    return [
        # the validation cavity in FP64, a stretch of its run to steady state
        single("f64 64x64 run", "f64", c1.nx, c1.ny, c1.r, c1.gamma, c1.nu, c1.u_lid, "run", 200),
        # the paper's deep cavity at Re 1000 without preconditioning, FP64: the plain arm of the step-count study
        single("f64 100x150 run", "f64", 100, 150, deep.r, 1.0, deep.nu, deep.u_lid, "run", 100),
        # a 512-wide FP64 reference run against which reduced precision is checked
        single("f64 512x128 step", "f64", 512, 128, 0.5, 0.25, 0.05 * 64 / 500.0, 0.05, "step", 40),
        # a program that watches the residual of a small preconditioned cavity: many short calls
        single("f32 128x128 poll", "f32", c2.nx, c2.ny, c2.r, c2.gamma, c2.nu, c2.u_lid, "poll", 200),
        # the square-lattice grid of the rectangular-versus-square study
        single("f32 400x100 run", "f32", 400, 100, 1.0, 1.0, 0.06 * I.CS_STAR, 0.06 * I.CS_STAR, "run", 400),
        # the FP16 transient of the precision schedule on the paper's shallow cavity (odd row count)
        single("f16 100x125 run", "f16", 100, 125, 0.2, 0.1, u02 * 25.0 / 100.0, u02, "run", 1000),
        # one cavity of the sweep's upper end, odd sizes
        single("f32 1023x511 step", "f32", 1023, 511, 0.5, 0.25, 0.05 * 255.5 / 1000.0, 0.05, "step", 100),
        # body-force-driven channel: periodic in x, odd row count
        single("f32 channel 512x257", "f32", 512, 257, 0.5, 0.5, 0.02, 0.01, "step", 100, "channel", 1e-6),
        # the throughput workload, FP32 and FP16 storage
        single("f32 8192x2048 step", "f32", c3.nx, c3.ny, c3.r, c3.gamma, c3.nu, c3.u_lid, "step", 40),
        single("f16 8192x2048 step", "f16", c3h.nx, c3h.ny, c3h.r, c3h.gamma, c3h.nu, c3h.u_lid, "step", 40),
        # 24 uneven cavities of the batched sweep, one chunk
        {"name": "batch sweep f32", "kind": "batch", "dtype": "f32", "mix": "sweep", "mix_seed": 0, "count": 24,
         "steps": 200},
        # what a solve server holds: a few requests of the serving mix in FP16, one chunk
        {"name": "batch serving f16", "kind": "batch", "dtype": "f16", "mix": "serving", "mix_seed": 0, "count": 6,
         "steps": 100},
    ]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a batch in one of five, else a single solve of any size,
    storage type and wall type of the ranges above."""
    if rng.random() < 0.2:
        mix = rng.choice(("sweep", "serving"))
        c = {"kind": "batch", "dtype": rng.choice(("f32", "f16")), "mix": mix, "mix_seed": rng.randrange(1, 10 ** 6),
             "count": rng.randint(2, 24) if mix == "sweep" else rng.randint(1, 6)}
        nodes = sum(q[0] * q[1] for q in cavities(c))
        c["steps"] = 20 * max(1, min(10, int(MAX_NODE_STEPS / nodes / 20.0)))
        return c
    dtype = rng.choice(("f32", "f32", "f16", "f64"))
    nx, ny = log_int(rng, 48, 8192), log_int(rng, 32, 2048)
    r = math.exp(rng.uniform(math.log(0.2), math.log(2.0)))
    gamma = math.exp(rng.uniform(math.log(0.1), 0.0))
    bc = rng.choice(("cavity", "cavity", "cavity", "channel", "periodic"))
    u = I.lid_speed_for_mach(r, I.sweep_mach(gamma))
    nu = stable_nu(r, gamma, u * ny * r / math.exp(rng.uniform(math.log(100.0), math.log(1000.0))))
    most = MAX_NODE_STEPS / (40.0 if dtype == "f64" else 1.0) / (nx * ny)
    steps = 20 * max(1, min(20, int(most / 20.0)))
    c = single("", dtype, nx, ny, r, gamma, nu, 0.0 if bc == "periodic" else u, rng.choice(("run", "step", "poll")),
               steps, bc, 1e-6 if bc == "channel" else 0.0)
    del c["name"]
    return c


def stable_nu(r, gamma, nu):
    """The viscosity, raised where the shear relaxation rate would pass 1.75,
    so that a run of any length stays finite."""
    return max(nu, gamma * min(1.0, r) ** 2 / 3.0 * (1.0 / 1.75 - 0.5))


def cavities(case):
    """The cavities of a case's mix: (nx, ny, r, gamma, nu, u_lid)."""
    if case["mix"] == "sweep":
        cs = I.batched_sweep(case["mix_seed"], case["count"])
    else:
        cs = [q.cavity for q in I.serving_requests(case["mix_seed"], case["count"])]
    return [(c.nx, c.ny, c.r, c.gamma, stable_nu(c.r, c.gamma, c.nu), c.u_lid) for c in cs]


def start_fields(seed, nx, ny, r, gamma):
    """A smooth random flow at a fraction of the sweeps' Mach number, on the GPU."""
    g = I.rng(seed)
    x = (torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) * (2 * math.pi / nx)
    y = (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) * (2 * math.pi / ny)
    u = I.lid_speed_for_mach(r, I.sweep_mach(gamma))
    out = []
    for amp in (5e-4, 0.25 * u, 0.25 * u):
        f = torch.zeros((ny, nx), dtype=torch.float64, device="cuda")
        for k in range(1, 4):
            a, px, py = float(g.standard_normal()), float(g.uniform(0, 6.28)), float(g.uniform(0, 6.28))
            f += (amp * a / k) * torch.outer(torch.sin(k * y + py), torch.cos(int(g.integers(1, 4)) * x + px))
        out.append(f)
    out[0] += 1.0
    return out


def params_of(case):
    return L.lbm_params_init(case["nx"], case["ny"], case["r"], case["gamma"], case["nu"], case["u_lid"],
                             L.DTYPE_CODES[case["dtype"]], bc=BC[case["bc"]], fx=case["fx"])


def init_from_device(h, fields):
    s = L.load().lbm_init_fields(h.h, *[f.data_ptr() for f in fields], 1)
    if s != L.OK:
        raise L.LbmError(s, "lbm_init_fields")


def prepare(case, seed):
    if case["kind"] == "single":
        fields = start_fields(seed, case["nx"], case["ny"], case["r"], case["gamma"])
        torch.cuda.synchronize()
        return {"case": case, "h": L.Lbm(params_of(case)), "fields": fields,
                "out": [torch.empty_like(f) for f in fields]}
    dtype = L.DTYPE_CODES[case["dtype"]]
    mix = cavities(case)
    b = L.Batch(len(mix), dtype)
    nodes = [c[0] * c[1] for c in mix]
    for k, (nx, ny, r, gamma, nu, u) in enumerate(mix):
        p = L.lbm_params_init(nx, ny, r, gamma, nu, u, dtype)
        fields = start_fields(seed + 1000 * k, nx, ny, r, gamma)
        f = torch.empty((9, ny, nx), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        h = L.Lbm(p)
        init_from_device(h, fields)
        s = L.load().lbm_get_populations(h.h, f.data_ptr(), 1)
        h.close()
        if s != L.OK:
            raise L.LbmError(s, "lbm_get_populations")
        b.set_populations_from_device(b.add(p, 0.0, 10 ** 12), f.data_ptr())
    return {"case": case, "b": b, "nodes": nodes,
            "out": [torch.empty(sum(nodes), dtype=torch.float64, device="cuda") for _ in range(3)]}


def run(state):
    case, out, n = state["case"], state["out"], state["case"]["steps"]
    if case["kind"] == "single":
        h = state["h"]
        init_from_device(h, state["fields"])
        if case["calls"] == "run":     # towards a tolerance that this stretch does not reach
            h.run(1e-30, n)
        elif case["calls"] == "step":
            h.step(n)
        else:                          # a look at the residual every 20 steps
            for _ in range(n // 20):
                h.step(20)
                h.residual()
        L.lbm_fields_device(h.h, *[v.data_ptr() for v in out])
        return {"rho": out[0], "ux": out[1], "uy": out[2], "residual": h.residual()}
    b, at = state["b"], 0
    b.run(n)
    for slot, nodes in enumerate(state["nodes"]):
        s = L.load().lbm_batch_fields(b.b, slot, *[v.data_ptr() + 8 * at for v in out], 1)
        if s != L.OK:
            raise L.LbmError(s, "lbm_batch_fields")
        at += nodes
    return {"rho": out[0], "ux": out[1], "uy": out[2],
            "residual": np.array([b.query(k)[0].residual for k in range(len(state["nodes"]))])}


def work(case):
    if case["kind"] == "single":
        nodes, moved = case["nx"] * case["ny"], 48    # three FP64 fields in, three out
    else:
        nodes = sum(c[0] * c[1] for c in cavities(case))
        moved = 18 * ELEM[case["dtype"]] + 24         # the state in and out, three FP64 fields out
    return {"bytes": nodes * moved, "flops": nodes * case["steps"] * FLOPS}


# ---------------------------------------------------------------------------
# the same runs in FP64 torch operations

def from_moments(m, r):
    """Populations of the raw moments m[a][b] = sum f c_x^a c_y^b."""
    x = [(m[0][b] - m[2][b], 0.5 * (m[2][b] + m[1][b]), 0.5 * (m[2][b] - m[1][b])) for b in range(3)]
    f = [None] * 9
    for i in range(9):
        a, b, c = (x[k][EX[i]] for k in range(3))    # index -1 is the last entry: e_x = -1
        f[i] = a - c / r ** 2 if EY[i] == 0 else 0.5 * (c / r ** 2 + EY[i] * b / r)
    return torch.stack(f)


def equilibrium(rho, ux, uy, r, g, c2):
    a, b = ux * ux, uy * uy
    return from_moments([[rho, rho * uy, c2 * rho + rho * b / g],
                         [rho * ux, rho * ux * uy / g, rho * (c2 + b / g ** 2) * ux],
                         [c2 * rho + rho * a / g, rho * (c2 + a / g ** 2) * uy,
                          rho * (c2 * c2 + c2 * (a + b) + a * b)]], r)


def velocity(f, r, fx, g):
    rho = f.sum(0)
    jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7])
    jy = r * ((f[2] - f[4]) + (f[5] + f[6]) - (f[7] + f[8]))
    return rho, (jx + fx / (2 * g)) / rho, jy / rho


def stream(ft, bc, lid):
    f = torch.empty_like(ft)
    for i in range(9):
        f[i] = torch.roll(ft[i], (EY[i], EX[i]), (0, 1))
    for i in range(1, 9):
        if bc != "periodic" and EY[i]:
            y = 0 if EY[i] > 0 else -1
            f[i, y] = ft[OPPOSITE[i], y]
            if y == -1 and EX[i]:
                f[i, y] += EX[i] * lid
        if bc == "cavity" and EX[i]:
            x = 0 if EX[i] > 0 else -1
            f[i, :, x] = ft[OPPOSITE[i], :, x]
            if EY[i] < 0:
                f[i, -1, x] += EX[i] * lid
    return f


def gradients(rho, bc, r):
    """Isotropic second-order differences, zero normal gradient at walls."""
    p = torch.nn.functional.pad(rho[None, None], (1, 1, 0, 0), "replicate" if bc == "cavity" else "circular")
    p = torch.nn.functional.pad(p, (0, 0, 1, 1), "circular" if bc == "periodic" else "replicate")[0, 0]
    e, w, c = p[:, 2:], p[:, :-2], p[:, 1:-1]
    dx, dy = e - w, p[2:] - p[:-2]
    return ((4 * dx[1:-1] + dx[2:] + dx[:-2]) / 12,
            (4 * dy[:, 1:-1] + dy[:, 2:] + dy[:, :-2]) / (12 * r))


def collide(f, dxr, dyr, r, g, c2, wn, fx):
    """Central moments about u, relaxed towards the corrected preconditioned
    equilibria (bulk rate and higher-order rates 1)."""
    rho, ux, uy = velocity(f, r, fx, g)
    c = [[0.0] * 3 for _ in range(3)]
    for i in range(9):
        px, py = EX[i] - ux, r * EY[i] - uy
        c[2][0] = c[2][0] + f[i] * px * px
        c[0][2] = c[0][2] + f[i] * py * py
        c[1][1] = c[1][1] + f[i] * px * py
    a, b = ux * ux, uy * uy
    P, Q, U, h = 4 / g ** 2 - 1 / g, 1 / g ** 2 - 1 / g, 2 / g + 1, 1 / g - 1
    s, d = c[2][0] + c[0][2], c[2][0] - c[0][2]
    A, B = 0.5 * (U * c2 - 1) * ux * dxr, 0.5 * (U * c2 - r * r) * uy * dyr
    Rs, Rd = s - 2 * c2 * rho - h * (a + b) * rho - A - B, d - h * (a - b) * rho - A + B
    kx, ky = 3 * c2 - 1, 3 * c2 - r * r
    bx, by = (-2 * c2 + (P * a + Q * b + kx) / 2) * rho, (-2 * c2 + (P * b + Q * a + ky) / 2) * rho
    sx, sy = (-2 * c2 / wn + (P * a - Q * b + kx) / 2) * rho, (2 * c2 / wn + (-P * b + Q * a - ky) / 2) * rho
    X = (sy * Rs - by * Rd) / (bx * sy - sx * by)
    Y = (Rs - bx * X) / by
    t = 1 / wn - 0.5
    es = 2 * c2 * rho + h * rho * (a + b) - 0.5 * rho * ((P * a + Q * b + kx) * X + (P * b + Q * a + ky) * Y) - A - B
    ed = h * rho * (a - b) - t * (rho * ((P * a - Q * b + kx) * X + (-P * b + Q * a - ky) * Y) + 2 * A - 2 * B)
    e11 = h * rho * ux * uy - t * (Q * rho * ux * uy * (X + Y) + h * c2 * (uy * dxr + ux * dyr))
    ts = es + 0.5 * 2 * Q * fx * ux
    td = d + wn * (ed - d) + (1 - wn / 2) * 2 * Q * fx * ux
    t11 = c[1][1] + wn * (e11 - c[1][1]) + (1 - wn / 2) * Q * fx * uy
    t10 = fx / (2 * g)
    a3 = 1 / g ** 2 - 3 / g + 2
    t20, t02, t21, t12, t22 = (ts + td) / 2, (ts - td) / 2, a3 * rho * a * uy, a3 * rho * ux * b, c2 * c2 * rho
    m = [[rho, rho * uy, t02 + rho * b],
         [t10 + rho * ux, t11 + t10 * uy + rho * ux * uy, t12 + 2 * uy * t11 + ux * t02 + t10 * b + rho * ux * b],
         [t20 + 2 * ux * t10 + rho * a, t21 + 2 * ux * t11 + uy * t20 + 2 * ux * uy * t10 + rho * a * uy,
          t22 + 2 * uy * t21 + 2 * ux * t12 + a * t02 + b * t20 + 4 * ux * uy * t11 + 2 * ux * b * t10 +
          rho * a * b]]
    return from_moments(m, r)


def exact_run(fields, nx, ny, r, g, nu, u_lid, steps, bc="cavity", fx=0.0):
    c2 = min(1.0, r) ** 2 / 3.0
    wn = 1.0 / (nu / (g * c2) + 0.5)
    f = equilibrium(*fields, r, g, c2)
    before = None
    for k in range(steps):
        if k == steps - 20:
            before = velocity(f, r, -fx, g)[1] if k else fields[1]
        f = stream(f, bc, c2 * u_lid / (2 * r * r))
        dxr, dyr = gradients(f.sum(0), bc, r)
        f = collide(f, dxr, dyr, r, g, c2, wn, fx)
    rho, ux, uy = velocity(f, r, -fx, g)
    return rho, ux, uy, float((ux - before).square().sum().sqrt())


def exact(case, seed):
    # in FP16 the residual of a few steps is mostly the storage's rounding noise
    with_residual = case["dtype"] != "f16"
    if case["kind"] == "single":
        fields = start_fields(seed, case["nx"], case["ny"], case["r"], case["gamma"])
        rho, ux, uy, res = exact_run(fields, case["nx"], case["ny"], case["r"], case["gamma"], case["nu"],
                                     case["u_lid"], case["steps"], case["bc"], case["fx"])
        return {"rho": rho, "ux": ux, "uy": uy, "residual": res if with_residual else None}
    parts = []
    for k, (nx, ny, r, gamma, nu, u) in enumerate(cavities(case)):
        parts.append(exact_run(start_fields(seed + 1000 * k, nx, ny, r, gamma), nx, ny, r, gamma, nu, u,
                               case["steps"]))
    cat = [torch.cat([p[q].reshape(-1) for p in parts]) for q in range(3)]
    return {"rho": cat[0], "ux": cat[1], "uy": cat[2],
            "residual": np.array([p[3] for p in parts]) if with_residual else None}
