"""The work a user of this library has it do, as timed cases.

Every case is one call sequence of a real program: start fields in, a number of time steps, density
and velocity out (or, for a restart, the raw state in and out; for the learned closure, training
data and a training epoch).  `listed()` names the sizes of the repository's own configurations,
`draw()` gives more cases of the same ranges.  `exact()` advances the same method in 64 bits with
plain torch, for judging how far the computed fields are from it.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2410_09739_gb300 import fpclbm as F

STORED = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}
BOUNDARY = {"periodic": F.FPCLBM_BC_PERIODIC, "channel": F.FPCLBM_BC_WALLS_Y, "cavity": F.FPCLBM_BC_BOX,
            "half_channel": F.FPCLBM_BC_HALF_CHANNEL}
DIFFUSION = {"fp": F.FPCLBM_DIFF_FP, "mcm": F.FPCLBM_DIFF_EQUILIBRIUM, "learned": F.FPCLBM_DIFF_FP_LEARNED,
             "smagorinsky": F.FPCLBM_DIFF_FP_SMAGORINSKY}
U_STAR = 0.005   # friction velocity of the channels
C_S, A_PLUS = 0.1, 26.0


def _box(name, bc, nx, ny, nz, precision, steps, **more):
    c = {"kind": "box", "bc": bc, "nx": nx, "ny": ny, "nz": nz, "precision": precision, "steps": steps,
         "tau": 0.6, "drift": 0.0, "diffusion": "fp", "re_tau": 0.0, "lid": 0.0, "restart": False}
    c.update(more)
    return {"name": name, **c} if name else c


def listed():
    return [
        # the parity configuration: a small vortex in double precision, 200 steps in one call
        _box("vortex_32_fp64", "periodic", 32, 32, 32, "fp64", 200),
        # a restart of a small ragged box: raw state from the host, steps, raw state back
        _box("restart_45x37x53_fp32", "periodic", 45, 37, 53, "fp32", 512, diffusion="mcm", tau=0.55, restart=True),
        # the headline: Taylor-Green vortex at Re 1600, fp32 and the 16-bit storage that halves its memory
        _box("vortex_256_fp32", "periodic", 256, 256, 256, "fp32", 64, tau=0.50382),
        _box("vortex_256_bf16", "periodic", 256, 256, 256, "bf16", 64, tau=0.50382),
        # general rates of the higher orders (omega_FP = 0.3), fp16 storage, an odd number of steps
        _box("vortex_192_fp16_rates", "periodic", 192, 192, 192, "fp16", 63, tau=0.503, drift=0.3),
        # the Re_tau = 180 channel: walls, body force, bf16 storage
        _box("channel_384x192x192_bf16", "channel", 384, 192, 192, "bf16", 64, tau=0.508, re_tau=180.0),
        # the lid-driven cavity: walls on all faces, a moving lid
        _box("cavity_150_fp32", "cavity", 150, 150, 150, "fp32", 64, tau=0.525981, lid=0.1 / math.sqrt(3.0)),
        # the half-channel large-eddy simulation: Smagorinsky model with van Driest damping
        _box("half_channel_402x64x201_les", "half_channel", 402, 64, 201, "fp32", 64, tau=0.5053333,
             diffusion="smagorinsky", re_tau=180.0),
        # the learned closure on its coarse channel
        _box("learned_192x96x96_bf16", "channel", 192, 96, 96, "bf16", 64, tau=0.5018228, diffusion="learned",
             re_tau=395.0),
        # many small boxes of uneven size and viscosity advanced together (a parameter study)
        {"name": "ensemble_64_fp32", "kind": "ensemble", "boxes": 64, "sides": "32,48,64,96", "pick": 2410,
         "steps": 32},
        # the two-dimensional method on doubly periodic shear layers
        {"name": "shear_layers_4096_fp32", "kind": "d2q9", "nx": 4096, "ny": 4096, "precision": "fp32", "steps": 64,
         "tau": 0.5473, "drift": 0.0, "diffusion": "fp", "lid": 0.0},
        # training data from a fine box and one epoch of training the closure network on it
        {"name": "closure_256_r4", "kind": "closure", "n": 256, "r": 4, "precision": "fp32", "batch": 1024},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dims(rng, cells):
    """Three sides with a product of about `cells`: aspect ratios up to 3, odd and even, multiples of 16 too."""
    s = cells ** (1.0 / 3.0)
    d = [max(8, int(round(s * 3.0 ** rng.uniform(-0.5, 0.5)))) for _ in range(2)]
    d.append(max(8, int(round(cells / (d[0] * d[1])))))
    if rng.random() < 0.5:
        d[0] = max(16, d[0] // 16 * 16)
    return d


def draw(rng):
    what = rng.choice(["vortex", "vortex", "vortex", "channel", "channel", "cavity", "half_channel", "ensemble",
                       "d2q9", "closure"])
    tau = 0.502 + _log_int(rng, 10, 3000) * 1e-4
    if what == "vortex":
        precision = rng.choice(["fp64", "fp32", "fp32", "fp16", "bf16"])
        cells = _log_int(rng, 8e3, 1.2e5 if precision == "fp64" else 1.2e7)
        nx, ny, nz = _dims(rng, cells)
        most = 2.0e7 if precision == "fp64" else 6.0e8
        steps = min(_log_int(rng, 16, 256), max(8, int(most / (nx * ny * nz))))
        return _box(None, "periodic", nx, ny, nz, precision, steps, tau=tau, drift=rng.choice([0.0, 0.0, 0.3]),
                    diffusion=rng.choice(["fp", "fp", "mcm"]), restart=precision == "fp32" and cells < 2e5)
    if what == "channel":
        diffusion = rng.choice(["fp", "fp", "smagorinsky", "learned"])
        nx, ny, nz = _dims(rng, _log_int(rng, 1e5, 1.0e7 if diffusion == "fp" else 4.0e6))
        return _box(None, "channel", nx, ny, nz, rng.choice(["fp32", "bf16"]), rng.randrange(20, 60),
                    tau=0.5 + 3 * U_STAR * (ny / 2) / 395.0, re_tau=395.0, diffusion=diffusion)
    if what == "cavity":
        n = _log_int(rng, 32, 170)
        return _box(None, "cavity", n, n, n, "fp32", rng.randrange(20, 100), tau=max(tau, 0.51),
                    lid=rng.uniform(0.05, 0.2) / math.sqrt(3.0), diffusion=rng.choice(["fp", "mcm"]))
    if what == "half_channel":
        h = _log_int(rng, 24, 72)
        return _box(None, "half_channel", int(round(2 * math.pi * h)), h, int(round(math.pi * h)), "fp32",
                    rng.randrange(20, 60), tau=0.5 + 3 * U_STAR * h / 180.0, re_tau=180.0,
                    diffusion=rng.choice(["smagorinsky", "fp"]))
    if what == "ensemble":
        sides = ",".join(str(rng.randrange(24, 97)) for _ in range(4))
        return {"kind": "ensemble", "boxes": _log_int(rng, 8, 64), "sides": sides, "pick": rng.randrange(10 ** 6),
                "steps": rng.randrange(16, 33)}
    if what == "d2q9":
        precision = rng.choice(["fp64", "fp32", "fp32", "bf16", "fp16"])
        nx = _log_int(rng, 64, 512 if precision == "fp64" else 4096)
        ny = max(32, int(nx * rng.uniform(0.5, 1.0)))
        return {"kind": "d2q9", "nx": nx, "ny": ny, "precision": precision, "steps": rng.randrange(32, 65),
                "tau": tau, "drift": rng.choice([0.0, 0.0, 0.25]), "diffusion": rng.choice(["fp", "mcm"]),
                "lid": rng.choice([0.0, 0.0, 0.05])}
    r = rng.choice([2, 4])
    return {"kind": "closure", "n": r * _log_int(rng, 24, 256 // r), "r": r,
            "precision": rng.choice(["fp32", "bf16"]), "batch": rng.choice([512, 1024, 2048])}


# --- inputs ---------------------------------------------------------------------------------

def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & (2 ** 62 - 1))
    return g


def _uniform(g, shape, lo=-1.0, hi=1.0):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _axes(nx, ny, nz):
    f = lambda n, at: torch.arange(n, device="cuda", dtype=torch.float64).reshape([n if i == at else 1 for i in range(3)])
    return f(nx, 2), f(ny, 1), f(nz, 0)


def _vortex(nx, ny, nz, g, u0=0.05):
    """A Taylor-Green vortex at a seeded phase with its pressure field, and a second, finer wave."""
    x, y, z = _axes(nx, ny, nz)
    ph = _uniform(g, (6,), 0.0, 2 * math.pi).tolist()
    X, Y, Z = (2 * math.pi * a / n + p for a, n, p in ((x, nx, ph[0]), (y, ny, ph[1]), (z, nz, ph[2])))
    ux = u0 * torch.sin(X) * torch.cos(Y) * torch.cos(Z)
    uy = -u0 * torch.cos(X) * torch.sin(Y) * torch.cos(Z)
    uz = 0.2 * u0 * torch.sin(2 * X + ph[3]) * torch.cos(2 * Y + ph[4]) + 0 * Z
    ux = ux + 0.2 * u0 * torch.sin(2 * Z + ph[5])
    rho = 1.0 + 3.0 * u0 * u0 / 16.0 * (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2.0)
    return [rho, ux, uy, uz]


def _channel(nx, ny, nz, g, half):
    """The laminar profile of bulk velocity 16 u*, 10 % noise on every component."""
    _, y, _ = _axes(nx, ny, nz)
    eta = (y + 0.5) / (2 * ny if half else ny)
    ub = 16.0 * U_STAR
    shape, amp = (nz, ny, nx), 0.1 * 1.5 * ub
    ux = 6.0 * ub * eta * (1.0 - eta) + amp * _uniform(g, shape)
    return [torch.ones(shape, device="cuda", dtype=torch.float64), ux, amp * _uniform(g, shape), amp * _uniform(g, shape)]


def _cavity(n, g, lid):
    """A flow that has begun to turn: a vortex that vanishes on the walls, of a seeded strength."""
    x, y, z = _axes(n, n, n)
    X, Y, Z = (math.pi * (a + 0.5) / n for a in (x, y, z))
    a = _uniform(g, (2,), 0.2, 0.5).tolist()
    s = torch.sin(Z) ** 2
    ux = -a[0] * lid * torch.sin(X) ** 2 * torch.sin(2 * Y) * s
    uy = a[0] * lid * torch.sin(2 * X) * torch.sin(Y) ** 2 * s
    uz = 0.1 * a[1] * lid * torch.sin(X) * torch.sin(Y) * torch.sin(2 * Z)
    return [1.0 + 0.001 * torch.cos(X) * torch.cos(Y) * torch.cos(Z), ux, uy, uz]


def _fields(case, seed):
    g = _rng(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["bc"] == "periodic":
        f = _vortex(nx, ny, nz, g)
    elif case["bc"] == "cavity":
        f = _cavity(nx, g, case["lid"])
    else:
        f = _channel(nx, ny, nz, g, case["bc"] == "half_channel")
    return [a.expand(nz, ny, nx).contiguous() for a in f]


def _force(case):
    h = case["ny"] if case["bc"] == "half_channel" else case["ny"] / 2
    return U_STAR ** 2 / h if case["re_tau"] > 0 else 0.0


def _weights(seed):
    """A closure network as training leaves it: standardised inputs folded into the first layer, an
    output that mostly lowers the rate.  bf16 values, in the library's order, as a float64 tensor."""
    g = np.random.default_rng(seed)
    sd = np.array([2e-3] * 6 + [0.03, 0.01, 0.01])
    w1 = g.normal(0, 1 / 3.0, (64, 9)) / sd
    mu = np.array([0.0] * 6 + [0.08, 0.0, 0.0])
    b1 = g.normal(0, 0.1, 64) - w1 @ mu
    w = np.concatenate([w1.ravel(), b1, g.normal(0, 1 / 8.0, 64 * 64), g.normal(0, 0.1, 64),
                        g.normal(0, 0.1 / 8.0, 64), [-0.05]])
    return torch.from_numpy(w).to(torch.bfloat16)


def _ensemble(case):
    r = np.random.default_rng(case["pick"])
    sides = r.choice(np.array([int(s) for s in case["sides"].split(",")]), size=case["boxes"])
    return [int(s) for s in sides], [float(t) for t in r.uniform(0.505, 0.6, size=case["boxes"])]


def _ensemble_fields(case, seed):
    g = _rng(seed)
    sides, _ = _ensemble(case)
    boxes = [[a.expand(s, s, s) for a in _vortex(s, s, s, g, 0.04)] for s in sides]
    return [torch.cat([b[q].reshape(-1) for b in boxes]) for q in range(4)]


def _layers(case, seed):
    """Two shear layers across y, rolled up by a seeded transverse wave; in a closed box a vortex."""
    g = _rng(seed)
    nx, ny = case["nx"], case["ny"]
    x = ((torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5) / nx)[None, :]
    y = ((torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5) / ny)[:, None]
    p = _uniform(g, (2,), 0.0, 1.0).tolist()
    U = 0.2 / math.sqrt(3.0)
    if case["lid"]:
        a = (0.2 + 0.3 * p[0]) * case["lid"]
        ux = -a * torch.sin(math.pi * x) ** 2 * torch.sin(2 * math.pi * y)
        uy = a * torch.sin(2 * math.pi * x) * torch.sin(math.pi * y) ** 2
    else:
        ux = torch.where(y <= 0.5, U * torch.tanh(80 * (y - 0.25)), U * torch.tanh(80 * (0.75 - y))) + 0 * x
        uy = U * 0.05 * torch.sin(2 * math.pi * (x + p[0])) + 0 * y
    rho = 1.0 + 0.002 * torch.cos(2 * math.pi * (x + p[1])) + 0 * y
    return [a.expand(ny, nx).contiguous() for a in (rho, ux, uy)]


# --- the calls -----------------------------------------------------------------------------

def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "box":
        lat = F.Lattice(case["nx"], case["ny"], case["nz"], case["precision"], BOUNDARY[case["bc"]], stream=_stream())
        if case["diffusion"] == "learned":
            lat.set_closure(_weights(seed).view(torch.int16).numpy().view(np.uint16))
        lat.set_params(case["tau"], case["drift"], DIFFUSION[case["diffusion"]])
        if case["diffusion"] == "smagorinsky":
            lat.set_smagorinsky(C_S, U_STAR, A_PLUS)
        if case["re_tau"] > 0:
            lat.set_force(_force(case))
        if case["lid"]:
            lat.set_wall_velocity(case["lid"])
        s["fields"] = [a.reshape(-1) for a in _fields(case, seed)]
        if case["restart"]:
            F.fpclbm_init_fields(lat.h, *s["fields"], on_device=1)
            s["state"], _ = lat.get_state()
    elif case["kind"] == "ensemble":
        sides, taus = _ensemble(case)
        lat = F.Lattice.ensemble([(n, n, n) for n in sides], taus, "fp32", stream=_stream())
        s["fields"] = _ensemble_fields(case, seed)
    elif case["kind"] == "d2q9":
        lat = F.Lattice2D(case["nx"], case["ny"], case["precision"], stream=_stream())
        lat.set_params(case["tau"], 0.0, case["drift"], DIFFUSION[case["diffusion"]])
        if case["lid"]:
            lat.set_boundary(F.FPCLBM_BC_BOX, case["lid"])
        s["fields"] = [a.reshape(-1) for a in _layers(case, seed)]
    else:
        n = case["n"]
        lat = F.Lattice(n, n, n, case["precision"], stream=_stream())
        lat.set_params(0.51)
        f = [a.expand(n, n, n).contiguous().reshape(-1) for a in _eddies(n, _rng(seed))]
        F.fpclbm_init_fields(lat.h, *f, on_device=1)
        nc = (n // case["r"]) ** 3
        s["X"] = torch.empty(nc, 9, device="cuda", dtype=torch.float32)
        s["T"] = torch.empty(nc, device="cuda", dtype=torch.float32)
        s["seed"] = int(seed) % 1000003
    s["lat"] = lat
    if "fields" in s:
        s["out"] = torch.empty(len(s["fields"]), lat.ncells, device="cuda", dtype=torch.float64)
    return s


def run(state):
    case, lat = state["case"], state["lat"]
    if case["kind"] == "closure":
        X, T = state["X"], state["T"]
        F.fpclbm_closure_sample(lat.h, case["r"], TAU_COARSE, X, T, on_device=1)
        w, loss = F.fpclbm_closure_train(X, T, X.shape[0], 1, case["batch"], 1e-3, seed=state["seed"],
                                         stream=_stream())
        return {"features": X, "labels": T, "weights": torch.from_numpy(w.view(np.int16)).view(torch.bfloat16),
                "loss": loss.astype(np.float32)}
    if case["kind"] == "box" and case["restart"]:
        lat.set_state(state["state"], 0)
        lat.step(case["steps"])
        raw, steps = lat.get_state()
        return {"deviations": raw.view(np.float32).reshape(27, -1)[:, :lat.ncells], "steps": steps}
    two = case["kind"] == "d2q9"
    (F.fpclbm2d_init_fields if two else F.fpclbm_init_fields)(lat.h, *state["fields"], on_device=1)
    lat.step(case["steps"])
    out = state["out"]
    (F.fpclbm2d_moments if two else F.fpclbm_moments)(lat.h, *out, on_device=1)
    kept = STORED[case.get("precision", "fp32")]  # the fields in the precision that the run carries
    return {"rho": out[0].to(kept), "u": out[1:].to(kept)}


def _cells(case):
    if case["kind"] == "ensemble":
        return sum(s ** 3 for s in _ensemble(case)[0])
    if case["kind"] == "closure":
        return case["n"] ** 3
    return case["nx"] * case["ny"] * case.get("nz", 1)


def work(case):
    """A step reads and writes every population once; the fields come in and go out in 64 bits.  A
    cell update of the three-dimensional method is about 300 operations (transforms, attractors and
    back), of the two-dimensional one about 60, of the closure network 9,472."""
    n = _cells(case)
    if case["kind"] == "closure":
        b = torch.empty((), dtype=STORED[case["precision"]]).element_size()
        nc = (case["n"] // case["r"]) ** 3
        return {"bytes": n * 27 * b + nc * 40 * 2, "flops": n * 150 + nc * 9472 * 3}
    b = torch.empty((), dtype=STORED[case.get("precision", "fp32")]).element_size()
    q, fields, ops = (9, 3, 60) if case["kind"] == "d2q9" else (27, 4, 300)
    if case.get("diffusion") == "learned":
        ops += 9472
    io = 2 * q * b if case.get("restart") else fields * (8 + 8)
    return {"bytes": n * (2.0 * q * b * case["steps"] + io), "flops": float(n) * ops * case["steps"]}


# --- the same in 64 bits ---------------------------------------------------------------------

TAU_COARSE = 0.505


def _w(i):
    return 2.0 / 3.0 if i == 1 else 1.0 / 6.0


def _rates(tau, drift):
    order = [0, 1, 1, 1] + [2] * 6 + [3] * 7 + [4] * 6 + [5] * 3 + [6]
    om = [1.0 if k <= 1 else 1.0 / tau if k == 2 else (k * drift if drift > 0 else 1.0) for k in order]
    om[7] = 1.0
    return om


def _equilibrium(rho, u):
    """Product form, f[ex + 3 ey + 9 ez] with the indices 0, 1, 2 of e = -1, 0, +1."""
    ph = [[0.5 * (v * v - v) + 1 / 6.0, 2 / 3.0 - v * v, 0.5 * (v * v + v) + 1 / 6.0] for v in u]
    if len(u) == 2:
        return [rho * ph[0][s % 3] * ph[1][s // 3] for s in range(9)]
    return [rho * ph[0][s % 3] * ph[1][(s // 3) % 3] * ph[2][s // 9] for s in range(27)]


def _sums(f, dims):
    rho = sum(f[1:], f[0])
    j = []
    for d in range(dims):
        e = lambda s: (s // 3 ** d) % 3 - 1
        j.append(sum(f[s] for s in range(len(f)) if e(s) > 0) - sum(f[s] for s in range(len(f)) if e(s) < 0))
    return rho, j


def _line(f, d, u, back):
    """One axis of the central-moment transform, in place over the list."""
    st = 3 ** d
    for s in range(len(f)):
        if (s // st) % 3:
            continue
        a, b, c = f[s], f[s + st], f[s + 2 * st]
        if back:
            m1 = b + u * a
            m2 = c + 2.0 * u * b + u * u * a
            f[s], f[s + st], f[s + 2 * st] = 0.5 * (m2 - m1), a - m2, 0.5 * (m2 + m1)
        else:
            p, q = a + c, c - a
            t = p + b
            f[s], f[s + st], f[s + 2 * st] = t, q - u * t, p - 2.0 * u * q + u * u * t


def _network(w, x):
    w = w.double().cuda()
    W1, b1, W2, b2 = w[:576].reshape(64, 9), w[576:640], w[640:4736].reshape(64, 64), w[4736:4800]
    out = []
    for part in x.split(1 << 19):
        h = torch.tanh(part @ W1.T + b1)
        out.append(torch.tanh(h @ W2.T + b2) @ w[4800:4864] + w[4864])
    return torch.cat(out)


def _collide3(f, om, force, mode, net, smag):
    """Appendix D of the paper: central moments, relaxation toward the attractors, back."""
    rho, j = _sums(f, 3)
    ux, uy, uz = ((a + 0.5 * b) / rho for a, b in zip(j, force))
    for d, u in enumerate((ux, uy, uz)):
        _line(f, d, u, False)
    K = lambda m, n, p: f[m + 3 * n + 9 * p]

    def put(m, n, p, v):
        f[m + 3 * n + 9 * p] = v

    w4 = w5 = w6 = w8 = w9 = None
    if net is not None:
        x = torch.stack([K(2, 0, 0) - rho / 3, K(0, 2, 0) - rho / 3, K(0, 0, 2) - rho / 3, K(1, 1, 0), K(1, 0, 1),
                         K(0, 1, 1), ux, uy, uz], -1).reshape(-1, 9)
        w4 = torch.clamp_min(om[4] + torch.clamp_max(_network(net, x).reshape(rho.shape), 0.0), 0.02)
        w5 = w6 = w8 = w9 = w4
    elif smag is not None:
        p = [K(2, 0, 0) - rho / 3, K(0, 2, 0) - rho / 3, K(0, 0, 2) - rho / 3]
        tr = (p[0] + p[1] + p[2]) / 3
        pp = sum((q - tr) ** 2 for q in p) + 2 * (K(1, 1, 0) ** 2 + K(1, 0, 1) ** 2 + K(0, 1, 1) ** 2)
        t0 = 1.0 / om[4]
        w4 = 2.0 / (t0 + torch.sqrt(t0 * t0 + 18.0 * smag * torch.sqrt(2.0 * pp) / rho))
        w5 = w6 = w8 = w9 = w4
    else:
        w4, w5, w6, w8, w9 = om[4], om[5], om[6], om[8], om[9]

    fx, fy, fz = (a / rho for a in force)
    on = any(force)
    S = {}
    if on:
        S = {"120": fx * K(0, 2, 0) + 2 * fy * K(1, 1, 0), "102": fx * K(0, 0, 2) + 2 * fz * K(1, 0, 1),
             "210": 2 * fx * K(1, 1, 0) + fy * K(2, 0, 0), "012": fy * K(0, 0, 2) + 2 * fz * K(0, 1, 1),
             "201": 2 * fx * K(1, 0, 1) + fz * K(2, 0, 0), "021": 2 * fy * K(0, 1, 1) + fz * K(0, 2, 0),
             "111": fx * K(0, 1, 1) + fy * K(1, 0, 1) + fz * K(1, 1, 0),
             "220": 2 * (fx * K(1, 2, 0) + fy * K(2, 1, 0)), "202": 2 * (fx * K(1, 0, 2) + fz * K(2, 0, 1)),
             "022": 2 * (fy * K(0, 1, 2) + fz * K(0, 2, 1)),
             "211": 2 * fx * K(1, 1, 1) + fy * K(2, 0, 1) + fz * K(2, 1, 0),
             "121": fx * K(0, 2, 1) + 2 * fy * K(1, 1, 1) + fz * K(1, 2, 0),
             "112": fx * K(0, 1, 2) + fy * K(1, 0, 2) + 2 * fz * K(1, 1, 1),
             "122": fx * K(0, 2, 2) + 2 * (fy * K(1, 1, 2) + fz * K(1, 2, 1)),
             "212": fy * K(2, 0, 2) + 2 * (fx * K(1, 1, 2) + fz * K(2, 1, 1)),
             "221": fz * K(2, 2, 0) + 2 * (fx * K(1, 2, 1) + fy * K(2, 1, 1)),
             "222": 2 * (fx * K(1, 2, 2) + fy * K(2, 1, 2) + fz * K(2, 2, 1))}
    src = lambda name: S.get(name, 0.0)
    relax = lambda y, a, i, s: y + om[i] * (a - y) + (1.0 - 0.5 * om[i]) * s

    for (m, n, p), a in zip(((1, 0, 0), (0, 1, 0), (0, 0, 1)), force):
        put(m, n, p, K(m, n, p) + a)
    # order 2
    a, b, c = K(2, 0, 0), K(0, 2, 0), K(0, 0, 2)
    t1 = relax(a + b + c, rho, 7, 0.0)
    t2, t3 = (1 - w8) * (a - b), (1 - w9) * (a - c)
    A, B, C = (t1 + t2 + t3) / 3, (t1 - 2 * t2 + t3) / 3, (t1 + t2 - 2 * t3) / 3
    put(2, 0, 0, A), put(0, 2, 0, B), put(0, 0, 2, C)
    p, q, r = (1 - w4) * K(1, 1, 0), (1 - w5) * K(1, 0, 1), (1 - w6) * K(0, 1, 1)
    put(1, 1, 0, p), put(1, 0, 1, q), put(0, 1, 1, r)
    # order 3
    for i, (x, y) in zip((10, 12, 14), (("120", "102"), ("210", "012"), ("201", "021"))):
        X, Y = K(*map(int, x)), K(*map(int, y))
        s = relax(X + Y, 0.0, i, src(x) + src(y))
        d = relax(X - Y, 0.0, i + 1, src(x) - src(y))
        put(*map(int, x), 0.5 * (s + d)), put(*map(int, y), 0.5 * (s - d))
    put(1, 1, 1, relax(K(1, 1, 1), 0.0, 16, src("111")))
    # order 4
    mcm = mode == "mcm"
    zero = torch.zeros_like(rho)
    a4 = {"220": rho / 9 if mcm else (A * B + 2 * p * p) / rho, "202": rho / 9 if mcm else (A * C + 2 * q * q) / rho,
          "022": rho / 9 if mcm else (B * C + 2 * r * r) / rho, "211": zero if mcm else (A * r + 2 * p * q) / rho,
          "121": zero if mcm else (B * q + 2 * p * r) / rho, "112": zero if mcm else (C * p + 2 * r * q) / rho}
    x, y, z = K(2, 2, 0), K(2, 0, 2), K(0, 2, 2)
    ax, ay, az = a4["220"], a4["202"], a4["022"]
    sx, sy, sz = src("220"), src("202"), src("022")
    t1 = relax(x + y + z, ax + ay + az, 17, sx + sy + sz)
    t2 = relax(x + y - z, ax + ay - az, 18, sx + sy - sz)
    t3 = relax(x - y, ax - ay, 19, sx - sy)
    put(2, 2, 0, 0.25 * (t1 + t2 + 2 * t3)), put(2, 0, 2, 0.25 * (t1 + t2 - 2 * t3)), put(0, 2, 2, 0.5 * (t1 - t2))
    for i, name in ((20, "211"), (21, "121"), (22, "112")):
        put(*map(int, name), relax(K(*map(int, name)), a4[name], i, src(name)))
    # order 5
    k111 = K(1, 1, 1)
    a5 = {"122": B * K(1, 0, 2) + C * K(1, 2, 0) + 4 * r * k111 + 2 * (q * K(0, 2, 1) + p * K(0, 1, 2)),
          "212": A * K(0, 1, 2) + C * K(2, 1, 0) + 4 * q * k111 + 2 * (p * K(1, 0, 2) + r * K(2, 0, 1)),
          "221": A * K(0, 2, 1) + B * K(2, 0, 1) + 4 * p * k111 + 2 * (r * K(2, 1, 0) + q * K(1, 2, 0))}
    for i, name in ((23, "122"), (24, "212"), (25, "221")):
        put(*map(int, name), relax(K(*map(int, name)), zero if mcm else 0.4 * a5[name] / rho, i, src(name)))
    # order 6
    a6 = rho / 27 if mcm else (A * K(0, 2, 2) + B * K(2, 0, 2) + C * K(2, 2, 0) +
                               4 * (p * K(1, 1, 2) + q * K(1, 2, 1) + r * K(2, 1, 1))) / (3 * rho)
    put(2, 2, 2, relax(K(2, 2, 2), a6, 26, src("222")))
    for d, u in ((2, uz), (1, uy), (0, ux)):
        _line(f, d, u, True)


def _stream3(f, bc, lid):
    """Streaming with wrap, half-way bounce-back (a moving lid's correction) or the symmetry plane."""
    w = [_w(s % 3) * _w((s // 3) % 3) * _w(s // 9) for s in range(27)]
    if bc == "cavity":
        rho = sum((a[:, -1, :] for a in f[1:]), f[0][:, -1, :])
        for s in range(27):
            if (s // 3) % 3 == 2 and s % 3 != 1:
                f[s][:, -1, :] -= 6.0 * w[s] * rho * (s % 3 - 1) * lid
    out = []
    for s in range(27):
        e = (s % 3 - 1, (s // 3) % 3 - 1, s // 9 - 1)
        g = torch.roll(f[s], (e[2], e[1], e[0]), (0, 1, 2))
        back = f[26 - s]
        cut = lambda d: slice(0, 1) if e[d] > 0 else slice(-1, None)
        if bc != "periodic" and e[1]:
            if bc == "half_channel" and e[1] < 0:
                g[:, -1:, :] = torch.roll(f[s + 6], (e[2], e[0]), (0, 2))[:, -1:, :]
            else:
                g[:, cut(1), :] = back[:, cut(1), :]
        if bc == "cavity":
            if e[0]:
                g[:, :, cut(0)] = back[:, :, cut(0)]
            if e[2]:
                g[cut(2), :, :] = back[cut(2), :, :]
        out.append(g)
    return out


def _collide2(f, om, mode):
    rho, j = _sums(f, 2)
    ux, uy = j[0] / rho, j[1] / rho
    _line(f, 0, ux, False)
    _line(f, 1, uy, False)
    s = f[2] + f[6]
    s, d = s + om[3] * (2.0 / 3.0 * rho - s), (1 - om[4]) * (f[2] - f[6])
    f[4] = (1 - om[5]) * f[4]
    f[2], f[6] = 0.5 * (s + d), 0.5 * (s - d)
    f[5], f[7] = (1 - om[6]) * f[5], (1 - om[7]) * f[7]
    a = rho / 9 if mode == "mcm" else (f[2] * f[6] + 2 * f[4] ** 2) / rho
    f[8] = f[8] + om[8] * (a - f[8])
    _line(f, 1, uy, True)
    _line(f, 0, ux, True)


def _stream2(f, lid):
    if lid:
        rho = sum((a[-1] for a in f[1:]), f[0][-1])
        for s in (6, 8):
            f[s][-1] -= 6.0 * _w(s % 3) * _w(2) * rho * (s % 3 - 1) * lid
    out = []
    for s in range(9):
        ex, ey = s % 3 - 1, s // 3 - 1
        g = torch.roll(f[s], (ey, ex), (0, 1))
        if lid:
            if ey:
                at = slice(0, 1) if ey > 0 else slice(-1, None)
                g[at] = f[8 - s][at]
            if ex:
                at = slice(0, 1) if ex > 0 else slice(-1, None)
                g[:, at] = f[8 - s][:, at]
        out.append(g)
    return out


def _damping(case):
    """(C_s D)^2 per row, D the van Driest factor of the distance to the nearest wall."""
    ny = case["ny"]
    y = torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5
    y = torch.minimum(y, ny - y) if case["bc"] == "channel" else y
    nu = (case["tau"] - 0.5) / 3.0
    return ((C_S * (1.0 - torch.exp(-(y * U_STAR / nu) / A_PLUS))) ** 2)[None, :, None]


def _read(f, force=(0.0, 0.0, 0.0)):
    dims = 2 if len(f) == 9 else 3
    rho, j = _sums(f, dims)
    return rho.reshape(-1), torch.stack([((a + 0.5 * b) / rho).reshape(-1) for a, b in zip(j, force)])


def _exact_box(case, fields, tau, net=None):
    om = _rates(tau, case["drift"])
    force = (_force(case), 0.0, 0.0)
    smag = _damping(case) if case["diffusion"] == "smagorinsky" else None
    f = _equilibrium(fields[0], fields[1:])
    for _ in range(case["steps"]):
        _collide3(f, om, force, case["diffusion"], net, smag)
        f = _stream3(f, case["bc"], case["lid"])
    return f, force


def _eddies(n, g, count=12):
    """A sum of seeded solenoidal waves of wavenumbers 1 to 8."""
    x, y, z = _axes(n, n, n)
    X, Y, Z = (2 * math.pi * a / n for a in (x, y, z))
    u = [0.0, 0.0, 0.0]
    for _ in range(count):
        k = [int(v) for v in torch.randint(1, 9, (3,), generator=g, device="cuda").tolist()]
        p = _uniform(g, (3,), 0.0, 2 * math.pi).tolist()
        a = _uniform(g, (3,)).tolist()
        dot = sum(s * t for s, t in zip(a, k)) / sum(t * t for t in k)
        a = [s - dot * t for s, t in zip(a, k)]
        # cos(k.x + p) by parts, so that only products of one-axis waves are formed
        c = torch.cos(k[0] * X + p[0]) * torch.cos(k[1] * Y + p[1]) - torch.sin(k[0] * X + p[0]) * torch.sin(k[1] * Y + p[1])
        s = torch.sin(k[0] * X + p[0]) * torch.cos(k[1] * Y + p[1]) + torch.cos(k[0] * X + p[0]) * torch.sin(k[1] * Y + p[1])
        wave = c * torch.cos(k[2] * Z + p[2]) - s * torch.sin(k[2] * Z + p[2])
        for d in range(3):
            u[d] = u[d] + 0.02 * a[d] * wave
    return [torch.ones_like(u[0])] + u


def _exact_closure(case, seed):
    n, r = case["n"], case["r"]
    m = n // r
    rho, *u = _eddies(n, _rng(seed))
    box = lambda a: a.reshape(m, r, m, r, m, r).mean((1, 3, 5))
    U = [box(a) for a in u]
    R = box(rho)
    # array axes are z, y, x: component j varies along axis 2 - j
    grad = [[0.5 * (torch.roll(U[i], -1, 2 - j) - torch.roll(U[i], 1, 2 - j)) for j in range(3)] for i in range(3)]
    S = [[0.5 * (grad[i][j] + grad[j][i]) for j in range(3)] for i in range(3)]
    tau = [[box(u[i] * u[j]) - U[i] * U[j] for j in range(3)] for i in range(3)]
    tr = (tau[0][0] + tau[1][1] + tau[2][2]) / 3
    num = sum((tau[i][j] - (tr if i == j else 0.0)) * S[i][j] for i in range(3) for j in range(3))
    den = sum(S[i][j] ** 2 for i in range(3) for j in range(3))
    nut = torch.clamp_min(torch.where(den > 0, -num / (2 * den), torch.zeros_like(den)), 0.0)
    nu = (TAU_COARSE - 0.5) / 3
    label = 1.0 / (3 * (nu + nut) + 0.5) - 1.0 / (3 * nu + 0.5)
    c = -2.0 * R * TAU_COARSE / 3
    X = torch.stack([c * S[0][0], c * S[1][1], c * S[2][2], c * S[0][1], c * S[0][2], c * S[1][2], *U], -1)
    # the order of the samples and the first weights are the library's own draws: no value for those outputs
    return {"features": X.reshape(-1, 9), "labels": label.reshape(-1), "weights": None, "loss": None}


def exact(case, seed):
    if case["kind"] == "closure":
        return _exact_closure(case, seed)
    if case["kind"] == "d2q9":
        fields = _layers(case, seed)
        om = [1.0] * 9
        om[4] = om[5] = 1.0 / case["tau"]
        if case["drift"] > 0:
            om[6] = om[7] = 3.0 * case["drift"]
            om[8] = 4.0 * case["drift"]
        f = _equilibrium(fields[0], fields[1:])
        for _ in range(case["steps"]):
            _collide2(f, om, case["diffusion"])
            f = _stream2(f, case["lid"])
        rho, u = _read(f)
        return {"rho": rho, "u": u}
    if case["kind"] == "ensemble":
        sides, taus = _ensemble(case)
        flat = _ensemble_fields(case, seed)
        one = {"drift": 0.0, "diffusion": "fp", "bc": "periodic", "lid": 0.0, "re_tau": 0.0, "ny": 1,
               "steps": case["steps"]}
        at, got = 0, []
        for s, tau in zip(sides, taus):
            f, _ = _exact_box(one, [a[at:at + s ** 3].reshape(s, s, s) for a in flat], tau)
            got.append(_read(f))
            at += s ** 3
        return {"rho": torch.cat([a for a, _ in got]), "u": torch.cat([b for _, b in got], 1)}
    net = _weights(seed) if case["diffusion"] == "learned" else None
    f, force = _exact_box(case, _fields(case, seed), case["tau"], net)
    if case["restart"]:
        w = [_w(s % 3) * _w((s // 3) % 3) * _w(s // 9) for s in range(27)]
        dev = [a - b for a, b in zip(f, w)]
        if case["steps"] % 2:  # after an odd step count a slot holds what left its cell in the opposite direction
            dev = [torch.roll(dev[26 - s], ((s // 9 - 1), ((s // 3) % 3 - 1), (s % 3 - 1)), (0, 1, 2)) for s in range(27)]
        return {"deviations": torch.stack([a.reshape(-1) for a in dev]), "steps": None}
    rho, u = _read(f, force)
    return {"rho": rho, "u": u}
