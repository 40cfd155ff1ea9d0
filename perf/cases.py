"""The work that a user of libpf has it do, as measurable cases.

Six kinds of program, each through the package's public entry points:
  grid      a Sim restarted from a checkpoint held on the GPU, stepped and read
            back on the GPU (set_clock, set_fields, step, get_fields)
  energies  the same with F_h recorded after every step (step_energies)
  monitor   the diagnostics of a state: energy, solute_total, front
  stream    states that arrive from page-locked host memory, one step each, the
            stepped fields going back to page-locked host memory
  batch     many 1D pulled fronts at once (run_batch)
  adjoint   the derivatives of their partition coefficients (adjoint)

exact() restates the model in plain 64-bit torch, for the same discretisation:
centred cell gradients, fluxes at faces from one-sided normal and averaged
transverse differences, the conservative (c, d) update, forward Euler.
"""
import math

import numpy as np
import torch

from paper_2303_09671_gb300 import pf
from paper_2303_09671_gb300 import workloads as wl

NP = {"fp32": np.float32, "fp64": np.float64}
TORCH = {"fp32": torch.float32, "fp64": torch.float64}


def listed():
    return [
        # a short line stepped between two looks at it: the smallest call, bound
        # by launches; the moving window drops cells on the way
        {"name": "pulled1d_1000_fp32", "kind": "grid", "shape": "pulled", "nx": 1000, "ny": 1, "nz": 1,
         "precision": "fp32", "steps": 32, "lap": 3, "V": 2.0, "A": 1.0, "b": 1.0, "a": 0.0, "periodic": False},
        # the 1D planar front in FP64 whose free energy is followed at every step
        {"name": "planar1d_1024_fp64", "kind": "energies", "shape": "planar", "nx": 1024, "ny": 1, "nz": 1,
         "precision": "fp64", "steps": 256, "lap": 3, "V": 0.0, "A": 1.0, "b": 1.0, "a": 0.0, "periodic": False},
        # the FP64 check of a 2D run on a crop of it
        {"name": "front2d_128_fp64", "kind": "grid", "shape": "front", "nx": 128, "ny": 128, "nz": 1,
         "precision": "fp64", "steps": 20, "lap": 9, "V": 0.0, "A": 1.0, "b": 1.0, "a": 0.0, "periodic": True},
        # the 2D perturbed front at its full size
        {"name": "front2d_1024_fp32", "kind": "grid", "shape": "front", "nx": 1024, "ny": 1024, "nz": 1,
         "precision": "fp32", "steps": 20, "lap": 9, "V": 0.0, "A": 1.0, "b": 1.0, "a": 0.0, "periodic": True},
        # an odd 3D box, periodic across the growth direction, with the a != 0 shape
        {"name": "front3d_150x97x83_fp32", "kind": "grid", "shape": "front", "nx": 150, "ny": 97, "nz": 83,
         "precision": "fp32", "steps": 10, "lap": 19, "V": 0.0, "A": 1.5, "b": 0.3, "a": -0.3, "periodic": True},
        # the FP64 run that a 3D FP32 run is compared with
        {"name": "seed3d_96_fp64", "kind": "grid", "shape": "seed", "nx": 96, "ny": 96, "nz": 96,
         "precision": "fp64", "steps": 4, "lap": 19, "V": 0.0, "A": 1.0, "b": 1.0, "a": 0.0, "periodic": False},
        # the headline: a 3D seed in a closed box
        {"name": "seed3d_256_fp32", "kind": "grid", "shape": "seed", "nx": 256, "ny": 256, "nz": 256,
         "precision": "fp32", "steps": 10, "lap": 19, "V": 0.0, "A": 1.0, "b": 1.0, "a": 0.0, "periodic": False},
        # the checks of a long run between two blocks of steps
        {"name": "monitor3d_256_fp32", "kind": "monitor", "shape": "seed", "nx": 256, "ny": 256, "nz": 256,
         "precision": "fp32", "steps": 0, "lap": 19, "V": 0.0, "A": 1.0, "b": 1.0, "a": 0.0, "periodic": False},
        # states from the host, one step, fields back to the host
        {"name": "stream3d_256_fp32", "kind": "stream", "shape": "seed", "nx": 256, "ny": 256, "nz": 256,
         "precision": "fp32", "steps": 1, "lap": 19, "V": 0.0, "A": 1.0, "b": 1.0, "a": 0.0, "periodic": False},
        # the k(V) sweep: fronts of uneven length and speed
        {"name": "sweep_256_fp32", "kind": "batch", "instances": 256, "n_lo": 512, "n_hi": 8192, "v_lo": 1e-3,
         "v_hi": 10.0, "precision": "fp32", "steps": 500, "A": 1.0, "b": 1.0, "mode": ""},
        # one calibration step on 16 fronts: derivatives by the tangent run ...
        {"name": "tangent_16x2048_fp32", "kind": "adjoint", "instances": 16, "n_lo": 2048, "n_hi": 2048,
         "v_lo": 0.05, "v_hi": 5.0, "precision": "fp32", "steps": 128, "A": 1.1, "b": 1.0, "mode": "tangent"},
        # ... and by the reverse sweep with checkpoints
        {"name": "reverse_16x2048_fp32", "kind": "adjoint", "instances": 16, "n_lo": 2048, "n_hi": 2048,
         "v_lo": 0.05, "v_hi": 5.0, "precision": "fp32", "steps": 196, "A": 1.1, "b": 1.0, "mode": "reverse"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["line", "energies", "plane", "plane", "box", "box", "monitor", "stream", "batch", "batch",
                       "tangent", "reverse"])
    precision = rng.choice(["fp32", "fp32", "fp64"])
    A, b, a = rng.choice([(1.0, 1.0, 0.0), (1.0, 1.0, 0.0), (0.4, 1.0, 0.0), (1.5, 0.3, -0.3)])
    if kind in ("batch", "tangent", "reverse"):
        # lengths up to what an instance may hold, fewer of them where the run is long
        inst = _log_int(rng, 4, 256 if kind == "batch" else 24)
        top = {"batch": 8192, "tangent": 2048, "reverse": 2048}[kind]
        if precision == "fp64":
            inst, top = min(inst, 16 if kind == "batch" else 8), top // 8 if kind == "batch" else top // 4
        lo = _log_int(rng, 64, top)
        hi = rng.randint(lo, top)
        steps = _log_int(rng, 40, 200 if precision == "fp64" else {"batch": 500, "tangent": 128, "reverse": 196}[kind])
        return {"kind": "batch" if kind == "batch" else "adjoint", "instances": inst, "n_lo": lo, "n_hi": hi,
                "v_lo": rng.choice([1e-3, 0.05]), "v_hi": rng.choice([2.0, 5.0, 10.0]), "precision": precision,
                "steps": steps, "A": 1.0 if kind == "batch" else 1.1, "b": 1.0,
                "mode": "" if kind == "batch" else kind}
    if kind == "energies":
        precision = "fp64"   # the F_h of every step is followed in FP64 runs
    case = {"kind": "grid", "shape": "front", "nx": 1, "ny": 1, "nz": 1, "precision": precision, "steps": 1,
            "lap": 3, "V": 0.0, "A": A, "b": b, "a": a, "periodic": bool(rng.randint(0, 1))}
    if kind in ("line", "energies"):
        case.update(kind="grid" if kind == "line" else "energies", nx=_log_int(rng, 64, 8192), periodic=False,
                    steps=_log_int(rng, 1, 200), shape="pulled" if kind == "line" and rng.random() < 0.6 else "planar")
        if case["precision"] == "fp64":
            case["nx"] = min(case["nx"], rng.randint(512, 2048))
        if case["shape"] == "pulled":
            case.update(V=rng.choice([0.1, 1.0, 2.0]), A=1.0, b=1.0, a=0.0)
    elif kind == "plane":
        top = 1024 if precision == "fp32" else 320
        case.update(nx=_log_int(rng, 40, top), ny=_log_int(rng, 40, top), lap=rng.choice([5, 9, 9]),
                    steps=_log_int(rng, 1, 20))
    else:
        top = 256 if precision == "fp32" else 96
        n = [_log_int(rng, 24, top) for _ in range(3)]
        if rng.random() < 0.5:   # rows of whole 16-byte words, as most boxes have
            n[0] = (n[0] + 7) // 8 * 8
        case.update(nx=n[0], ny=n[1], nz=n[2], lap=rng.choice([7, 19, 19]), steps=_log_int(rng, 1, 10),
                    shape=rng.choice(["front", "seed"]))
        if case["shape"] == "seed":
            case["periodic"] = False
        if kind == "monitor":
            case.update(kind="monitor", steps=0)
        if kind == "stream":
            case.update(kind="stream", steps=1)
    return case


# ------------------------------------------------------------------- inputs

def _dims(case):
    n = (case["nx"], case["ny"], case["nz"])
    return 3 if n[2] > 1 else 2 if n[1] > 1 else 1


def _params(case):
    dim = _dims(case)
    n = (case["nx"], case["ny"], case["nz"])[:dim]
    kw = dict(A=case["A"], b=case["b"], a=case["a"], lap=case["lap"])
    if case["shape"] == "pulled":
        return wl.pulled_front_1d(N=n[0], dx=0.5, V=case["V"], G_theta=5.25e-3, **kw)[0]
    if case["shape"] == "planar":
        return wl.planar_1d(N=n[0], front_cell=n[0] // 4, **kw)[0]
    if case["periodic"]:
        kw.update(bc_lo=("noflux",) + ("periodic",) * (dim - 1), bc_hi=("noflux",) + ("periodic",) * (dim - 1))
    k_e, u, D_s = (0.15, 0.3, 1e-3) if case["shape"] == "front" else (0.1, 0.5, 1e-4)
    return wl.scaled_params(dim, n, 0.5, k_e, wl.theta_from_undercooling(k_e, u), D_s, **kw)


def _fields(case, pr, seed, device="cuda"):
    """(phi, c_s, c_l) in 64 bits on the device, then rounded to the run's type: a
    tanh front whose position is modulated by seeded long waves, or a seeded
    rough sphere, c_s = k_e and c_l = 1 everywhere."""
    g = np.random.default_rng(seed)
    dim, dx = pr["dim"], pr["dx"]
    shape = tuple(pr["n"][::-1])
    ax = [(torch.arange(n, dtype=torch.float64, device=device) + 0.5).reshape((-1,) + (1,) * k)
          for k, n in enumerate(pr["n"])]   # x, y, z, each along its own dimension of [z][y][x]
    if case["shape"] == "seed":
        r2 = sum((x - n / 2) ** 2 for x, n in zip(ax, pr["n"]))
        r = r2.sqrt().clamp_min(1e-12)
        R = torch.full(shape, min(20.0, 0.3 * min(pr["n"])), dtype=torch.float64, device=device)
        amp = g.uniform(0.2, 1.0, 8)
        for m in range(8):
            k = g.integers(-2, 3, 3)
            R += amp[m] / amp.sum() * torch.cos(sum(int(q) * (x - n / 2) for q, x, n in zip(k, ax, pr["n"])) / r +
                                                g.uniform(0, 2 * math.pi))
        dist = (r - R) * dx
    else:
        front = pr["x0"] / dx if case["shape"] == "pulled" else pr["n"][0] / 4
        xf = torch.full(shape[:-1] + (1,), front + g.uniform(-0.5, 0.5), dtype=torch.float64, device=device)
        if dim > 1:
            pert = torch.zeros_like(xf)
            for _ in range(6):
                ph = sum(2 * math.pi * int(g.integers(0, max(1, n // 16) + 1)) / n * x
                         for x, n in zip(ax[1:], pr["n"][1:]))
                pert = pert + g.uniform(0.5, 1.0) * torch.cos(ph + g.uniform(0, 2 * math.pi))
            xf = xf + 2.0 * pert / pert.abs().max().clamp_min(1e-12)
        dist = (ax[0] - xf) * dx
    phi = 1.0 / (1.0 + torch.exp(math.sqrt(2.0) * dist))
    dtype = TORCH[case["precision"]]
    cs = torch.full(shape, pr["k_e"] * pr["c_inf"], dtype=dtype, device=device)
    cl = torch.full(shape, pr["c_inf"], dtype=dtype, device=device)
    return phi.to(dtype).contiguous(), cs, cl


def _fronts(case, seed):
    """The packed pulled fronts of a batch: lengths fixed by the case, speeds and
    front positions by the seed."""
    g, gl = np.random.default_rng(seed), np.random.default_rng(case["instances"])
    N = case["instances"]
    lengths = gl.integers(case["n_lo"], case["n_hi"] + 1, size=N)
    v = np.exp(np.linspace(math.log(case["v_lo"]), math.log(case["v_hi"]), N)) * g.uniform(0.9, 1.0, N)
    off = np.concatenate([[0], np.cumsum(lengths)])
    phi, dts = np.empty(off[-1]), []
    cell = min(128 if case["kind"] == "batch" else 256, case["n_lo"] // 4)   # theta_ref and x0 are shared
    for i, n in enumerate(lengths):
        pr = wl.pulled_front_1d(N=int(n), dx=0.5, V=float(v[i]), G_theta=5.25e-3, front_cell=cell, A=case["A"],
                                b=case["b"])[0]
        phi[off[i]:off[i + 1]] = wl.tanh_profile(wl.cell_centres(int(n), 0.5), pr["x0"] + g.uniform(-0.25, 0.25))
        dts.append(min(0.9 * wl.stable_dt(pr), 0.5 * pr["dx"] / v[i]))
    dtype = NP[case["precision"]]
    cs = np.full(off[-1], pr["k_e"], dtype)
    cl = np.full(off[-1], 1.0, dtype)
    return pr, lengths, v, np.array(dts), phi.astype(dtype), cs, cl


def _k_target(v):
    return (0.1 + v) / (1.0 + v)


# ---------------------------------------------------------------- the passes

def prepare(case, seed):
    if case["kind"] in ("batch", "adjoint"):
        return {"case": case, "fronts": _fronts(case, seed)}
    pr = _params(case)
    sim = pf.Sim(pr, case["precision"])
    if case["kind"] == "stream":
        frames = []
        for k in range(2):
            f = [t.cpu().pin_memory() for t in _fields(case, pr, 2 * seed + k)]
            o = [torch.empty_like(t).pin_memory() for t in f]
            frames.append(([t.numpy() for t in f], [t.numpy() for t in o], f, o))
        return {"case": case, "sim": sim, "frames": frames}
    f = _fields(case, pr, seed)
    if case["kind"] == "monitor":   # the state is there: the run holds it
        sim.set_fields(*f)
        return {"case": case, "sim": sim}
    return {"case": case, "sim": sim, "fields": f, "out": [torch.empty_like(t) for t in f]}


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        pr, lengths, v, dts, phi, cs, cl = state["fronts"]
        steps = case["steps"]
        r = pf.run_batch(pr, lengths, v, phi, cs, cl, precision=case["precision"], dt=dts, max_steps=steps,
                         steps_per_launch=max(1, steps // 4), launches_per_graph=4, check_every=steps, tol=-1.0,
                         want_fields=True)
        # k_v is c_inf over a value of c, which the run holds in its own type
        return {"k": r["k_v"].astype(NP[case["precision"]]), "steps": r["steps"], "phi": r["phi"], "cs": r["cs"],
                "cl": r["cl"]}
    if case["kind"] == "adjoint":
        pr, lengths, v, dts, phi, cs, cl = state["fronts"]
        r = pf.adjoint(pr, lengths, v, phi, cs, cl, case["steps"], k_target=_k_target(v), dt=dts,
                       precision=case["precision"], mode=case["mode"])
        t = NP[case["precision"]]   # the type of the run whose values and derivatives these are
        return {"k": r["k"].astype(t), "dk": r["dk"].astype(t), "loss": t(r["loss"]), "grad": r["grad"].astype(t)}
    sim = state["sim"]
    if case["kind"] == "monitor":
        E, S = sim.energy(), sim.solute_total()
        x, _, c = sim.front()
        return {"energy": E, "solute": S, "x_front": x, "c_max": c}
    if case["kind"] == "stream":
        for ins, outs, _, _ in state["frames"]:
            sim.set_fields_step(*ins, n=1, wait=False)
            sim.get_fields_async(out_host=outs)
        sim.sync()
        return [outs for _, outs, _, _ in state["frames"]]
    sim.set_clock(0, 0)
    sim.set_fields(*state["fields"])
    F = None
    if case["kind"] == "energies":
        F = sim.step_energies(case["steps"])
    else:
        sim.step(case["steps"])
    sim.get_fields(out=state["out"])
    phi, cs, cl = state["out"]
    return {"energies": F, "phi": phi, "cs": cs, "cl": cl}


def work(case):
    """The fields in and out once, and the operations of the formulas: per
    cell-update 200 in 1D, 355 in 2D, 509 in 3D; 120 per cell of the energy with
    its gradient pairs."""
    size = 8 if case["precision"] == "fp64" else 4
    if case["kind"] in ("batch", "adjoint"):
        n = case["instances"] * (case["n_lo"] + case["n_hi"]) / 2
        # value and three derivatives; or forward, re-run and an adjoint of twice its operations
        per = {"": 200.0, "tangent": 800.0, "reverse": 800.0}[case["mode"]]
        return {"bytes": n * size * (6 if case["kind"] == "batch" else 3), "flops": n * case["steps"] * per}
    cells = case["nx"] * case["ny"] * case["nz"]
    per = {1: 200.0, 2: 355.0, 3: 509.0}[_dims(case)]
    if case["kind"] == "monitor":
        return {"bytes": 4.0 * cells * size, "flops": 120.0 * cells}
    passes = 2 if case["kind"] == "stream" else 1
    flops = cells * case["steps"] * (per + (80.0 if case["kind"] == "energies" else 0.0))
    return {"bytes": 6.0 * cells * size * passes, "flops": flops * passes}


# ------------------------------------------------ the model in plain 64 bits

class _Model:
    """One forward-Euler step on tensors whose last `dim` dimensions are the grid
    [z][y][x] (a batch of lines has one more in front)."""

    def __init__(self, pr, par=None):
        self.pr, self.dim, self.dx = pr, pr["dim"], pr["dx"]
        self.par = par or {k: pr[k] for k in ("M_phi", "A", "b")}
        self.dir = dict(phi=pr["dirichlet"][0], cs=pr["dirichlet"][1], cl=pr["dirichlet"][2])
        self.log_ke = math.log(pr["k_e"])

    def p(self, f):
        g = f * (1 - f)
        return f ** 3 * (10 - 15 * f + 6 * f * f) + self.pr["a"] * (f - 0.5) * g * g

    def dp(self, f):
        g = f * (1 - f)
        return 30 * g * g + self.pr["a"] * (g * g + (f - 0.5) * 2 * g * (1 - 2 * f))

    def pad(self, f, k, ghost):
        """One ghost on both sides of axis k (0 = x): mirror, wrap or `ghost`."""
        d = f.dim() - 1 - k
        n = f.shape[d]

        def side(name, near, far):
            bc = self.pr[name][k]
            if bc == "periodic":
                return f.narrow(d, far, 1)
            if bc == "dirichlet":
                return torch.full_like(f.narrow(d, near, 1), ghost)
            return f.narrow(d, near, 1)

        return torch.cat([side("bc_lo", 0, n - 1), f, side("bc_hi", n - 1, 0)], d)

    def pad_all(self, f, ghost):
        for k in reversed(range(self.dim)):
            f = self.pad(f, k, ghost)
        return f

    def at(self, F, *shift):
        """The interior of a padded field, shifted by cells along (x, y, z)."""
        for k in range(self.dim):
            d = F.dim() - 1 - k
            F = F.narrow(d, 1 + (shift[k] if k < len(shift) else 0), F.shape[d] - 2)
        return F

    def e(self, k, s=1):
        return tuple(s if q == k else 0 for q in range(self.dim))

    def laplacian(self, F):
        c, dim, lap = self.at(F), self.dim, self.pr["lap"]
        near = sum(self.at(F, *self.e(k, s)) - c for k in range(dim) for s in (-1, 1))
        if lap in (3, 5, 7):
            return near / self.dx ** 2
        diag = 0
        for i in range(dim):
            for j in range(i):
                for s in (-1, 1):
                    for t in (-1, 1):
                        sh = [0] * dim
                        sh[i], sh[j] = s, t
                        diag = diag + (self.at(F, *sh) - c)
        w = (2 / 3, 1 / 6) if lap == 9 else (1 / 3, 1 / 6)
        return (w[0] * near + w[1] * diag) / self.dx ** 2

    def pointwise(self, phi, c, d):
        p = self.p(phi)
        cs, cl = c + (1 - p) * d, c - p * d
        mus, mul = cs.log() - self.log_ke, cl.log()
        return p, cs, cl, mus, mul, mul + p * (mus - mul)

    def step(self, phi, c, d, theta, dt, real=None):
        """The state after one step; `real`: mask of the cells that exist (others
        hold the Dirichlet state)."""
        pr, dx, dim = self.pr, self.dx, self.dim
        A, b, M_phi = self.par["A"], self.par["b"], self.par["M_phi"]
        p, cs, cl, mus, mul, Y = self.pointwise(phi, c, d)
        g = self.dir
        gp = float(self.p(torch.tensor(g["phi"], dtype=torch.float64)))
        gs, gl = math.log(g["cs"]) - self.log_ke, math.log(g["cl"])
        ghost = (g["phi"], gl + gp * (gs - gl), gs, gl)
        four = (phi, Y, mus, mul)
        pads = [self.pad_all(f, q) for f, q in zip(four, ghost)]
        grad = [[(self.at(F, *self.e(k)) - self.at(F, *self.e(k, -1))) / (2 * dx) for k in range(dim)] for F in pads]
        D_s, D_l = pr["D_s"], pr["D_l"]
        Ms, Ml = D_s * cs, D_l * cl
        q = 1 - p
        Mbar = Ms * q + b * Ml * p
        G = sum(x * x for x in grad[0]) + pr["delta"] ** 2
        cross = sum((Ms * s - b * Ml * m) * f for f, s, m in zip(grad[0], grad[2], grad[3]))
        dd = cs - cl
        K = 1 / M_phi + (1 - A) ** 2 * dd * dd * b * p * q / (G * Mbar * (b * p + q))
        D = (Ms * q * (1 - A * q) + A * b * Ml * p * p) / Mbar
        dG = cs * (mus - mul) - dd - (1 - pr["k_e"]) * theta - D * dd * (mus - mul)
        R = (pr["sigma"] * self.laplacian(pads[0]) - pr["H"] * 2 * phi * (1 - phi) * (1 - 2 * phi) - dG * self.dp(phi)
             + (1 - A) * dd * p * q * cross / (Mbar * G))
        rate = R / K
        if real is not None:
            rate = torch.where(real, rate, torch.zeros_like(rate))
        dc = dd_ = 0
        for k in range(dim):
            ax = phi.dim() - 1 - k
            n = phi.shape[ax]

            def both(f, gh, k=k, ax=ax, n=n):
                F = self.pad(f, k, gh)
                return F.narrow(ax, 0, n + 1), F.narrow(ax, 1, n + 1)

            nrm = [(r - l) / dx for l, r in (both(f, q_) for f, q_ in zip(four, ghost))]
            mean = [0.5 * (l + r) for l, r in (both(phi, g["phi"]), both(cs, g["cs"]), both(cl, g["cl"]),
                                               both(rate, 0.0))]
            fphi, fcs, fcl, frate = mean
            trn = [[0.5 * sum(both(grad[f][m], 0.0)) for m in range(dim) if m != k] for f in range(4)]
            fp = self.p(fphi)
            fq = 1 - fp
            fMs, fMl = D_s * fcs, D_l * fcl
            fM = fMs * fq + b * fMl * fp
            t2 = sum(x * x for x in trn[0]) + pr["delta"] ** 2
            r = 1 / (nrm[0] * nrm[0] + t2)
            qn = fMs * fMl * (b * fp + fq) / fM
            normal = qn * nrm[0] * (nrm[0] * nrm[1] + sum(x * y for x, y in zip(trn[0], trn[1]))) * r
            at = (1 - A) * (fcs - fcl) * frate * nrm[0] * r
            Ts = fMs * (nrm[2] * t2 - nrm[0] * sum(x * y for x, y in zip(trn[0], trn[2]))) * r
            Tl = fMl * (nrm[3] * t2 - nrm[0] * sum(x * y for x, y in zip(trn[0], trn[3]))) * r
            Fs = normal + Ts + at * fMs * fq / fM
            Fl = normal + Tl - at * b * fMl * fp / fM
            F = [fp * Fs + fq * Fl, Fs - Fl]
            open_ = torch.ones([n + 1 if x == ax else 1 for x in range(phi.dim())], dtype=torch.float64,
                               device=phi.device)
            if pr["bc_lo"][k] == "noflux":
                open_.narrow(ax, 0, 1).zero_()
            if pr["bc_hi"][k] == "noflux":
                open_.narrow(ax, n, 1).zero_()
            F = [x * open_ for x in F]
            dc = dc + (F[0].narrow(ax, 1, n) - F[0].narrow(ax, 0, n)) / dx
            dd_ = dd_ + (F[1].narrow(ax, 1, n) - F[1].narrow(ax, 0, n)) / dx
        new = (phi + dt * rate, c + dt * dc, d + dt * dd_)
        if real is not None:
            new = tuple(torch.where(real, x, o) for x, o in zip(new, (phi, c, d)))
        return new

    def state(self, phi, cs, cl):
        p = self.p(phi)
        return phi, p * cs + (1 - p) * cl, cs - cl

    def fields(self, phi, c, d):
        p = self.p(phi)
        return phi, c + (1 - p) * d, c - p * d

    def theta(self, x, t, shifts):
        pr = self.pr
        return pr["theta_ref"] + pr["G_theta"] * (pr["x0"] + pr["v_pull"] * t - shifts * self.dx) - pr["G_theta"] * x

    def fresh(self):
        return self.state(*(torch.tensor(v, dtype=torch.float64) for v in self.pr["dirichlet"]))

    def energy(self, phi, c, d, theta):
        pr = self.pr
        p, cs, cl, mus, mul, _ = self.pointwise(phi, c, d)
        fs = -(1 - pr["k_e"]) * theta + cs * (mus - 1)
        fl = cl * (mul - 1)
        F = self.pad_all(phi, self.dir["phi"])
        g2 = 0
        lap = pr["lap"]
        for i in range(3 ** self.dim):
            sh = [i // 3 ** k % 3 - 1 for k in range(self.dim)]
            m = sum(map(abs, sh))
            w = {3: (0, 1), 5: (0, 1), 9: (0, 2 / 3, 1 / 6), 7: (0, 1), 19: (0, 1 / 3, 1 / 6)}[lap]
            if 0 < m < len(w):
                g2 = g2 + w[m] * (self.at(F, *sh) - phi) ** 2
        e = pr["H"] * phi ** 2 * (1 - phi) ** 2 + p * fs + (1 - p) * fl + 0.25 * pr["sigma"] * g2 / self.dx ** 2
        return float(e.sum()) * self.dx ** self.dim


def _exact_grid(case, seed):
    pr = _params(case)
    M = _Model(pr)
    x = (torch.arange(pr["n"][0], dtype=torch.float64, device="cuda") + 0.5) * pr["dx"]
    outs = []
    for k in range(2 if case["kind"] == "stream" else 1):
        f = _fields(case, pr, 2 * seed + k if case["kind"] == "stream" else seed)
        s = M.state(*(t.double() for t in f))
        if case["kind"] == "monitor":
            lo, hi = s[0].narrow(-1, 0, pr["n"][0] - 1), s[0].narrow(-1, 1, pr["n"][0] - 1)
            cross = (x[:-1] + (lo - 0.5) / (lo - hi) * pr["dx"])
            cross = torch.where((lo >= 0.5) & (hi < 0.5), cross, torch.full_like(cross, -math.inf))
            return {"energy": M.energy(*s, M.theta(x, 0.0, 0)), "solute": float(s[1].sum()) * pr["dx"] ** pr["dim"],
                    "x_front": float(cross.max()), "c_max": float(s[1].max())}
        shifts, F = 0, []
        for i in range(case["steps"]):
            s = M.step(*s, M.theta(x, i * pr["dt"], shifts), pr["dt"])
            while pr["shift"] and pr["v_pull"] * ((i + 1) * pr["dt"]) >= (shifts + 1) * pr["dx"]:
                s = tuple(torch.cat([a[1:], w.to(a.device).reshape(1)]) for a, w in zip(s, M.fresh()))
                shifts += 1
            if case["kind"] == "energies":
                F.append(M.energy(*s, M.theta(x, (i + 1) * pr["dt"], shifts)))
        outs.append(M.fields(*s))
    if case["kind"] == "stream":
        return [list(o) for o in outs]
    phi, cs, cl = outs[0]
    return {"energies": np.array(F) if F else None, "phi": phi, "cs": cs, "cl": cl}


def _exact_fronts(case, fronts, par=None):
    """(state, mask) after the case's steps of all fronts, one per row, cells
    beyond a front's end holding the Dirichlet state."""
    pr, lengths, v, dts, phi0, cs0, cl0 = fronts
    pr = dict(pr, bc_lo=("noflux",), bc_hi=("dirichlet",))
    M = _Model(pr, par)
    N, n = len(lengths), int(max(lengths))
    L = torch.tensor(lengths, device="cuda").reshape(-1, 1)
    real = torch.arange(n, device="cuda") < L
    packed = [torch.from_numpy(np.asarray(a, np.float64)).cuda() for a in (phi0, cs0, cl0)]
    rows = [torch.full((N, n), g, dtype=torch.float64, device="cuda") for g in pr["dirichlet"]]
    for r, a in zip(rows, packed):
        r[real] = a
    s = M.state(*rows)
    fresh = [w.cuda() for w in M.fresh()]
    x = (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * pr["dx"]
    dt = torch.tensor(dts, device="cuda").reshape(-1, 1)
    shifts = np.zeros(N, np.int64)
    for i in range(case["steps"]):
        th0 = pr["theta_ref"] + pr["G_theta"] * (pr["x0"] + v * (i * dts) - shifts * pr["dx"])
        s = M.step(*s, torch.tensor(th0, device="cuda").reshape(-1, 1) - pr["G_theta"] * x, dt, real)
        while True:
            due = v * ((i + 1) * dts) >= (shifts + 1) * pr["dx"]
            if not due.any():
                break
            mask = torch.tensor(due, device="cuda").reshape(-1, 1)
            s = tuple(torch.where(mask, torch.cat([a[:, 1:], w.expand(N, 1)], 1), a) for a, w in zip(s, fresh))
            shifts[due] += 1
    return M, s, real


def exact(case, seed):
    if case["kind"] == "batch":
        fronts = _fronts(case, seed)
        M, s, real = _exact_fronts(case, fronts)
        f = [t[real] for t in M.fields(*s)]
        cmax = torch.where(real, s[1], torch.full_like(s[1], -math.inf)).amax(1)
        return {"k": 1.0 / cmax, "steps": None, "phi": f[0], "cs": f[1], "cl": f[2]}
    if case["kind"] == "adjoint":
        pr, lengths, v, dts, *packed = _fronts(case, seed)
        N, names = len(lengths), ("M_phi", "A", "b")
        # three copies of the fronts, the derivative of copy j along parameter j
        fronts = (pr, np.tile(lengths, 3), np.tile(v, 3), np.tile(dts, 3), *[np.tile(a, 3) for a in packed])
        theta = torch.tensor([[pr[k]] for k in names], dtype=torch.float64, device="cuda").expand(3, 3 * N).clone()
        along = torch.eye(3, dtype=torch.float64, device="cuda").repeat_interleave(N, 1)

        def k_of(th):
            _, s, real = _exact_fronts(case, fronts, {q: t.reshape(-1, 1) for q, t in zip(names, th)})
            return 1.0 / torch.where(real, s[1], torch.full_like(s[1], -math.inf)).max(1).values

        k, dk = torch.func.jvp(k_of, (theta,), (along,))
        k, dk = k[:N], dk.reshape(3, N).T.contiguous()
        res = k - torch.from_numpy(_k_target(v)).cuda()
        return {"k": k, "dk": dk, "loss": float((res * res).sum()), "grad": (2 * res[:, None] * dk).sum(0)}
    return _exact_grid(case, seed)
