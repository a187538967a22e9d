"""The measured cases: what a program does with this framework through its public entry points.

Three kinds of case:

* ``solver``    some time steps of one flow (``binding.Solver.step``), then the flag's state on the
                host, as a campaign loop reads it; outputs are the whole velocity fields on the
                device and the flag's X, V, F. With ``inflow`` the run is driven by the learned
                generator: a keyframe every ``stride`` steps and interpolated planes in between.
* ``ensemble``  time steps of several uneven cases advanced together (``binding.Ensemble``).
* ``generator`` the learned inflow's network: training steps on recorded planes, or forward passes.

Fields start from U plus a smooth perturbation of turbulence intensity 0.1 (a sum of Fourier modes),
the level behind a bar grid. ``exact`` computes the same outputs in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

from paper_2103_08246_gb300 import binding, inflow, inputs

PRECISION = {"fp64": binding.IBM_FP64, "fp32": binding.IBM_FP32, "mixed": binding.IBM_MIXED}
RELAX, NOISE, STRIDE, TU = 0.01, 0.03, 10, 0.1


# ------------------------------------------------------------------ the cases
def _solver(name, nx, ny, nz, h, precision, steps, bars="markers", flag=True, re=200.0, dt=-1.0, bending=0.005,
            flag_x=3.0, flag_n=0, span=1.0, inflow=False):
    """flag_n: flag vertices along the chord (0: at the grid spacing)."""
    c = {"kind": "solver", "nx": nx, "ny": ny, "nz": nz, "h": h, "precision": precision, "steps": steps,
         "bars": bars, "flag": flag, "re": re, "dt": dt, "bending": bending, "flag_x": flag_x,
         "flag_n": flag_n or int(round(1.0 / h)) + 1, "span": span, "inflow": inflow}
    return {**c, "name": name} if name else c


def listed():
    return [
        # the smallest workload, as the parity and smoke runs step it: a call is latency and launches
        _solver("tiny-fp64", 64, 32, 32, 1 / 16, "fp64", 10, re=100.0, dt=2e-3, bending=0.01, flag_x=2.0),
        # a short ragged box without a flag (odd nx, ny != nz), bars forced on Eulerian nodes
        _solver("ragged-fp32", 91, 32, 64, 1 / 16, "fp32", 10, bars="eulerian", flag=False),
        # a fine 65 x 65 flag in a small box: the structure weighs as much as the flow
        _solver("flagbox-fp64", 96, 64, 128, 1 / 64, "fp64", 10, bars="none", dt=2e-3, flag_x=0.25),
        # the laminar flag validation at h = 1/32: the ordinary size, in the three precisions of its comparison
        _solver("laminar-fp32", 256, 128, 128, 1 / 32, "fp32", 10, bars="none", dt=6e-3),
        _solver("laminar-mixed", 256, 128, 128, 1 / 32, "mixed", 10, bars="none", dt=6e-3),
        _solver("laminar-fp64", 256, 128, 128, 1 / 32, "fp64", 5, bars="none", dt=6e-3),
        # the production workload (bars and 65 x 65 flag, CFL steps), in each precision
        _solver("production-mixed", 512, 256, 256, 1 / 64, "mixed", 10),
        _solver("production-fp32", 512, 256, 256, 1 / 64, "fp32", 10),
        _solver("production-fp64", 512, 256, 256, 1 / 64, "fp64", 3),
        # the flag driven by generated inflow planes (rollout of the trained network, then the step)
        _solver("driven-fp32", 384, 256, 256, 1 / 64, "fp32", 10, bars="none", flag_x=1.0, inflow=True),
        # sixteen uneven cases stepped together
        {"name": "ensemble-mixed", "kind": "ensemble", "members": 16, "seed": 0, "precision": "mixed", "steps": 10},
        # training the inflow generator at the campaign's size
        {"name": "generator-train", "kind": "generator", "what": "train", "ny": 256, "nz": 256, "blocks": 13,
         "batch": 8, "steps": 4},
    ]


def draw(rng):
    kind = rng.choice(["solver"] * 7 + ["ensemble", "generator", "generator"])
    if kind == "ensemble":
        return {"kind": "ensemble", "members": rng.randint(3, 16), "seed": rng.randint(1, 1000),
                "precision": rng.choice(["fp32", "mixed", "mixed", "fp64"]), "steps": rng.randint(3, 10)}
    if kind == "generator":
        what = rng.choice(["train", "forward"])
        return {"kind": "generator", "what": what, "ny": rng.choice([24, 64, 100, 128, 256]),
                "nz": rng.choice([128, 256]), "blocks": rng.randint(1, 13), "batch": rng.randint(1, 8),
                "steps": rng.randint(1, 3)}
    while True:
        h = 1.0 / rng.choice([16, 16, 32, 32, 64])
        ny, nz = (rng.choice([n for n in (16, 32, 64, 128, 256) if n * h >= 1.0]) for _ in range(2))
        flag = rng.random() < 0.7
        bars = rng.choice(["markers", "markers", "eulerian", "none"])
        low = (2.6 if flag else 1.0) / h
        nx = int(round(math.exp(rng.uniform(math.log(low), math.log(512)))))
        precision = rng.choice(["fp64", "fp32", "mixed"])
        steps = rng.randint(3, 10)
        if nx * ny * nz * steps * (8 if precision == "fp64" else 1) <= 512 * 256 * 256 * 20:
            break
    n = rng.choice([0, 0, rng.randint(int(0.5 / h), int(1 / h))])
    return _solver(None, nx, ny, nz, h, precision, steps, bars=bars, flag=flag, re=round(rng.uniform(100.0, 400.0), 1),
                   dt=rng.choice([-1.0, round(0.2 * h, 6)]), bending=round(10.0 ** rng.uniform(-3.0, -1.0), 6),
                   flag_x=round(rng.uniform(1.0, max(1.0, nx * h - 1.3)), 3), flag_n=n, span=rng.choice([1.0, 1.0, 0.5]))


# ------------------------------------------------------------------ what a program has in hand
def _workload(c):
    nx, ny, nz, h = c["nx"], c["ny"], c["nz"], c["h"]
    nt = max(3, int(round((c["flag_n"] - 1) * c["span"])) + 1)
    return inputs.Workload(name="case", nx=nx, ny=ny, nz=nz, lx=nx * h, ly=ny * h, lz=nz * h, re=c["re"],
                           bars_on=c["bars"] != "none", bar_forcing="eulerian" if c["bars"] == "eulerian" else "markers",
                           flag_on=c["flag"], flag_x_le=c["flag_x"], flag_span=c["span"], flag_ns=c["flag_n"], flag_nt=nt,
                           bending=c["bending"], dt=c["dt"])


def _perturbation(wl, seed):
    """Three host arrays (nx + 1, ny, nz): smooth, rms TU, zero on the faces a run does not perturb."""
    g = np.random.default_rng(seed)
    x, y, z = (torch.arange(n, dtype=torch.float64, device="cuda") / n for n in (wl.nx, wl.ny, wl.nz))
    out = []
    for comp in range(3):
        f = torch.zeros((wl.nx + 1, wl.ny, wl.nz), dtype=torch.float64, device="cuda")
        for _ in range(6):
            k = g.integers(1, 4, size=3)
            a, b, d = g.uniform(0.0, 2 * np.pi, size=3)
            f[:wl.nx] += (torch.sin(2 * np.pi * k[0] * x + a)[:, None, None] * torch.sin(2 * np.pi * k[1] * y + b)[:, None]
                          * torch.sin(2 * np.pi * k[2] * z + d))
        f *= TU / f[:wl.nx].square().mean().sqrt()
        f[wl.nx] = 0.0
        if comp == 0:
            f[0] = 0.0
        out.append(f.cpu().numpy())
    return out


def _record(ny, nz, n, seed):
    """n recorded planes [n, 3, ny, nz] on the device: smooth modes carried across z, as a fixed plane sees them."""
    g = np.random.default_rng(seed)
    t, y, z = torch.arange(n, device="cuda"), torch.arange(ny, device="cuda") / ny, torch.arange(nz, device="cuda") / nz
    out = torch.zeros((n, 3, ny, nz), dtype=torch.float32, device="cuda")
    for comp in range(3):
        for _ in range(8):
            ky, kz = g.integers(0, 9), g.integers(1, 9)
            a, b, speed = g.uniform(0, 2 * np.pi), g.uniform(0, 2 * np.pi), g.uniform(0.2, 1.0)
            phase = 2 * np.pi * kz * (z[None] - speed * t[:, None] / nz) + b
            out[:, comp] += torch.cos(2 * np.pi * ky * y + a)[None, :, None] * torch.cos(phase)[:, None, :]
        out[:, comp] *= (0.1 if comp == 0 else 0.05) / out[:, comp].square().mean().sqrt()
    out[:, 0] += 1.0
    return out


def _generator(ny, nz, blocks, batch, stride, planes, seed, stream=None):
    gen = binding.Generator(ny, nz, blocks=blocks, in_channels=6, batch=batch, stride=stride, stream=stream)
    weights = inputs.generator_params(seed, 128, blocks, 6)
    gen.set_params(weights)
    mean, std, rms, mean_plane = inflow.data_norm(planes)
    gen.set_norm(mean, std, rms)
    return gen, weights, (mean, std, rms, mean_plane)


class _Resident:
    """A solver's field where it is on the device; keeps the solver (and its workspace) alive."""

    def __init__(self, solver, ptr):
        wl, kind = solver.wl, "<f8" if solver.precision == binding.IBM_FP64 else "<f4"
        self.solver = solver
        self.__cuda_array_interface__ = {"shape": (wl.nx + 1, wl.ny, wl.nz), "typestr": kind, "data": (ptr, False), "version": 3}


def _velocity(s):
    """The whole u, v, w of a solver, not copied (device addresses of plane 0; x is the slowest axis)."""
    return [torch.as_tensor(_Resident(s, ptr), device="cuda") for ptr in binding.ibm_plane_device(s.state, 0)]


def _real(s):
    return np.float64 if s.precision == binding.IBM_FP64 else np.float32


def prepare(case, seed):
    if case["kind"] == "solver":
        wl = _workload(case)
        s = binding.Solver(wl, PRECISION[case["precision"]], noise=_perturbation(wl, seed), inflow=case["inflow"])
        state = {"case": case, "solver": s, "k": 0}
        if case["inflow"]:
            planes = _record(wl.ny, wl.nz, 2 * STRIDE, seed)
            gen, _, norm = _generator(wl.ny, wl.nz, 13, 1, STRIDE, planes, seed, s.stream)
            gen.set_relax(norm[3], RELAX)
            gen.rollout_init(planes[-1 - STRIDE].cpu().numpy(), planes[-1].cpu().numpy())
            state.update(gen=gen, ptrs=binding.ibm_inflow_planes(s.state))
        return state
    if case["kind"] == "ensemble":
        cases = inputs.ensemble_cases(case["members"], case["seed"])
        solvers = [binding.Solver(wl, PRECISION[case["precision"]], noise=_perturbation(wl, seed + i))
                   for i, wl in enumerate(cases)]
        return {"case": case, "solvers": solvers, "ensemble": binding.Ensemble(solvers)}
    ny, nz, batch = case["ny"], case["nz"], case["batch"]
    planes = _record(ny, nz, 64, seed)
    gen, _, _ = _generator(ny, nz, case["blocks"], batch, STRIDE, planes, seed)
    state = {"case": case, "gen": gen, "planes": planes, "rng": np.random.default_rng(seed)}
    if case["what"] == "train":
        gen.set_noise(NOISE, seed=17)
        gen.set_lr(5e-4)
    else:
        q = _forward_inputs(case, seed)
        state.update(q=q, delta=[torch.empty_like(a) for a, _ in q])
    return state


def _forward_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = (case["batch"], case["ny"], case["nz"], 3)
    return [tuple(torch.randn(shape, generator=g, device="cuda") for _ in range(2)) for _ in range(case["steps"])]


def _samples(rng, case):
    return rng.integers(STRIDE, 64 - STRIDE, size=case["batch"])


# ------------------------------------------------------------------ one pass
def run(state):
    case = state["case"]
    if case["kind"] == "solver":
        s = state["solver"]
        if case["inflow"]:
            for _ in range(case["steps"]):
                k = state["k"]
                if k % STRIDE == 0:
                    state["gen"].rollout(None, None, None, precision=s.precision)
                state["gen"].emit((k % STRIDE) / STRIDE, *state["ptrs"], precision=s.precision)
                s.step(1)
                state["k"] = k + 1
        else:
            s.step(case["steps"])
        flag = [a.astype(_real(s), copy=False) for a in s.flag()] if case["flag"] else []
        return _velocity(s) + flag
    if case["kind"] == "ensemble":
        state["ensemble"].step(case["steps"])
        return [_velocity(s) + [s.flag()[0].astype(_real(s), copy=False)] for s in state["solvers"]]
    gen = state["gen"]
    if case["what"] == "train":
        for n in range(case["steps"]):
            loss = gen.train_step(state["planes"], _samples(state["rng"], case), with_loss=n == case["steps"] - 1)
        return {"loss": loss, "params": gen.params().astype(np.float32)}
    for (q, q_prev), out in zip(state["q"], state["delta"]):
        binding.ibm_gen_forward(gen.handle, q.data_ptr(), q_prev.data_ptr(), out.data_ptr(), case["batch"])
    gen.sync()
    return state["delta"]


# ------------------------------------------------------------------ what a pass cannot do without
def _solver_work(nx, ny, nz, size, steps, markers):
    """Per step: u, v, w, p and the previous advection term read and written once; per cell the explicit
    stage (about 110 operations), nine implicit line solves (6 each), the divergence and the projection
    (30), four FFT passes (2.5 log2 n each) and the tridiagonal solve along x (5); per marker 27 nodes of three
    components, interpolated and spread."""
    cells = nx * ny * nz
    flops = cells * (199 + 5 * (math.log2(ny) + math.log2(nz))) + markers * 27 * 3 * 6
    return {"bytes": steps * cells * 14.0 * size, "flops": steps * float(flops)}


def _marker_count(c):
    n = c["flag_n"] ** 2 if c["flag"] else 0
    if c["bars"] == "markers":
        across = math.ceil(0.1 / c["h"]) + 1
        n += across * across * 4 * c["ny"] * c["nz"] * c["h"]
    return n


def work(case):
    if case["kind"] == "solver":
        w = _solver_work(case["nx"], case["ny"], case["nz"], 8 if case["precision"] == "fp64" else 4, case["steps"],
                         _marker_count(case))
        if case["inflow"]:
            w["flops"] += case["steps"] / STRIDE * _conv_flops(case["ny"], case["nz"], 13)
        return w
    if case["kind"] == "ensemble":
        size = 8 if case["precision"] == "fp64" else 4
        parts = [_solver_work(wl.nx, wl.ny, wl.nz, size, case["steps"], 289 + 9 * 4 * wl.ny * wl.nz / 16)
                 for wl in inputs.ensemble_cases(case["members"], case["seed"])]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    # activations of 128 channels in 16 bits and the 32-bit residual stream, once per layer and direction
    pixels, layers = case["ny"] * case["nz"] * case["batch"], case["blocks"] + 1
    train = 3 if case["what"] == "train" else 1
    return {"bytes": float(case["steps"] * train * layers * pixels * 128 * 6),
            "flops": case["steps"] * train * case["batch"] * _conv_flops(case["ny"], case["nz"], case["blocks"])}


def _conv_flops(ny, nz, blocks):
    return 2.0 * 9 * ny * nz * 128 * (blocks * 128 + 9)


# ------------------------------------------------------------------ the same in 64 bits, plain torch
def exact(case, seed):
    with torch.no_grad():
        if case["kind"] == "solver":
            return _exact_solver(case, seed)
        if case["kind"] == "ensemble":
            cases = inputs.ensemble_cases(case["members"], case["seed"])
            if sum(wl.cells for wl in cases) * case["steps"] > 4e8:
                return None                             # minutes in all
            out = []
            for i, wl in enumerate(cases):
                f = _Flow(wl, _perturbation(wl, seed + i))
                for _ in range(case["steps"]):
                    f.step()
                out.append([*f.q, f.X])
            return out
        return _exact_generator(case, seed)


def _exact_solver(case, seed):
    wl = _workload(case)
    f = _Flow(wl, _perturbation(wl, seed))
    if case["inflow"]:
        planes = _record(wl.ny, wl.nz, 2 * STRIDE, seed)
        mean, std, rms, ref = (torch.as_tensor(a, device="cuda") for a in inflow.data_norm(planes))
        net = _network(torch.as_tensor(inputs.generator_params(seed, 128, 13, 6), device="cuda"), 13)
        col = (slice(None), None, None)
        q_prev, q = ((planes[i].double() - mean[col]) / std[col] for i in (-1 - STRIDE, -1))
        ref = (ref - mean[col]) / std[col]
    for k in range(case["steps"]):
        planes_in = None
        if case["inflow"]:
            if k % STRIDE == 0:
                new = q + _forward(net, torch.cat([q, q_prev])) - RELAX * (q - ref)
                new = new - new.mean(dim=(1, 2), keepdim=True)
                q, q_prev = new * (rms / new.square().mean(dim=(1, 2)).sqrt())[col], q
            a = (k % STRIDE) / STRIDE
            planes_in = mean[col] + std[col] * ((1 - a) * q_prev + a * q)
        f.step(planes_in)
    return [*f.q] + ([f.X, f.V, f.F] if case["flag"] else [])


def _delta(r):
    """Three-point regularised delta kernel of Roma, Peskin and Berger (1999)."""
    a = r.abs()
    inner = (1 + torch.sqrt((1 - 3 * a * a).clamp(min=0))) / 3
    outer = (5 - 3 * a - torch.sqrt((1 - 3 * (1 - a) ** 2).clamp(min=0))) / 6
    return torch.where(a <= 0.5, inner, torch.where(a < 1.5, outer, torch.zeros_like(a)))


class _Flow:
    """The fractional step of the paper's Sec. II.B in 64 bits: dense direct solves along x, FFTs in y and z."""

    def __init__(self, wl, noise):
        self.wl, self.h, self.nu = wl, wl.lx / wl.nx, 1.0 / wl.re
        dev = dict(dtype=torch.float64, device="cuda")
        self.q = [torch.as_tensor(a).cuda() for a in noise]
        self.q[0] = self.q[0] + 1.0
        self.p = torch.zeros((wl.nx, wl.ny, wl.nz), **dev)
        self.qin, self.N, self.dt_old = [None, None, None], None, None
        n, i = wl.nx, torch.arange(wl.nx, **dev)
        # orthonormal cosine basis: it diagonalises the second difference with zero end gradients
        self.C = math.sqrt(2.0 / n) * torch.cos(math.pi / n * i[:, None] * (i[None] + 0.5))
        self.C[0] /= math.sqrt(2.0)
        lam = [2 * torch.cos(math.pi * i / n) - 2] + [2 * torch.cos(2 * math.pi * torch.arange(m, **dev) / m) - 2 for m in (wl.ny, wl.nz)]
        self.lam = (lam[0][:, None, None] + lam[1][:, None] + lam[2]) / self.h ** 2
        self.lam[0, 0, 0] = 1.0
        self.lam_yz = lam[1:]
        self.X = self.V = self.F = None
        X, dv = [], []
        if wl.flag_on:
            self._flag()
            dv.append(self.area * self.h)
        self.alpha = None
        if wl.bars_on and wl.bar_forcing == "eulerian":
            self.alpha = [self._solid(c) for c in range(3)]
        elif wl.bars_on:
            X.append(self._bars())
            d, (a, b) = wl.bar_width, (round(wl.ly / wl.bar_mesh), round(wl.lz / wl.bar_mesh))
            volume = d * d * (a * wl.lz + b * wl.ly) - a * b * d ** 3
            dv.append(torch.full((len(X[0]),), volume / len(X[0]), **dev))
        self.Xb = torch.cat(X) if X else torch.zeros((0, 3), **dev)
        self.dv = torch.cat(dv) if dv else torch.zeros(0, **dev)
        self._project(self._poisson(self._div()), 1.0)

    # bodies
    def _bars(self):
        wl, d, M, h = self.wl, self.wl.bar_width, self.wl.bar_mesh, self.h
        nw = math.ceil(d / h - 1e-12) + 1
        across = d * (np.arange(nw) / (nw - 1) - 0.5)
        yc, zc = ((np.arange(round(n / M)) + 0.5) * M for n in (wl.ly, wl.lz))
        along = [(np.arange(m) + 0.5) * n / m for n in (wl.ly, wl.lz) for m in [math.ceil(n / h - 1e-12)]]
        gap = np.abs(along[0][:, None] - yc)
        free = np.minimum(gap, wl.ly - gap).min(axis=1) > 0.5 * d + 1e-12
        parts = [np.stack(np.meshgrid(wl.bar_x + across, along[0][free], (zc[:, None] + across).ravel(), indexing="ij"), -1),
                 np.stack(np.meshgrid(wl.bar_x + across, (yc[:, None] + across).ravel(), along[1], indexing="ij"), -1)]
        return torch.as_tensor(np.concatenate([a.reshape(-1, 3) for a in parts])).cuda()

    def _solid(self, comp):
        """Fraction of each velocity node's cell inside the bars."""
        wl, d, M, h = self.wl, self.wl.bar_width, self.wl.bar_mesh, self.h

        def overlap(c, mid):
            return np.clip(np.minimum(c + h / 2, mid + d / 2) - np.maximum(c - h / 2, mid - d / 2), 0.0, None)

        def rods(c, period):
            return sum(overlap(c, m + s) for m in (np.arange(round(period / M)) + 0.5) * M for s in (-period, 0.0, period))
        x, y, z = ((np.arange(n) + (0.0 if comp == k else 0.5)) * h for k, n in enumerate((wl.nx + 1, wl.ny, wl.nz)))
        ox, oy, oz = overlap(x, wl.bar_x), rods(y, wl.ly), rods(z, wl.lz)
        a = ox[:, None, None] * (h * oz + oy[:, None] * h - oy[:, None] * oz) / h ** 3
        a[wl.nx] = 0.0
        if comp == 0:
            a[0] = 0.0
        return torch.as_tensor(a).cuda()

    def _flag(self):
        wl = self.wl
        ns, nt, ds, dt = wl.flag_ns, wl.flag_nt, wl.flag_len / (wl.flag_ns - 1), wl.flag_span / (wl.flag_nt - 1)
        v = np.arange(ns * nt).reshape(ns, nt)
        c00, c10, c01, c11 = (a.ravel() for a in (v[:-1, :-1], v[1:, :-1], v[:-1, 1:], v[1:, 1:]))
        springs = [np.stack(a, -1).reshape(-1, 2) for a in ((v[:-1], v[1:]), (v[:, :-1], v[:, 1:]), (c00, c11), (c10, c01))]
        tris, pairs, edges = [], [], []
        for split in (((0, 1, 3), (0, 3, 2)), ((0, 1, 2), (1, 3, 2))):       # both diagonals of every cell
            corner = np.stack([c00, c10, c01, c11], -1)
            t = np.stack([corner[:, list(k)] for k in split], 1).reshape(-1, 3)
            e = np.sort(np.stack([t[:, [0, 1]], t[:, [1, 2]], t[:, [2, 0]]], 1).reshape(-1, 2), -1)
            key = e[:, 0] * (ns * nt) + e[:, 1]
            order = np.argsort(key, kind="stable")
            two = np.nonzero(key[order][1:] == key[order][:-1])[0]
            base = sum(len(a) for a in tris)
            pairs.append(np.stack([order[two] // 3, order[two + 1] // 3], -1) + base)
            edges.append(e[order[two]])
            tris.append(t)
        springs, tris, pairs, edges = (np.concatenate(a) for a in (springs, tris, pairs, edges))
        da, db = (np.abs(edges[:, 0] // nt - edges[:, 1] // nt) * ds, np.abs(edges[:, 0] % nt - edges[:, 1] % nt) * dt)
        e2, cell = da ** 2 + db ** 2, ds * dt
        k = 0.5 * np.where((da > 0) & (db > 0), 2 * wl.bending * cell / e2, wl.bending * e2 / cell)
        area = np.zeros(ns * nt)
        for c in (c00, c10, c01, c11):
            np.add.at(area, c, 0.25 * cell)
        four = np.sort(np.concatenate([tris[pairs[:, 0]], tris[pairs[:, 1]]], -1), -1)
        stiff = np.zeros(ns * nt)
        for col in range(6):
            new = np.ones(len(four), bool) if col == 0 else four[:, col] != four[:, col - 1]
            np.add.at(stiff, four[new, col], k[new])
        mass = wl.mass_ratio * area
        w2 = (2 * wl.stretch * np.bincount(springs.ravel(), minlength=ns * nt) + 8 * stiff / min(ds, dt) ** 2) / mass
        self.omega = math.sqrt(w2[nt:].max())
        s, t = np.arange(ns) * ds, np.arange(nt) * dt
        X = np.zeros((ns, nt, 3))
        X[:, :, 0] = (wl.flag_x_le + s * math.cos(wl.pitch0))[:, None]
        X[:, :, 1] = (0.5 * wl.ly + s * math.sin(wl.pitch0))[:, None]
        X[:, :, 2] = 0.5 * wl.lz - 0.5 * wl.flag_span + t
        self.X = torch.as_tensor(X.reshape(-1, 3)).cuda()
        self.V, self.F = torch.zeros_like(self.X), torch.zeros_like(self.X)
        self.springs, self.tris, self.pairs, self.k, self.area, self.mass = (
            torch.as_tensor(a).cuda() for a in (springs, tris, pairs, k, area, mass[:, None]))
        self.free = (torch.arange(ns * nt, device="cuda") >= nt)[:, None]
        self.rest = (self.X[self.springs[:, 1]] - self.X[self.springs[:, 0]]).norm(dim=1)

    def _acc(self):
        with torch.enable_grad():
            X = self.X.detach().requires_grad_()
            length = (X[self.springs[:, 1]] - X[self.springs[:, 0]]).norm(dim=1)
            a, b, c = (X[self.tris[:, k]] for k in range(3))
            n = torch.linalg.cross(b - a, c - a)
            n = n / n.norm(dim=1, keepdim=True)
            cos = (n[self.pairs[:, 0]] * n[self.pairs[:, 1]]).sum(dim=1)
            energy = 0.5 * self.wl.stretch * (length - self.rest).square().sum() + (self.k * (1 - cos)).sum()
            (g,) = torch.autograd.grad(energy, X)
        return torch.where(self.free, (self.F - g) / self.mass, 0.0)

    def _stencil(self, X, comp):
        """Flat node numbers and weights [M, 27] of component comp's lattice (non-unknowns weigh nothing)."""
        wl, n, node, weight = self.wl, (self.wl.nx, self.wl.ny, self.wl.nz), [], []
        for d in range(3):
            r = X[:, d] / self.h - (0.0 if d == comp else 0.5)
            i = torch.round(r).long()[:, None] + torch.arange(-1, 2, device="cuda")
            w = _delta(i - r[:, None])
            if d == 0:
                ok = (i >= (1 if comp == 0 else 0)) & (i < wl.nx)
                i, w = torch.where(ok, i, 0), torch.where(ok, w, 0.0)
            node.append(i if d == 0 else i % n[d])
            weight.append(w)
        at = (node[0][:, :, None, None] * wl.ny + node[1][:, None, :, None]) * wl.nz + node[2][:, None, None, :]
        w = weight[0][:, :, None, None] * weight[1][:, None, :, None] * weight[2][:, None, None, :]
        return at.reshape(len(X), -1), w.reshape(len(X), -1)

    def _force(self, q, dt):
        if self.alpha:
            for a, f in zip(q, self.alpha):
                a *= 1 - f
        X = torch.cat([self.X, self.Xb]) if self.X is not None else self.Xb
        if not len(X):
            return
        target = torch.zeros_like(X)
        nf = len(self.X) if self.X is not None else 0
        if nf:
            target[:nf] = self.V
        star = torch.empty_like(X)
        for c in range(3):
            at, w = self._stencil(X, c)
            star[:, c] = (w * q[c].view(-1)[at]).sum(dim=1)
            q[c].view(-1).index_add_(0, at.view(-1), (w * (self.dv / self.h ** 3 * (target - star)[:, c])[:, None]).view(-1))
        if nf:
            self.F = -(target - star)[:nf] / dt * self.dv[:nf, None]
            sub = max(1, math.ceil(dt * self.omega / 1.8))
            acc = self._acc()
            for _ in range(sub):
                self.V = self.V + 0.5 * dt / sub * acc
                self.X = self.X + dt / sub * self.V
                acc = self._acc()
                self.V = self.V + 0.5 * dt / sub * acc
            self.V = torch.where(self.free, self.V, 0.0)

    # operators
    def _ghost(self, c):
        q = self.q[c]
        first = -q[:1] if self.qin[c] is None else 2 * self.qin[c] - q[:1]
        return torch.cat([first, q])

    def _explicit(self):
        """The advection term (flux form) and the Laplacian of each component, on the unknowns' planes."""
        u, v, w = self.q
        nx, h = self.wl.nx, self.h
        up = lambda a, d: torch.roll(a, -1, d)  # noqa: E731
        dn = lambda a, d: torch.roll(a, 1, d)   # noqa: E731
        vg, wg, vi, wi = self._ghost(1), self._ghost(2), v[:nx], w[:nx]
        xx, yy, zz = ((0.5 * (a + b)) ** 2 for a, b in ((u[1:], u[:-1]), (vi, up(vi, 1)), (wi, up(wi, 2))))
        xy = 0.25 * (u + dn(u, 1)) * (vg[:-1] + vg[1:])
        xz = 0.25 * (u + dn(u, 2)) * (wg[:-1] + wg[1:])
        yz = 0.25 * (vi + dn(vi, 2)) * (wi + dn(wi, 1))
        N = [xx[1:] - xx[:-1] + (up(xy, 1) - xy)[1:nx] + (up(xz, 2) - xz)[1:nx],
             xy[1:] - xy[:-1] + yy - dn(yy, 1) + up(yz, 2) - yz,
             xz[1:] - xz[:-1] + up(yz, 1) - yz + zz - dn(zz, 2)]

        def lap(g):
            m = g[1:-1]
            return g[2:] + g[:-2] + up(m, 1) + dn(m, 1) + up(m, 2) + dn(m, 2) - 6 * m
        return [a / h for a in N], [lap(g) / h ** 2 for g in (u, vg, wg)]

    def _grad(self, p):
        return [(p[1:] - p[:-1]) / self.h, (p - torch.roll(p, 1, 1)) / self.h, (p - torch.roll(p, 1, 2)) / self.h]

    def _div(self):
        u, v, w = self.q
        v, w = v[:self.wl.nx], w[:self.wl.nx]
        return (u[1:] - u[:-1] + torch.roll(v, -1, 1) - v + torch.roll(w, -1, 2) - w) / self.h

    def _poisson(self, D):
        nx = self.wl.nx
        hat = (self.C @ D.reshape(nx, -1)).view_as(D)
        hat = torch.fft.fft2(hat) / self.lam
        hat[0, 0, 0] = 0.0
        return (self.C.T @ torch.fft.ifft2(hat).real.reshape(nx, -1)).view_as(D)

    def _project(self, phi, dt):
        for c, g in enumerate(self._grad(phi)):
            self.q[c][1 if c == 0 else 0:self.wl.nx] -= dt * g

    def _implicit(self, b, r, comp, first, last):
        """(1 - r D_x)(1 - r D_y)(1 - r D_z) increment = b; first, last: the boundary increments along x."""
        m = b.shape[0]
        A = torch.diag(torch.full((m,), 1 + 2 * r, dtype=b.dtype, device=b.device))
        off = torch.full((m - 1,), -r, dtype=b.dtype, device=b.device)
        A += torch.diag(off, 1) + torch.diag(off, -1)
        if comp:
            A[0, 0] = 1 + 3 * r
        b[-1] += r * last
        if first is not None:
            b[0] += (r if comp == 0 else 2 * r) * first
        x = torch.linalg.solve(A, b.reshape(m, -1)).view_as(b)
        ly, lz = self.lam_yz
        return torch.fft.ifft2(torch.fft.fft2(x) / ((1 - r * ly)[:, None] * (1 - r * lz))).real

    def step(self, planes=None):
        wl, h, nu, nx, q = self.wl, self.h, self.nu, self.wl.nx, self.q
        if wl.dt > 0:
            dt = wl.dt
        else:
            c = [0.5 * (q[0][1:] + q[0][:-1])] + [0.5 * (a[:nx] + torch.roll(a[:nx], -1, d)) for d, a in ((1, q[1]), (2, q[2]))]
            dt = wl.cfl * h / float(sum(a.abs() for a in c).max())
        beta = 0.0 if self.N is None else -dt / (2 * self.dt_old)
        out = [a[nx] - dt / h * (a[nx] - a[nx - 1]) for a in q]
        N, L = self._explicit()
        G, r = self._grad(self.p), nu * dt / (2 * h * h)
        inc = [None] * 3
        if planes is not None:
            face = planes[0] - planes[0].mean() + 1.0
            old = [0.0 if a is None else a for a in self.qin]
            inc = [face - q[0][0], planes[1] - old[1], planes[2] - old[2]]
        star = []
        for c in range(3):
            rhs = dt * (nu * L[c] - G[c] - (1 - beta) * N[c] - (beta * self.N[c] if self.N else 0.0))
            d = self._implicit(rhs, r, c, inc[c], out[c] - q[c][nx])
            a = q[c].clone()
            a[1 if c == 0 else 0:nx] += d
            a[nx] = out[c]
            star.append(a)
        if planes is not None:
            star[0][0] = face
            self.qin = [None, planes[1], planes[2]]
        self._force(star, dt)
        star[0][nx] += (star[0][0] - star[0][nx]).sum() * h * h / (wl.ly * wl.lz)
        self.q = star
        phi = self._poisson(self._div() / dt)
        self._project(phi, dt)
        g = torch.cat([phi[:1], phi, phi[-1:]])
        lap = g[2:] + g[:-2] + sum(torch.roll(phi, s, d) for s in (1, -1) for d in (1, 2)) - 6 * phi
        self.p = self.p + phi - 0.5 * nu * dt / h ** 2 * lap
        self.N, self.dt_old = N, dt


def _network(flat, blocks):
    """[(W [9, out, in], b)] from the flat parameters."""
    out, at = [], 0
    for o, i in [(128, 6)] + [(128, 128)] * blocks + [(3, 128)]:
        out.append((flat[at:at + 9 * o * i].view(9, o, i), flat[at + 9 * o * i:at + 9 * o * i + o]))
        at += 9 * o * i + o
    return out


def _conv(layer, x):
    W, b = layer
    y = b[:, None]
    for tap in range(9):
        y = y + W[tap] @ torch.roll(x, (1 - tap // 3, 1 - tap % 3), (1, 2)).reshape(x.shape[0], -1)
    return y.view(-1, *x.shape[1:])


def _forward(net, x):
    act = lambda a: torch.where(a > 0, a, a / 8)  # noqa: E731
    a = _conv(net[0], x)
    for layer in net[1:-1]:
        a = a + _conv(layer, act(a))
    return _conv(net[-1], act(a))


def _gaussian(key, counter):
    """Box-Muller of SplitMix64 (Steele, Lea and Flood 2014), as the training noise is documented."""
    with np.errstate(over="ignore"):
        z = np.uint64(key) + (counter + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    u1, u2 = (z >> np.uint64(32)).astype(np.float64), (z & np.uint64(0xFFFFFFFF)).astype(np.float64)
    return np.sqrt(-2 * np.log((u1 + 1) / 2.0 ** 32)) * np.cos(2 * np.pi * u2 / 2.0 ** 32)


def _exact_generator(case, seed):
    ny, nz, batch = case["ny"], case["nz"], case["batch"]
    train = case["what"] == "train"
    if (3 if train else 1) * case["steps"] * batch * _conv_flops(ny, nz, case["blocks"]) > 1e13:
        return None                                     # over twenty seconds in 64 bits
    w = torch.as_tensor(inputs.generator_params(seed, 128, case["blocks"], 6)).cuda()
    if not train:
        net = _network(w, case["blocks"])
        pair = [(q.double().movedim(-1, 1), p.double().movedim(-1, 1)) for q, p in _forward_inputs(case, seed)]
        return [torch.stack([_forward(net, torch.cat([q[b], p[b]])) for b in range(batch)]).movedim(1, -1) for q, p in pair]
    planes = _record(ny, nz, 64, seed)
    mean, std, _, _ = (torch.as_tensor(a, device="cuda") for a in inflow.data_norm(planes))
    rng, m, v = np.random.default_rng(seed), torch.zeros_like(w), torch.zeros_like(w)
    for t in range(1, case["steps"] + 1):
        idx, grad, loss = _samples(rng, case), torch.zeros_like(w), 0.0
        for b, i in enumerate(idx):
            new, q, old = ((planes[k].double() - mean[:, None, None]) / std[:, None, None] for k in (i + STRIDE, i, i - STRIDE))
            pixel = (np.uint64(b) * np.uint64(ny * nz) + np.arange(ny * nz, dtype=np.uint64)) * np.uint64(6)
            noise = np.stack([_gaussian(17 + t - 1, pixel + np.uint64(c)) for c in range(6)]).reshape(6, ny, nz)
            x = torch.cat([q, old]) + NOISE * torch.as_tensor(noise).cuda()
            with torch.enable_grad():
                leaf = w.detach().requires_grad_()
                part = (_forward(_network(leaf, case["blocks"]), x) - (new - x[:3])).square().sum() / (batch * 3 * ny * nz)
                (g,) = torch.autograd.grad(part, leaf)
            grad, loss = grad + g, loss + float(part)
        m, v = 0.9 * m + 0.1 * grad, 0.999 * v + 0.001 * grad * grad
        w = w - 5e-4 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return {"loss": loss, "params": w}
