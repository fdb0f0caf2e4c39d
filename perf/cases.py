"""The work a user of this library has it do, as a list of timed cases.

Every case is one call sequence through the public entry points (the
``Simulation``, ``Batch`` and ``UNet`` classes and the C ABI behind them), on
inputs made from a seed alone.  ``listed`` names the workloads of the
configurations, tests and benchmark of this repository; ``draw`` gives more of
the same ranges, odd and ragged sizes among them.  ``exact`` states the same
computation in plain FP64 torch.

Kinds:
  lb        lbm_step on one domain, then the device-side field readback a
            surrogate or a recorder takes (fields_nhwc)
  sweep     lbm_batch_step on many uneven domains, then every domain's fields
  flow      lbm_step_flow: the flow model alone past a frozen solid
  metrics   lbm_get_metrics: tips, solid fraction, conserved sums, to the host
  forward   one surrogate prediction
  train     one training step of the surrogate, and its gradients
  conv      one 3 x 3 convolution layer of it
"""
import ctypes
import math

import numpy as np
import torch

from paper_2209_01444_gb300 import lbm as L
from paper_2209_01444_gb300 import surrogate as S
from paper_2209_01444_gb300 import workloads as W

STORAGE_BYTES = {"fp32": 24 * 4, "fp16": 21 * 2 + 3 * 4, "bf16": 21 * 2 + 3 * 4}  # populations of a node


def _lb(name, scene, nx, ny, storage, steps, seeds):
    return {"name": name, "kind": "lb", "scene": scene, "nx": nx, "ny": ny, "storage": storage, "steps": steps,
            "seeds": seeds}


def listed():
    return [
        # the plain method on its smallest grid, as parity checks and short studies run it: latency counts
        _lb("box_128", "box", 128, 128, "fp32", 64, 1),
        # the dendrite in forced flow, one 50-step window, as the rollouts and the tip recorder advance it
        _lb("forced_1024", "forced", 1024, 1024, "fp32", 50, 1),
        # a ragged mid-size grid in the other 16-bit storage, walls on all sides
        _lb("forced_777x500_bf16", "forced", 777, 500, "bf16", 50, 1),
        # multi-seed thermosolutal convection at production size, plain and half-precision storage
        _lb("multi_4096", "multi", 4096, 4096, "fp32", 16, 64),
        _lb("multi_4096_fp16", "multi", 4096, 4096, "fp16", 16, 64),
        # the paper's alloy in flow with its two time scales: 15 flow sub-steps in each coupled step
        _lb("alloy_flow_1024", "alloy", 1024, 1024, "fp32", 4, 1),
        # a parameter sweep of uneven domains in one batch, FP16 storage
        {"name": "sweep_48_fp16", "kind": "sweep", "count": 48, "lmin": 128, "lmax": 1024, "storage": "fp16",
         "steps": 16},
        # flow past the stationary cylinder: the flow model alone on the paper's (70 x 40) R_s grid
        {"name": "cylinder_1400x800", "kind": "flow", "nx": 1400, "ny": 800, "storage": "fp32", "steps": 32},
        # the reductions a long run records as it goes
        {"name": "metrics_2048", "kind": "metrics", "nx": 2048, "ny": 2048, "storage": "fp32"},
        # one surrogate prediction of the whole 1024 x 1024 field
        {"name": "unet_forward_1024", "kind": "forward", "batch": 1, "h": 1024, "w": 1024},
        # one training step on 512 x 512 patches
        {"name": "unet_train_4x512", "kind": "train", "batch": 4, "h": 512, "w": 512},
        # the surrogate's widest layer alone: 32 -> 32 channels at full resolution
        {"name": "conv_4x512_32", "kind": "conv", "batch": 4, "h": 512, "w": 512, "cin": 32, "cout": 32},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lb", "lb", "lb", "lb", "sweep", "flow", "metrics", "forward", "train", "conv"])
    if kind == "lb":
        scene = rng.choice(["box", "forced", "multi", "alloy"])
        storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
        nx, ny = _log_int(rng, 64, 2400), _log_int(rng, 64, 2400)
        nodes = nx * ny
        steps = rng.randint(2, 6) if scene == "alloy" else max(8, min(rng.randint(16, 64), int(1.5e8 / nodes)))
        return {"kind": kind, "scene": scene, "nx": nx, "ny": ny, "storage": storage, "steps": steps,
                "seeds": rng.randint(2, 16) if scene == "multi" else 1}
    if kind == "sweep":
        return {"kind": kind, "count": rng.randint(8, 48), "lmin": rng.randint(64, 160), "lmax": rng.randint(300, 1024),
                "storage": rng.choice(["fp16", "fp16", "bf16", "fp32"]), "steps": rng.randint(8, 20)}
    if kind == "flow":
        return {"kind": kind, "nx": _log_int(rng, 96, 2000), "ny": _log_int(rng, 96, 1200),
                "storage": rng.choice(["fp32", "fp32", "fp16"]), "steps": rng.randint(8, 40)}
    if kind == "metrics":
        return {"kind": kind, "nx": _log_int(rng, 100, 2048), "ny": _log_int(rng, 100, 2048),
                "storage": rng.choice(["fp32", "fp16", "bf16"])}
    if kind == "conv":
        cin, cout = rng.choice([32, 64, 128, 256]), rng.choice([32, 64, 128, 256])
        w = rng.choice([32, 64, 128, 256, 384, 512])
        h = 16 * rng.randint(2, 32)
        batch = max(1, min(rng.randint(1, 4), int(2.0e10 / (9 * cin * cout * w * h))))
        return {"kind": kind, "batch": batch, "h": h, "w": w, "cin": cin, "cout": cout}
    # network inputs: sides multiples of 16; batch * (h/16) * (w/16) a multiple of 8
    while True:
        side = _log_int(rng, 64, 1024) if kind == "forward" else _log_int(rng, 64, 512)
        h, w = max(4, side // 16) * 16, max(4, int(side * rng.uniform(0.7, 1.4)) // 16) * 16
        batch = rng.choice([1, 1, 2, 4]) if kind == "forward" else rng.choice([1, 2, 4])
        if (batch * (h // 16) * (w // 16)) % 8 == 0 and batch * h * w <= 1024 * 1024:
            return {"kind": kind, "batch": batch, "h": h, "w": w}


# ------------------------------------------------------------------ problems
def _problem(case, seed):
    """(parameters, seeds, U0, theta0) of a single-domain case."""
    rng = np.random.Generator(np.random.PCG64(seed))
    nx, ny = case["nx"], case["ny"]
    scene = case.get("scene", "cylinder")
    r = float(rng.uniform(6.0, 10.0))
    # one seed near the workload's place, away from the walls
    cx = (0.375 if scene == "forced" else 0.5) * nx + float(rng.uniform(-2.0, 2.0))
    cy = 0.5 * ny + float(rng.uniform(-2.0, 2.0))
    flow_walls = ("inflow", "outflow", "symmetry", "symmetry")
    if scene == "box":
        p = W.thermosolutal_params(nx, ny, gbetaT=W.GBETA_T, gbetaC=W.GBETA_C)
        return p, np.array([[cx, cy, r, 0.0]]), 0.0, -0.55
    if scene == "forced":
        p = W.thermosolutal_params(nx, ny, bc=flow_walls, u_in=(0.01 * W.DX / W.DT, 0.0))
        return p, np.array([[cx, cy, r, float(rng.uniform(0.0, math.pi / 4))]]), 0.0, -0.55
    if scene == "multi":
        p = W.thermosolutal_params(nx, ny, eps_s=0.04, gbetaT=W.GBETA_T, gbetaC=W.GBETA_C, theta_ref=-0.45,
                                   bc=("periodic", "periodic", "noslip", "noslip"))
        n = case["seeds"]
        seeds = np.column_stack([rng.uniform(0.1 * nx, 0.9 * nx, n), rng.uniform(0.1 * ny, 0.9 * ny, n),
                                 rng.uniform(6.0, 10.0, n), rng.uniform(0.0, math.pi / 4, n)])
        return p, seeds, 0.0, -0.45
    if scene == "alloy":
        p = W.solutal_params(nx, flow=True, ny=ny)
        return p, np.array([[cx, cy, r, 0.0]]), -0.55, 0.0
    # flow past a disc of radius R at (20 R, 20 R) scaled to the grid, Re = 40
    R = 20.0 * nx / 1400.0 + float(rng.uniform(0.0, 1.0))
    p = W.cylinder_flow(nx=nx, ny=ny).params
    return p, np.array([[0.2857 * nx, 0.5 * ny, R, 0.0]]), 0.0, -0.55


def _sweep_domains(case, seed):
    # the sides follow the case, so that every seed's batch holds as many nodes
    sides = W.batch_domains(case["count"], 4, case["lmin"], case["lmax"])
    rng = np.random.Generator(np.random.PCG64(seed))
    for c in sides:
        n = c.params["nx"]
        delta = float(rng.uniform(0.3, 0.7))
        c.params.update(eps_s=float(rng.uniform(0.02, 0.06)), theta_ref=-delta,
                        u_in=(float(rng.uniform(0.0, 0.02)) * W.DX / W.DT, 0.0))
        c.theta0 = -delta
        c.seeds = np.array([[0.375 * n, 0.5 * n, 8.0, float(rng.uniform(0.0, math.pi / 4))]])
    return sides


def _smooth(g, b, h, w, modes=4):
    """Smooth periodic random fields [b, h, w] in about [-1, 1], FP64 on the GPU."""
    y = torch.arange(h, device="cuda", dtype=torch.float64)[:, None] * (2 * math.pi / h)
    x = torch.arange(w, device="cuda", dtype=torch.float64)[None, :] * (2 * math.pi / w)
    a = torch.randn(b, modes, modes, 2, generator=g).double()
    out = torch.zeros(b, h, w, device="cuda", dtype=torch.float64)
    for i in range(b):
        for kx in range(modes):
            for ky in range(modes):
                if kx + ky:
                    out[i] += float(a[i, kx, ky, 0]) / (kx * kx + ky * ky) * torch.cos(
                        kx * x + ky * y + 3.0 * float(a[i, kx, ky, 1]))
        out[i] /= out[i].abs().max()
    return out


def _random_fields(g, b, h, w):
    """phi, C, theta, ux, uy [b, h, w, 5]: solid and liquid with interfaces of a few nodes, smooth fields around."""
    phi = torch.tanh(8.0 * _smooth(g, b, h, w, 3) - 2.0)
    return torch.stack([phi, 1.0 + 0.2 * _smooth(g, b, h, w), -0.55 + 0.2 * _smooth(g, b, h, w),
                        0.2 * _smooth(g, b, h, w), 0.2 * _smooth(g, b, h, w)], dim=-1)


def _metric_fields(case, seed):
    """phi, U, theta, ux, uy, p planes [6, ny, nx]: one solid disc in smooth fields."""
    g = torch.Generator().manual_seed(seed)
    ny, nx = case["ny"], case["nx"]
    f = _smooth(g, 5, ny, nx)
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None] - 0.5 * ny
    x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :] - 0.5 * nx
    r = (0.2 + 0.1 * float(torch.rand(1, generator=g))) * min(nx, ny)
    phi = torch.tanh((r * (1.0 + 0.05 * torch.cos(4.0 * torch.atan2(y, x))) - torch.hypot(x, y)) / math.sqrt(2.0))
    return torch.stack([phi, -0.2 + 0.2 * f[0], -0.5 + 0.2 * f[1], 0.2 * f[2], 0.2 * f[3], 0.01 * f[4]])


def _net_inputs(case, seed):
    """Inputs x, targets t, the parameter vector and the normalisation of the network."""
    g = torch.Generator().manual_seed(seed)
    b, h, w = case["batch"], case["h"], case["w"]
    x = _random_fields(g, b, h, w)
    std_in = (x - x.mean(dim=(0, 1, 2))).square().mean(dim=(0, 1, 2)).sqrt().cpu().numpy()
    mean = x.mean(dim=(0, 1, 2)).cpu().numpy()
    t = x + torch.from_numpy(0.05 * std_in).cuda() * _random_fields(g, b, h, w)
    params = []
    for name, shape in S.param_shapes():
        v = torch.randn(shape, generator=g)
        if name.endswith(".b"):
            v *= 0.01
        else:  # He-normal, a small output projection, as the training starts
            v *= math.sqrt(2.0 / shape[1]) * (0.01 if name.startswith("out") else 1.0)
        params.append(v.reshape(-1))
    norm = [np.asarray(a, np.float32) for a in (mean, std_in, 0.05 * std_in)]
    return x.float(), t.float(), torch.cat(params).numpy(), norm


def _conv_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    b, h, w, cin, cout = (case[k] for k in ("batch", "h", "w", "cin", "cout"))
    x = torch.relu(torch.randn(b, h, w, cin, generator=g, device="cuda")).bfloat16()
    k = (torch.randn(cout, 9 * cin, generator=g, device="cuda") * math.sqrt(2.0 / (9 * cin))).bfloat16()
    return x, k, torch.randn(cout, generator=g, device="cuda") * 0.01


# ------------------------------------------------------------------- the API
def prepare(case, seed):
    kind = case["kind"]
    if kind == "lb" or kind == "flow":
        p, seeds, U0, theta0 = _problem(case, seed)
        sim = L.Simulation(p, storage=case["storage"])
        sim.init_seeds(seeds, U0, theta0)
        out = torch.empty(case["ny"], case["nx"], 5, device="cuda")
        return {"kind": kind, "sim": sim, "steps": case["steps"], "out": out}
    if kind == "sweep":
        cases = _sweep_domains(case, seed)
        b = L.Batch([c.params for c in cases], storage=case["storage"])
        outs = []
        for d, c in enumerate(cases):
            b.init_seeds(d, c.seeds, c.U0, c.theta0)
            outs.append(torch.empty(c.params["ny"], c.params["nx"], 5, device="cuda"))
        b.set_tiling(4, 1)  # what the tuner picks for such sweeps
        return {"kind": kind, "batch": b, "steps": case["steps"], "outs": outs}
    if kind == "metrics":
        p = W.thermosolutal_params(case["nx"], case["ny"], gbetaT=W.GBETA_T, gbetaC=W.GBETA_C)
        sim = L.Simulation(p, storage=case["storage"])
        sim.init_fields(_metric_fields(case, seed).cpu().numpy())
        return {"kind": kind, "sim": sim, "at": (0.5 * case["nx"], 0.5 * case["ny"])}
    if kind == "conv":
        x, k, bias = _conv_inputs(case, seed)
        out = torch.empty(*x.shape[:3], case["cout"], dtype=torch.bfloat16, device="cuda")
        return {"kind": kind, "lib": L.load(), "x": x, "k": k, "bias": bias, "out": out}
    x, t, vec, norm = _net_inputs(case, seed)
    net = S.UNet(case["batch"], case["h"], case["w"])
    net.set_params(vec)
    net.set_norm(*norm)
    return {"kind": kind, "net": net, "x": x, "t": t, "y": torch.empty_like(x)}


def run(s):
    kind = s["kind"]
    if kind == "lb":
        s["sim"].step(s["steps"])
        return s["sim"].fields_nhwc(s["out"])
    if kind == "flow":
        s["sim"].step_flow(s["steps"])
        return s["sim"].fields_nhwc(s["out"])
    if kind == "sweep":
        s["batch"].step(s["steps"])
        return [s["batch"].fields_nhwc(d, out) for d, out in enumerate(s["outs"])]
    if kind == "metrics":
        return s["sim"].metrics(*s["at"])
    if kind == "conv":
        x, k, out = s["x"], s["k"], s["out"]
        b, h, w, cin = x.shape
        p = ctypes.c_void_p
        rc = s["lib"].lbm_nn_conv3x3(p(x.data_ptr()), b, h, w, cin, cin, p(k.data_ptr()), 9 * cin, p(out.data_ptr()),
                                     out.shape[3], p(s["bias"].data_ptr()), out.shape[3], 0, 1,
                                     p(torch.cuda.current_stream().cuda_stream))
        if rc != L.LBM_OK:
            raise L.LBMError(rc, "lbm_nn_conv3x3")
        return out
    if kind == "forward":
        return s["net"].forward(s["x"], s["y"])
    s["net"].train_step(s["x"], s["t"], 1e-4)
    return s["net"].grads()


def work(case):
    """One coupled step reads and writes every population and history value once (48 bytes of history); its flow
    sub-steps, and the steps of a flow-only call, work on what was read.  Operations per node: about 450 of a coupled
    step, 130 of a flow step.  Networks: inputs, outputs and parameters once (a training step: parameters and the two
    Adam moments read and written, gradients written), two operations per multiply-add, three passes in training."""
    kind = case["kind"]
    if kind == "lb":
        nodes = case["nx"] * case["ny"]
        sub = 14 if case["scene"] == "alloy" else 0
        return {"bytes": nodes * (case["steps"] * (2 * STORAGE_BYTES[case["storage"]] + 48) + 20),
                "flops": nodes * case["steps"] * (450 + 130 * sub)}
    if kind == "sweep":
        nodes = sum(c.nodes for c in W.batch_domains(case["count"], 4, case["lmin"], case["lmax"]))
        return {"bytes": nodes * (case["steps"] * (2 * STORAGE_BYTES[case["storage"]] + 48) + 20),
                "flops": nodes * case["steps"] * 450}
    if kind == "flow":
        nodes = case["nx"] * case["ny"]
        flow = 36 if case["storage"] == "fp32" else 18
        return {"bytes": nodes * (STORAGE_BYTES[case["storage"]] + flow + 20), "flops": nodes * case["steps"] * 130}
    if kind == "metrics":
        nodes = case["nx"] * case["ny"]
        return {"bytes": nodes * STORAGE_BYTES[case["storage"]], "flops": nodes * 60}
    if kind == "conv":
        px = case["batch"] * case["h"] * case["w"]
        return {"bytes": 2 * (px * (case["cin"] + case["cout"]) + 9 * case["cin"] * case["cout"]),
                "flops": 2 * 9 * px * case["cin"] * case["cout"]}
    px = case["batch"] * case["h"] * case["w"]
    macs = params = 0
    for name, shape in S.param_shapes():
        params += int(np.prod(shape))
        if name.endswith(".W"):
            level = 0 if name.startswith("out") else int(name[3 if name[0] in "ed" else 2])
            macs += int(np.prod(shape)) * px // 4 ** (level + (1 if name.startswith("up") else 0))
    if kind == "forward":
        return {"bytes": 2 * px * 20 + 4 * params, "flops": 2 * macs}
    return {"bytes": 2 * px * 20 + 4 * params * 7, "flops": 6 * macs}


# --------------------------------------------------------- the method in FP64
C5 = ((0, 0), (1, 0), (0, 1), (-1, 0), (0, -1))
C9 = C5 + ((1, 1), (-1, 1), (-1, -1), (1, -1))
W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


class _Exact:
    """The four lattice Boltzmann models on one domain, whole populations in FP64 torch."""

    def __init__(self, p):
        self.p = p
        W_, tau, ns = p["W0"] / p["dx"], p["tau0"] / p["dt"], p["n_sub"]
        dtf, dx = p["dt"] / ns, p["dx"]
        self.W, self.tau, self.ns, self.vf = W_, tau, ns, dtf / dx
        self.kappa = 3.0 * W_ * W_ / tau
        self.D = p["D"] * p["dt"] / dx**2
        self.sC = 1.0 / (3.0 * self.D * (1.0 - p["k"]) + 0.5)
        self.sT = 1.0 / (3.0 * p["alpha"] * p["dt"] / dx**2 + 0.5)
        self.sU = 1.0 / (3.0 * p["nu"] * dtf / dx**2 + 0.5)
        ff = dtf * dtf / dx
        self.Fx, self.Fy = p["force"][0] * ff, p["force"][1] * ff
        self.gT, self.gC = p["gbetaT"] * ff, p["gbetaC"] * ff
        self.lat = 0.0 if p["isothermal"] else 0.5
        self.bc = p["bc"]
        self.px, self.py = self.bc[0] == "periodic", self.bc[2] == "periodic"
        self.uin = (p["u_in"][0] * self.vf, p["u_in"][1] * self.vf)

    # macros of Eqs. (15), (20), (23), (26); pops: dict of lists f, n, g, h
    def U_of(self, C, phi):
        k = self.p["k"]
        return (2.0 * C / (1.0 + k - (1.0 - k) * phi) - 1.0) / (1.0 - k)

    def flow_macros(self, h, phi, Fy):
        jx, jy = h[1] - h[3] + h[5] - h[6] - h[7] + h[8], h[2] - h[4] + h[5] + h[6] - h[7] - h[8]
        rest = h[1] + h[2] + h[3] + h[4] + h[5] + h[6] + h[7] + h[8]
        w = 0.5 * (1.0 + phi)  # 1 - q~
        sx, sy = jx + 0.5 * self.Fx, jy + 0.5 * Fy
        ux, uy = sx - 0.5 * w * sx, sy - 0.5 * w * sy
        return ux, uy, 0.6 * (rest - (2.0 / 3.0) * (ux * ux + uy * uy)), self.Fx - w * sx, Fy - w * sy

    def macros(self, f, n, g, h):
        phi, C, H = sum(f), sum(n), sum(g)
        th = H + self.lat * phi
        Fy = self.Fy + self.gT * (th - self.p["theta_ref"]) + self.gC * (C - self.p["C_ref"])
        ux, uy, p, Fpx, Fpy = self.flow_macros(h, phi, Fy)
        return {"phi": phi, "C": C, "H": H, "th": th, "U": self.U_of(C, phi), "ux": ux, "uy": uy, "p": p, "Fpx": Fpx,
                "Fpy": Fpy, "Fy": Fy}

    def eq_phi(self, phi):
        return [phi / 3.0] + [phi / 6.0] * 4

    def eq_scalar(self, A, Cv, jx, jy):
        return [A - (2.0 / 3.0) * Cv, Cv / 6.0 + 0.5 * jx, Cv / 6.0 + 0.5 * jy, Cv / 6.0 - 0.5 * jx, Cv / 6.0 - 0.5 * jy]

    def eq_flow(self, p, ux, uy):
        uu = 1.5 * (ux * ux + uy * uy)
        out = [self.p["rho0"] - (5.0 / 3.0) * p - (4.0 / 9.0) * uu]
        for (cx, cy), w in zip(C9[1:], W9[1:]):
            cu = cx * ux + cy * uy
            out.append(w * (3.0 * p + 3.0 * cu + 4.5 * cu * cu - uu))
        return out

    def eq_all(self, phi, C, U, th, ux, uy, p):
        H, s = th - self.lat * phi, self.ns
        return (self.eq_phi(phi), self.eq_scalar(C, 0.5 * (1.0 - phi) * U, C * ux * s, C * uy * s),
                self.eq_scalar(H, th, H * ux * s, H * uy * s), self.eq_flow(p, ux, uy))

    def Q(self, phi, th, U):
        w = 1.0 - phi * phi
        return phi * w - self.p["lambda_"] * (th + self.p["Mc_inf"] * U) * w * w

    def start(self, phi, U, th, ux, uy, p, co, so):
        k = self.p["k"]
        C = 0.5 * (1.0 + k - (1.0 - k) * phi) * (1.0 + (1.0 - k) * U)
        self.f, self.n, self.g, self.h = self.eq_all(phi, C, U, th, ux, uy, p)
        self.co, self.so = co, so
        m = self.macros(self.f, self.n, self.g, self.h)
        self.remember(m)

    def remember(self, m):
        s = self.ns
        self.hist = (m["phi"], self.Q(m["phi"], m["th"], m["U"]), m["C"] * m["ux"] * s, m["C"] * m["uy"] * s,
                     m["H"] * m["ux"] * s, m["H"] * m["uy"] * s)

    def seeds(self, seeds, U0, theta0):
        nx, ny = self.p["nx"], self.p["ny"]
        y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None]
        x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :]
        best = near = None
        co = so = torch.zeros(ny, nx, device="cuda", dtype=torch.float64)
        for sx, sy, R, o in np.asarray(seeds).tolist():
            dx, dy = x - sx, y - sy
            if self.px:
                dx = dx - nx * torch.round(dx / nx)
            if self.py:
                dy = dy - ny * torch.round(dy / ny)
            d = torch.hypot(dx, dy)
            a = (R - d) / (math.sqrt(2.0) * self.W)
            best = a if best is None else torch.maximum(best, a)
            closer = torch.ones_like(d, dtype=torch.bool) if near is None else d < near
            near = d if near is None else torch.minimum(near, d)
            co, so = torch.where(closer, math.cos(o), co), torch.where(closer, math.sin(o), so)
        z = torch.zeros_like(best)
        self.start(torch.tanh(best), z + U0, z + theta0, z, z, z, co, so)

    def grad(self, phi):
        q = torch.nn.functional.pad(phi[None, None], (1, 1, 0, 0), mode="circular" if self.px else "reflect")
        q = torch.nn.functional.pad(q, (0, 0, 1, 1), mode="circular" if self.py else "reflect")[0, 0]
        ny, nx = phi.shape
        at = lambda dx, dy: q[1 + dy:1 + dy + ny, 1 + dx:1 + dx + nx]  # noqa: E731
        e, w, n, s = at(1, 0), at(-1, 0), at(0, 1), at(0, -1)
        ne, nw, se, sw = at(1, 1), at(-1, 1), at(1, -1), at(-1, -1)
        return (e - w) / 3.0 + (ne - nw + se - sw) / 12.0, (n - s) / 3.0 + (ne - se + nw - sw) / 12.0

    def anisotropy(self, gx, gy):
        px, py = self.co * gx + self.so * gy, self.co * gy - self.so * gx
        m2 = px * px + py * py
        flat = m2 < 1e-12
        inv = 1.0 / torch.where(flat, 1.0, m2 * m2)
        eps = self.p["eps_s"]
        a = 1.0 - 3.0 * eps + 4.0 * eps * (px**4 + py**4) * inv
        t = 16.0 * eps * a * px * py * (px * px - py * py) * inv
        nx, ny = t * py, -t * px
        z = torch.zeros_like(a)
        return (torch.where(flat, 1.0, a), torch.where(flat, z, self.co * nx - self.so * ny),
                torch.where(flat, z, self.so * nx + self.co * ny))

    def collide5(self, d, A, Bx, By, Cv, s1, Gx, Gy, S0):
        m1, m2, k1 = d[1] - d[3], d[2] - d[4], 1.0 - 0.5 * s1
        r1, r2 = m1 - s1 * (m1 - Bx) + k1 * Gx, m2 - s1 * (m2 - By) + k1 * Gy
        e = (Cv + S0) / 3.0
        return [A + S0 - 2.0 * e, 0.5 * (e + r1), 0.5 * (e + r2), 0.5 * (e - r1), 0.5 * (e - r2)]

    def collide9(self, h, ux, uy, p, Fx, Fy):
        mxx = h[1] + h[3] + h[5] + h[6] + h[7] + h[8]
        myy = h[2] + h[4] + h[5] + h[6] + h[7] + h[8]
        mxy = h[5] - h[6] + h[7] - h[8]
        s = self.sU
        r1, r2 = ux + 0.5 * Fx, uy + 0.5 * Fy
        r3, r4 = mxx - s * (mxx - p - ux * ux), myy - s * (myy - p - uy * uy)
        r5, r6, r7 = mxy - s * (mxy - ux * uy), r2 / 3.0, r1 / 3.0
        r8 = (p + ux * ux + uy * uy) / 3.0
        return [self.p["rho0"] - r3 - r4 + r8, 0.5 * (r1 + r3 - r7 - r8), 0.5 * (r2 + r4 - r6 - r8),
                0.5 * (-r1 + r3 + r7 - r8), 0.5 * (-r2 + r4 + r6 - r8), 0.25 * (r5 + r6 + r7 + r8),
                0.25 * (-r5 + r6 - r7 + r8), 0.25 * (r5 - r6 - r7 + r8), 0.25 * (-r5 - r6 + r7 + r8)]

    @staticmethod
    def stream(v, dirs):
        return [torch.roll(a, (cy, cx), (0, 1)) if cx or cy else a for a, (cx, cy) in zip(v, dirs)]

    def wall(self, side, flow_only):
        """Non-equilibrium extrapolation on one side (0 left, 1 right, 2 bottom, 3 top)."""
        kind = self.bc[side]
        if kind == "periodic":
            return
        last = -1 if side % 2 else 0
        inner = -2 if side % 2 else 1
        if side < 2:
            b, i = (slice(None), last), (slice(None), inner)
        else:
            cols = slice(None) if self.px else slice(1, -1)
            b, i = (last, cols), (inner, cols)
        pick = lambda v: [a[i] for a in v]  # noqa: E731
        f, n, g, h = pick(self.f), pick(self.n), pick(self.g), pick(self.h)
        m = self.macros(f, n, g, h)
        ux = uy = torch.zeros_like(m["ux"])
        p = m["p"]
        if kind == "inflow":
            ux, uy = ux + self.uin[0], uy + self.uin[1]
        elif kind == "outflow":
            ux, uy, p = m["ux"], m["uy"], torch.zeros_like(p)
        elif kind == "symmetry":
            ux, uy = (ux, m["uy"]) if side < 2 else (m["ux"], uy)
        eb = self.eq_all(m["phi"], m["C"], m["U"], m["th"], ux, uy, p)
        ef = self.eq_all(m["phi"], m["C"], m["U"], m["th"], m["ux"], m["uy"], m["p"])
        for k, (pop, src) in enumerate(((self.f, f), (self.n, n), (self.g, g), (self.h, h))):
            if flow_only and k < 3:
                continue
            for q, a in enumerate(pop):
                a[b] = eb[k][q] + src[q] - ef[k][q]

    def walls(self, flow_only=False):
        for side in (2, 3, 0, 1):
            self.wall(side, flow_only)

    def flow_step(self, phi, Fy):
        ux, uy, p, Fpx, Fpy = self.flow_macros(self.h, phi, Fy)
        self.h = self.stream(self.collide9(self.h, ux, uy, p, Fpx, Fpy), C9)
        self.walls(True)

    def step(self):
        f, n, g, h, p = self.f, self.n, self.g, self.h, self.p
        m = self.macros(f, n, g, h)
        phi0, Q0, Cx0, Cy0, Hx0, Hy0 = self.hist
        self.remember(m)
        _, Q, Cx, Cy, Hx, Hy = self.hist
        gx, gy = self.grad(m["phi"])
        a, Nx, Ny = self.anisotropy(gx, gy)
        a2 = a * a
        fo = self.collide5(f, m["phi"], 0.0, 0.0, m["phi"], 1.0 / (self.kappa * a2 + 0.5), -Nx / (3.0 * a2),
                           -Ny / (3.0 * a2), (Q + 0.5 * a2 * (Q - Q0)) / self.tau)
        g2 = gx * gx + gy * gy
        c = -self.W / (2.0 * math.sqrt(2.0)) * (1.0 + (1.0 - p["k"]) * m["U"]) * (m["phi"] - phi0)
        c = torch.where(g2 < 1e-12, 0.0, c / torch.sqrt(torch.where(g2 < 1e-12, 1.0, g2)))
        Gx = (Cx - Cx0) + (-0.5 * m["U"] * gx + c * gx / self.D) / 3.0
        Gy = (Cy - Cy0) + (-0.5 * m["U"] * gy + c * gy / self.D) / 3.0
        no = self.collide5(n, m["C"], Cx, Cy, 0.5 * (1.0 - m["phi"]) * m["U"], self.sC, Gx, Gy, 0.0)
        go = self.collide5(g, m["H"], Hx, Hy, m["th"], self.sT, Hx - Hx0, Hy - Hy0, 0.0)
        ho = self.collide9(h, m["ux"], m["uy"], m["p"], m["Fpx"], m["Fpy"])
        # modified streaming of the phase field, Eq. (13)
        there = [torch.roll(v, (-cy, -cx), (0, 1)) for v, (cx, cy) in zip(f, C5)]
        fo = [v / a2 - (1.0 / a2 - 1.0) * t for v, t in zip(fo, there)]
        self.f, self.n, self.g = self.stream(fo, C5), self.stream(no, C5), self.stream(go, C5)
        self.h = self.stream(ho, C9)
        self.walls()
        for _ in range(1, self.ns):
            self.flow_step(m["phi"], m["Fy"])

    def fields(self):
        m = self.macros(self.f, self.n, self.g, self.h)
        return torch.stack([m["phi"], m["C"], m["th"], m["ux"] / self.vf, m["uy"] / self.vf], dim=-1)


def _exact_metrics(case, seed):
    p = W.thermosolutal_params(case["nx"], case["ny"], gbetaT=W.GBETA_T, gbetaC=W.GBETA_C)
    e = _Exact(p)
    v = _metric_fields(case, seed)
    one = torch.ones_like(v[0])
    e.start(v[0], v[1], v[2], v[3] * e.vf, v[4] * e.vf, v[5] * e.vf**2, one, 0.0 * one)
    m = e.macros(e.f, e.n, e.g, e.h)
    phi, (ny, nx) = m["phi"], v[0].shape
    cx, cy = 0.5 * nx, 0.5 * ny
    out = {}
    for key, (ex, ey) in {"tip_px": (1, 0), "tip_mx": (-1, 0), "tip_py": (0, 1)}.items():
        j = torch.arange(0, 2 * (nx + ny), device="cuda", dtype=torch.float64) * 0.5
        x, y = cx + j * ex, cy + j * ey
        ok = (x >= 0) & (y >= 0) & (x <= nx - 1) & (y <= ny - 1)
        x, y = x[ok], y[ok]
        i0, j0 = x.floor().long().clamp(max=nx - 2), y.floor().long().clamp(max=ny - 2)
        a, b = x - i0, y - j0
        s = ((1 - a) * (1 - b) * phi[j0, i0] + a * (1 - b) * phi[j0, i0 + 1] + (1 - a) * b * phi[j0 + 1, i0] +
             a * b * phi[j0 + 1, i0 + 1])
        k = int((s > 0).nonzero().max())
        out[key] = 0.5 * (k + (float(s[k] / (s[k] - s[k + 1])) if k + 1 < len(s) else 0.0))
    out["solid_fraction"] = float((0.5 * (1.0 + phi)).mean())
    out["sum_C"], out["sum_H"], out["sum_phi"] = (float(m[k].sum()) for k in ("C", "H", "phi"))
    out["sum_h"] = float(sum(h.sum() for h in e.h))
    out["max_u"] = float(torch.hypot(m["ux"], m["uy"]).max()) / e.vf
    out.update(nonfinite=0.0, step=None, rc=None)
    return out


# -------------------------------------------------------- the network in FP64
def _conv(x, k, bias):
    """3 x 3 zero-padded convolution of x [b, h, w, cin] with k [cout, (ky, kx, cin)]."""
    b, h, w, c = x.shape
    q = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    t = k.reshape(k.shape[0], 3, 3, c)
    out = bias
    for ky in range(3):
        for kx in range(3):
            out = out + q[:, ky:ky + h, kx:kx + w].reshape(-1, c) @ t[:, ky, kx].T
    return out.reshape(b, h, w, -1)


def _exact_net(case, seed):
    x, t, vec, norm = _net_inputs(case, seed)
    train = case["kind"] == "train"
    x, t = x.double(), t.double()
    mean, std_in, std_out = (torch.from_numpy(a).double().cuda() for a in norm)
    params, at = {}, 0
    for name, shape in S.param_shapes():
        size = int(np.prod(shape))
        v = torch.from_numpy(vec[at:at + size].reshape(shape)).double().cuda()
        params[name] = v.requires_grad_(train)
        at += size
    layer = lambda v, name: torch.relu(_conv(v, params[name + ".W"], params[name + ".b"]))  # noqa: E731
    v = torch.nn.functional.pad((x - mean) / std_in, (0, S.IN_PITCH - x.shape[3]))
    skips = []
    for l in range(S.LEVELS):
        v = layer(layer(v, f"enc{l}a"), f"enc{l}b")
        if l < S.LEVELS - 1:
            skips.append(v)
            b, h, w, c = v.shape
            v = v.reshape(b, h // 2, 2, w // 2, 2, c).amax(dim=(2, 4))
    for l in range(S.LEVELS - 2, -1, -1):
        b, h, w, c = v.shape
        u = v.reshape(-1, c) @ params[f"up{l}.W"].T + params[f"up{l}.b"]
        u = u.reshape(b, h, w, 2, 2, c // 2).permute(0, 1, 3, 2, 4, 5).reshape(b, 2 * h, 2 * w, c // 2)
        v = layer(layer(torch.cat([skips.pop(), u], dim=3), f"dec{l}a"), f"dec{l}b")
    out = v @ params["out.W"].T + params["out.b"]
    if not train:
        return x + std_out * out
    (out - (t - x) / std_out).square().mean().backward()
    return {name: v.grad for name, v in params.items()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "lb" or kind == "flow":
        p, seeds, U0, theta0 = _problem(case, seed)
        e = _Exact(p)
        e.seeds(seeds, U0, theta0)
        if kind == "flow":
            m = e.macros(e.f, e.n, e.g, e.h)
        for _ in range(case["steps"]):
            e.step() if kind == "lb" else e.flow_step(m["phi"], m["Fy"])
        return e.fields()
    if kind == "sweep":
        outs = []
        for c in _sweep_domains(case, seed):
            e = _Exact(c.params)
            e.seeds(c.seeds, c.U0, c.theta0)
            for _ in range(case["steps"]):
                e.step()
            outs.append(e.fields())
        return outs
    if kind == "metrics":
        return _exact_metrics(case, seed)
    if kind == "conv":
        x, k, bias = _conv_inputs(case, seed)
        return torch.relu(_conv(x.double(), k.double(), bias.double()))
    return _exact_net(case, seed)
