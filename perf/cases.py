"""What is timed: the work that programs have this solver do, through its public entry points.

A case is a dict of plain values.  Kinds:

  step      lb_step on one periodic grid, then the stored state (lb_get_state), in one of the
            modes: "plain", "walls" (a Couette channel), "nonideal" (isothermal fluid), "entropic"
            and "entropic_path" (exact entropic equilibrium), "stochastic" (BF16 store)
  batch     lb_batch_step of independent simulations on cubic grids of uneven edges
  snapshot  fields in, global sums, moments and populations out, populations back in
  apply     one application of the surrogate network
  layer     one convolution layer of the surrogate, forward and backward

listed() gives the cases timed by name, draw(rng) more of the same ranges, prepare(case, seed)
what a program holds before the call, run(state) one pass, work(case) the bytes and operations a
pass cannot do without, and exact(case, seed) what run returns for the same inputs in 64-bit torch
arithmetic, written from the model's formulas (arXiv:1909.08406).
"""
import itertools
import math

import numpy as np
import torch

from paper_1909_08406_gb300 import lb, sg
from paper_1909_08406_gb300 import surrogate as sur
from paper_1909_08406_gb300 import workloads as wl

F64 = torch.float64
DTYPE = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
SCALE = {"f64": 1.0, "f32": 1.0, "f16": 256.0, "bf16": 1.0}  # stored h times this
TAU = 0.01 / 0.2948964908710634  # viscosity 0.01
SR_SEED = 20191909
FLOPS_PER_NODE = 410  # moments and relaxation, about ten operations per velocity


def _step(name, nx, ny, nz, prec, steps, mode="plain", tau=TAU, eos=""):
    c = {"kind": "step", "nx": nx, "ny": ny, "nz": nz, "prec": prec, "steps": steps, "mode": mode, "tau": tau,
         "eos": eos}
    return {"name": name, **c} if name else c


def listed():
    return [
        # production runs: the benchmark's thermoacoustic case in 16-bit storage, half its grid so
        # that three states fit the card
        _step("box_f16", 512, 512, 256, "f16", 10),
        # the FP32 validation run (acoustic and thermal waves, 256^3)
        _step("cube_f32", 256, 256, 256, "f32", 10),
        # the FP64 parity run (32^3)
        _step("cube_f64", 32, 32, 32, "f64", 20),
        # the smallest runs, odd extents: launches and latency count
        _step("small_f32", 33, 18, 20, "f32", 100),
        # long BF16 runs store with stochastic rounding; ragged extents
        _step("stochastic_bf16", 150, 110, 90, "bf16", 20, "stochastic"),
        # a channel between kinetic walls (Couette, thermal flows)
        _step("walls_f32", 96, 80, 64, "f32", 20, "walls", 0.17),
        # two-phase work: the droplet box, van der Waals, 16-bit storage
        _step("nonideal_f16", 160, 200, 200, "f16", 5, "nonideal", 0.5, "vdw"),
        # the exact entropic equilibrium
        _step("entropic_f32", 64, 64, 64, "f32", 5, "entropic"),
        # a parameter sweep: uneven cubic grids, one relaxation time each
        {"name": "batch_f32", "kind": "batch", "edges": "32,48,64,96,128", "sims": 16, "prec": "f32", "steps": 10},
        # set up, diagnose, write a snapshot, restart from one
        {"name": "snapshot_f16", "kind": "snapshot", "nx": 192, "ny": 160, "nz": 144, "prec": "f16"},
        # a rollout hop of the surrogate (batch 1)
        {"name": "surrogate_apply", "kind": "apply", "batch": 1, "n": 64},
        # the layer a training step repeats four times, at its minibatch
        {"name": "surrogate_layer", "kind": "layer", "batch": 4, "nz": 64, "ny": 64, "cin": 32, "cout": 32,
         "dilation": 1},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["plain"] * 6 + ["stochastic", "walls", "walls", "nonideal", "nonideal", "entropic",
                                       "entropic_path", "batch", "snapshot", "apply", "layer", "layer"])
    if kind == "batch":
        edges = sorted(rng.sample([24, 32, 40, 48, 64, 72, 96, 128], rng.randint(2, 5)))
        return {"kind": "batch", "edges": ",".join(map(str, edges)), "sims": rng.randint(3, 20),
                "prec": rng.choice(["f32", "f32", "f16", "bf16"]), "steps": rng.randint(3, 12)}
    if kind == "apply":
        return {"kind": "apply", "batch": rng.randint(1, 6), "n": 64}
    if kind == "layer":
        d = rng.choice([1, 2, 4, 8])
        cin, cout = rng.choice([(16, 32), (32, 32), (32, 16)])
        return {"kind": "layer", "batch": rng.randint(1, 5), "nz": d * rng.randint(max(1, 24 // d), 80 // d),
                "ny": 4 * d * rng.randint(max(1, 8 // d), max(1, 20 // d)), "cin": cin, "cout": cout, "dilation": d}
    if kind == "snapshot":
        return {"kind": "snapshot", "nx": _log_int(rng, 17, 220), "ny": _log_int(rng, 17, 220),
                "nz": _log_int(rng, 17, 220), "prec": rng.choice(["f64", "f32", "f16", "bf16"])}
    prec = {"stochastic": ["bf16"], "plain": ["f16", "f16", "bf16", "f32", "f32", "f64"],
            "entropic": ["f64", "f32", "f32", "f16"], "entropic_path": ["f32", "f16"],
            "walls": ["f64", "f32", "f16"], "nonideal": ["f64", "f32", "f16", "bf16"]}[kind]
    prec = rng.choice(prec)
    slow = prec == "f64" or kind.startswith("entropic")
    top = 96 if slow else 340
    lo = 8 if kind == "walls" else 6
    nx, ny, nz = _log_int(rng, 12, top), _log_int(rng, lo, top), _log_int(rng, lo, top)
    if rng.random() < 0.5:  # rows of a multiple of 32, as production grids have
        nx = max(32, 32 * round(nx / 32))
    nodes = 2 * nx * ny * nz
    budget = (2.5e6 if kind == "entropic_path" else 1.2e7) if slow else 1.5e11 / (100 * BYTES[prec])
    steps = max(1, min(100, int(budget / nodes)))
    tau = 0.5 if kind == "nonideal" else round(math.exp(rng.uniform(math.log(0.03), math.log(1.0))), 4)
    eos = rng.choice(["vdw", "peng_robinson", "carnahan_starling"]) if kind == "nonideal" else ""
    return _step("", nx, ny, nz, prec, steps, kind, tau, eos)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _fields(nx, ny, nz, theta0, seed):
    """A Gaussian density pulse at a seeded place, shear waves, and a temperature field from a
    seeded Fourier box: the workloads' thermoacoustic recipe on any box, with a velocity."""
    r = np.random.default_rng(seed)
    X, Y, Z = wl.node_positions(nx, ny, nz, "cuda")
    r2 = 0
    for P, n in ((X, nx), (Y, ny), (Z, nz)):
        d = P - r.uniform(0, n)
        r2 = r2 + (d - n * torch.round(d / n)) ** 2
    rho = 1.0 + r.uniform(5e-3, 1e-2) * torch.exp(-r2 / (2 * r.uniform(4, 8) ** 2))
    del r2
    ph = r.uniform(0, 2 * math.pi, 3)
    amp = 4e-3
    u = torch.stack([amp * torch.sin(2 * math.pi * Y / ny + ph[0]), amp * torch.sin(2 * math.pi * Z / nz + ph[1]),
                     amp * torch.sin(2 * math.pi * X / nx + ph[2])])
    del X, Y, Z
    theta = theta0 * (1.0 + 1e-3 * wl.fourier_box_field(nx, ny, nz, seed + 7, kmax=4, device="cuda"))
    return rho.contiguous(), u.contiguous(), theta.contiguous()


def _walls(theta0):
    """Couette channel: still wall below, moving warmer wall above."""
    return (0.0, 0.0, theta0 * (1 - 1e-4)), (0.02, 0.0, theta0 * (1 + 1e-4))


KAPPA = 0.02
THETA_STAR = 1.1  # theta_0 / theta_c: one phase


class _Handle:
    """A context or batch of the library, destroyed with its last reference."""

    def __init__(self, h, destroy):
        self.h, self._destroy = h, destroy

    def __del__(self):
        if self.h:
            self._destroy(self.h)
            self.h = None


def _state_tensor(nx, ny, nz, prec):
    return torch.empty((2, 41, nz, ny, nx), dtype=DTYPE[prec], device="cuda")


def _batch_members(case, seed):
    edges = [int(e) for e in case["edges"].split(",")]
    n = [edges[k % len(edges)] for k in range(case["sims"])]
    tau = np.random.default_rng(4).uniform(0.51, 1.0, size=len(n))
    r = np.random.default_rng(seed)
    return n, [float(t) for t in tau], np.exp(r.uniform(math.log(1e-4), math.log(1e-2), size=len(n)))


def _layer_inputs(case, seed):
    d, b = case["dilation"], case["batch"]
    shape = (b * d * d, case["nz"] // d, case["ny"] // d, 64)
    g = torch.Generator(device="cuda").manual_seed(seed)

    def rnd(*s):
        return torch.randn(s, device="cuda", generator=g)

    cin, cout = case["cin"], case["cout"]
    x = rnd(*shape, cin).to(torch.bfloat16)
    w = (rnd(cout, 27, cin) / math.sqrt(27 * cin)).to(torch.bfloat16)
    bias = 0.1 * rnd(cout)
    z = rnd(*shape, cout)  # the pre-activation kept by an earlier forward pass
    dy = rnd(*shape, cout)
    return x, w, bias, z, dy


def _network_inputs(case, seed):
    """Weights of a trained network's size in every layer, and normalised fields."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    ws, bs = [], []
    for ci, co in ((16, 32), (32, 32), (32, 32), (32, 32), (32, 32), (32, 16)):
        ws.append(0.7 / math.sqrt(27 * ci) * torch.randn((co, 27, ci), device="cuda", generator=g))
        bs.append(0.05 * torch.randn(co, device="cuda", generator=g))
    n = case["n"]
    x = torch.zeros((case["batch"], n, n, n, 16), dtype=torch.bfloat16, device="cuda")
    for b in range(case["batch"]):
        rho, u, theta = _fields(n, n, n, 1.0, seed + 31 * b)
        for c, f in enumerate((rho[0] - 1, u[0, 0], u[1, 0], u[2, 0], theta[0] - 1)):
            x[b, ..., c] = (f / 5e-3).to(torch.bfloat16)
    return ws, bs, x


def prepare(case, seed):
    kind = case["kind"]
    if kind == "layer":
        x, w, bias, z, dy = _layer_inputs(case, seed)
        cin, cout, d = case["cin"], case["cout"], case["dilation"]
        act = sg.ACT_GELU if cout == 32 else sg.ACT_NONE
        out = x.shape[:-1] + (cout,)
        return {"kind": kind, "x": x, "w": w, "bias": bias, "z": z, "dy": dy, "act": act, "res": cin == cout,
                "xper": 64 // d, "y": torch.empty(out, dtype=torch.bfloat16, device="cuda"),
                "z_out": torch.empty(out, dtype=torch.float32, device="cuda"),
                "dw": torch.empty((cout, 27, cin), device="cuda"), "db": torch.empty(cout, device="cuda"),
                "scratch": sg.wgrad_scratch(x, cin, cout)}
    if kind == "apply":
        ws, bs, x = _network_inputs(case, seed)
        net = sur.Surrogate(seed=0)
        for k, (w, b) in enumerate(zip(ws, bs)):
            net.w32[k].copy_(w)
            net.b32[k].copy_(b)
        net.adam_step(0.0)  # a step of length zero: rounds the master weights to BF16
        return {"kind": kind, "net": net, "x": x}
    th0 = lb.lb_theta0()
    if kind == "batch":
        n, tau, amp = _batch_members(case, seed)
        b = _Handle(lb.lb_batch_init([(e, e, e) for e in n], tau, case["prec"]), lb.lb_batch_destroy)
        outs = []
        for k, e in enumerate(n):
            f = wl.standing_wave(e, e, e, th0, amplitude=float(amp[k]), device="cuda")
            lb.lb_set_fields(lb.lb_batch_sim(b.h, k), f["rho"], f["u"], f["theta"])
            outs.append(_state_tensor(e, e, e, case["prec"]))
        return {"kind": kind, "batch": b, "steps": case["steps"], "outs": outs}
    nx, ny, nz, prec = case["nx"], case["ny"], case["nz"], case["prec"]
    rho, u, theta = _fields(nx, ny, nz, th0, seed)
    if kind == "snapshot":
        ctx = _Handle(lb.lb_init((nx, ny, nz), TAU, prec), lb.lb_destroy)
        return {"kind": kind, "ctx": ctx, "grid": (nx, ny, nz), "prec": prec, "fields": (rho, u, theta),
                "f": _populations(nx, ny, nz, seed), "rho": torch.empty_like(rho), "u": torch.empty_like(u),
                "theta": torch.empty_like(theta), "raw": _state_tensor(nx, ny, nz, prec),
                "f_out": torch.empty((2, 41, nz, ny, nx), dtype=F64, device="cuda"),
                "sums": torch.empty(5, dtype=F64, device="cuda")}
    if rho.numel() > 1 << 23:
        torch.cuda.empty_cache()  # the library allocates beside torch
    mode = case["mode"]
    flags = {"entropic": lb.LB_FLAG_ENTROPIC, "entropic_path": lb.LB_FLAG_ENTROPIC | lb.LB_FLAG_ENTROPIC_PATH}.get(mode, 0)
    ctx = _Handle(lb.lb_init((nx, ny, nz), case["tau"], prec, flags=flags), lb.lb_destroy)
    lb.lb_set_fields(ctx.h, rho, u, theta)
    if mode == "walls":
        lb.lb_set_walls(ctx.h, *_walls(th0))
    elif mode == "nonideal":
        a, b = lb.lb_nonideal_constants(case["eos"], THETA_STAR)
        lb.lb_set_nonideal(ctx.h, a, b, KAPPA, 0.5, eos=case["eos"])
    elif mode == "stochastic":
        lb.lb_set_stochastic_rounding(ctx.h, SR_SEED)
    lb.lb_sync(ctx.h)
    del rho, u, theta
    if 2 * nx * ny * nz > 1 << 23:
        torch.cuda.empty_cache()
    return {"kind": kind, "ctx": ctx, "steps": case["steps"], "out": _state_tensor(nx, ny, nz, prec)}


def run(state):
    kind = state["kind"]
    if kind == "step":
        ctx = state["ctx"].h
        lb.lb_step(ctx, state["steps"])
        lb.lb_get_state(ctx, state["out"])
        return state["out"]
    if kind == "batch":
        b = state["batch"].h
        lb.lb_batch_step(b, state["steps"], lb.LB_BATCH_GRAPH)
        for k, o in enumerate(state["outs"]):
            lb.lb_get_state(lb.lb_batch_sim(b, k), o)
        return state["outs"]
    if kind == "snapshot":
        ctx = state["ctx"].h
        lb.lb_set_fields(ctx, *state["fields"])
        sums = lb.lb_conserved(ctx)
        lb.lb_get_moments(ctx, state["rho"], state["u"], state["theta"])
        lb.lb_get_populations(ctx, state["f_out"])
        lb.lb_set_populations(ctx, state["f"])
        lb.lb_get_state(ctx, state["raw"])
        lb.lb_conserved_noalloc(state["raw"], state["grid"], state["prec"], state["sums"])
        return [sums, state["rho"], state["u"], state["theta"], state["f_out"], state["raw"], state["sums"]]
    if kind == "apply":
        return state["net"].forward(state["x"])
    s = state
    y = sg.conv3d_fwd(s["x"], s["w"], s["bias"], act=s["act"], res_in=s["res"], z_out=s["z_out"], y=s["y"],
                      xper=s["xper"])
    dz = sg.act_backward(s["dy"], s["z"], s["act"])
    sg.conv3d_wgrad(s["x"], dz, s["dw"], s["db"], s["scratch"], xper=s["xper"])
    wt = sg.transpose_weights(s["w"])
    dx = sg.conv3d_fwd_f32(dz, wt, add=s["dy"] if s["res"] else None, xper=s["xper"])
    return [y, s["z_out"], dz, s["dw"], s["db"], dx]


def work(case):
    kind = case["kind"]
    if kind == "layer":
        vox = case["batch"] * case["nz"] * case["ny"] * 64
        cin, cout = case["cin"], case["cout"]
        # in: x, kept z, dy; out: y, z, dz, dx; weights and their gradient
        values = vox * (2 * cin + 4 * cout + 4 * cout + 2 * cout + 4 * cout + 2 * cout + 4 * cin)
        return {"bytes": values + 27 * cin * cout * 6, "flops": 3 * 2 * vox * 27 * cin * cout}
    if kind == "apply":
        vox = case["batch"] * case["n"] ** 3
        flops = 2 * vox * 27 * (16 * 32 + 4 * 32 * 32 + 32 * 16)
        # what the layers hand on in BF16: each read once and written once
        return {"bytes": vox * 2 * (16 + 2 * 5 * 32 + 16 + 16), "flops": flops}
    if kind == "batch":
        nodes = sum(2 * n ** 3 for n in _batch_members(case, 0)[0])
        b = 82 * BYTES[case["prec"]] * nodes
        return {"bytes": b * (case["steps"] + 1), "flops": FLOPS_PER_NODE * nodes * case["steps"]}
    nodes = 2 * case["nx"] * case["ny"] * case["nz"]
    es = BYTES[case["prec"]]
    if kind == "snapshot":
        # fields in and moments out (40 + 40), populations in and out in FP64, and the stored state:
        # written, read by the sums, the moments and the export, written again, copied, summed
        per = 80 + 2 * 41 * 8 + 8 * 41 * es
        return {"bytes": per * nodes, "flops": 4 * FLOPS_PER_NODE * nodes}
    per = 82 * es
    if case["mode"] == "nonideal":  # the forces need the streamed densities: a second gather
        per += 41 * es
    return {"bytes": nodes * (per * case["steps"] + 82 * es), "flops": FLOPS_PER_NODE * nodes * case["steps"]}


# ---------------------------------------------------------------------------
# 64-bit reference: the model's formulas in torch, on whole arrays in blocks of planes
# ---------------------------------------------------------------------------
def _velocities():
    """Doubled components in the documented population order: rest, then +-c pairs by shell."""
    out = [(0, 0, 0)]
    axes = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
    diag = [(1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
    cube = [(1, 1, 1), (1, 1, -1), (1, -1, 1), (-1, 1, 1)]
    for scale, dirs in ((2, axes), (4, axes), (2, diag), (2, cube), (1, cube)):
        for v in dirs:
            out += [tuple(scale * a for a in v), tuple(-scale * a for a in v)]
    return out


class _Exact:
    """RD3Q41 on an nx x ny x nz grid, float64: f[2][41][nz][ny][nx]."""

    def __init__(self, nx, ny, nz, tau, mode="plain", eos=""):
        self.shape, self.mode, self.eos = (nz, ny, nx), mode, eos
        self.beta = 1.0 / (2.0 * tau + 1.0)
        self.c2 = _velocities()
        c = np.array(self.c2, dtype=np.float64) / 2
        shell_w = {1.0: 0.04743040745116578, 4.0: 0.00165687664501576, 2.0: 0.00651175327832464,
                   3.0: 0.00454087801154440, 0.75: 0.04917980624482672}
        csq = (c * c).sum(1)
        w = np.array([0.0] + [shell_w[v] for v in csq[1:]])
        w[0] = 1.0 - w.sum()
        self.th0 = float((w * c[:, 0] ** 2).sum())

        def t(v):
            return torch.from_numpy(np.ascontiguousarray(v)).cuda().view(-1, 1, 1, 1)

        self.w, self.c, self.csq = t(w), [t(c[:, a]) for a in range(3)], t(csq)
        s = csq / self.th0
        self.p = [t(0.5 * (s - 3)), t((s * s - 10 * s + 15) / 8), t((s ** 3 - 21 * s * s + 105 * s - 105) / 48)]
        planes = max(1, int(1.5e6 / (nx * ny)))
        self.blocks = [(z, min(nz, z + planes)) for z in range(0, nz, planes)]

    def moments(self, f):
        rho = f.sum(0)
        u = [(f * c).sum(0) / rho for c in self.c]
        theta = ((f * self.csq).sum(0) / rho - sum(v * v for v in u)) / 3
        return rho, u, theta

    def series(self, rho, u, theta):
        """The rest equilibrium to third order in eta times the velocity series, with the momentum
        projection."""
        eta = theta / self.th0 - 1
        ft = self.w * rho * (1 + eta * (self.p[0] + eta * (self.p[1] + eta * self.p[2])))
        cx2, cy2 = self.c[0] ** 2, self.c[1] ** 2
        M2 = (ft * (self.csq * cx2)).sum(0) / (5 * rho * theta ** 2) - 1
        M2p = (ft * (cx2 * cy2)).sum(0) / (rho * theta ** 2) - 1
        A1 = 2.5 * M2 / (1 + 2.5 * M2)
        A2 = 5 * A1 * (1 - M2) - (3 + M2p - 5 * M2)
        usq = sum(v * v for v in u)
        g = usq / theta
        a = sum(c * v for c, v in zip(self.c, u)) / theta
        k = g * A1 * self.csq / (6 * theta)
        X = -0.5 * g * (1 - A1) - k + 0.5 * a * a + a * (1 + g * A2 / 6 - k) + a ** 3 / 6
        fe = ft * (1 + X)
        dj = [rho * v - (fe * c).sum(0) for c, v in zip(self.c, u)]
        return fe + ft * sum(c * v for c, v in zip(self.c, dj)) / (rho * theta)

    def entropic(self, rho, u, theta):
        """Minimiser of sum f ln(f / w) at the given moments: f = w rho exp(l . phi), Newton."""
        one = torch.ones_like(rho)
        th0 = self.th0
        usq = sum(v * v for v in u)
        t4 = usq + 3 * (theta - th0)
        tgt = torch.stack([0 * one, *u, t4], -1)
        lam = torch.stack([0 * one, *[v / th0 for v in u], t4 / (6 * th0 * th0)], -1)
        phi = torch.stack([torch.ones_like(self.csq), *self.c, self.csq - 3 * th0], -1).view(41, 5)
        w = self.w.view(41)
        pp = (phi[:, :, None] * phi[:, None, :]).reshape(41, 25)
        for _ in range(7):
            em = torch.expm1(lam @ phi.T)
            F = (em * w) @ phi - tgt
            J = (((em + 1) * w) @ pp).view(*rho.shape, 5, 5)
            lam = lam - torch.linalg.solve(J, F)
        return (rho[..., None] * w * torch.exp(lam @ phi.T)).movedim(-1, 0)

    def path_length(self, f, fe):
        """alpha with H(f + alpha (fe - f)) = H(f), H = sum f ln(f / w): bisection below the value
        at which a population reaches zero."""
        x = fe / f - 1
        lx = torch.log1p(x)

        def phi(y):
            small = y.abs() < 0.05
            ys = torch.where(small, y, torch.zeros_like(y))
            s = sum((-ys) ** (n - 2) / (n * (n - 1)) for n in range(2, 16)) * ys * ys
            return torch.where(small, s, (1 + y) * torch.log1p(y) - y)

        def dh(a):
            return (f * (phi(a * x) - a * x * lx)).sum(0)

        neg = (-x).amax(0)
        lim = torch.where(neg > 0, 1 / neg.clamp_min(1e-300), torch.full_like(neg, 1e300))
        lo, hi = torch.minimum(torch.ones_like(lim), 0.5 * lim), torch.minimum(3.0 * torch.ones_like(lim), lim * (1 - 1e-14))
        none = ~(dh(hi) > 0) | (x.abs().amax(0) <= 1e-9)
        for _ in range(52):
            mid = 0.5 * (lo + hi)
            up = dh(mid) > 0
            lo, hi = torch.where(up, lo, mid), torch.where(up, mid, hi)
        return torch.where(none, torch.full_like(lo, 2.0), 0.5 * (lo + hi))

    def equilibrium(self, rho, u, theta):
        return (self.entropic if self.mode.startswith("entropic") else self.series)(rho, u, theta)

    def init(self, rho, u, theta):
        nz, ny, nx = self.shape
        f = torch.empty((2, 41, nz, ny, nx), dtype=F64, device="cuda")
        for s in (0, 1):
            for a, b in self.blocks:
                f[s, :, a:b] = self.equilibrium(rho[s, a:b], [v[s, a:b] for v in u], theta[s, a:b])
        return f

    def pull(self, f, s, a, b):
        """f_i(x - c_i) of the planes [a, b) of sub-lattice s."""
        nz = self.shape[0]
        out = torch.empty((41, b - a) + self.shape[1:], dtype=F64, device="cuda")
        zz = torch.arange(a, b, device="cuda")
        for i, c in enumerate(self.c2):
            half = c[0] % 2
            dx, dy, dz = ((1 if v > 0 else 0) - s if half else v // 2 for v in c)
            src = f[1 - s if half else s, i].index_select(0, (zz - dz) % nz)
            out[i] = torch.roll(src, (dy, dx), (1, 2))
        return out

    def set_walls(self, walls):
        one = torch.ones((1, 1, 1), dtype=F64, device="cuda")
        self.wall_e = [self.series(one, [one * w[0], one * w[1], one * 0], one * w[2]).view(41) for w in walls]

    def wall_density(self, f):
        """rho_w[side][ny][nx]: each column's absorbed over its unit emission."""
        nz = self.shape[0]
        rho = []
        for side in (0, 1):
            acc = torch.zeros(self.shape[1:], dtype=F64, device="cuda")
            emit = 0.0
            for i, c in enumerate(self.c2):
                out, into = (c[2], -c[2]) if side else (-c[2], c[2])
                emit = emit + max(0, into) * self.wall_e[side][i]
                for j in range(max(0, out)):
                    z2 = 2 * nz - out + j if side else j
                    s = z2 % 2
                    acc += torch.roll(f[s, i, z2 // 2], ((s + c[1] + side) // 2, (s + c[0] + side) // 2), (0, 1))
            rho.append(acc / emit)
        return rho

    def wall_emission(self, v, s, a, rho_w):
        nz = self.shape[0]
        for i, c in enumerate(self.c2):
            for k in range(v.shape[1]):
                up = 2 * (a + k) + s - c[2]
                if 0 <= up < 2 * nz:
                    continue
                side = 0 if up < 0 else 1
                shift = (-((s - c[1] + side) // 2), -((s - c[0] + side) // 2))
                v[i, k] = self.wall_e[side][i] * torch.roll(rho_w[side], shift, (0, 1))

    def set_fluid(self, a, b):
        self.a, self.b = a, b

    def fluid(self, r):
        """mu and F of the nonideal fluid (ideal part removed)."""
        th, a, b = self.th0, self.a, self.b
        if self.eos == "vdw":
            L = torch.log1p(-b * r)
            return -th * L + th * b * r / (1 - b * r) - 2 * a * r, -th * r * L - a * r * r
        p = b * r / 4
        e = (4 * p - 3 * p * p) / (1 - p) ** 2
        de = p * (4 - 2 * p) / (1 - p) ** 3
        if self.eos == "carnahan_starling":
            return th * (e + de) - 2 * a * r, th * r * e - a * r * r
        q = math.sqrt(2.0)
        L = (torch.log1p((q + 1) * b * r) - torch.log1p(-(q - 1) * b * r)) / (2 * q * b)
        return th * (e + de) - a * L - a * r / (1 + 2 * b * r - (b * r) ** 2), th * r * e - a * r * L

    def neighbours(self, X):
        """(c, w, X(x + c)) over the 14 moving velocities of the bcc derivative stencil."""
        for ax in range(3):
            for sgn in (1, -1):
                c = [0.0, 0.0, 0.0]
                c[ax] = float(sgn)
                yield c, 1 / 36, torch.roll(X, -sgn, 3 - ax)
        for signs in itertools.product((1, -1), repeat=3):
            Y = torch.empty_like(X)
            for s in (0, 1):
                off = [-(s if g > 0 else s - 1) for g in reversed(signs)]
                Y[s] = torch.roll(X[1 - s], off, (0, 1, 2))
            yield [0.5 * g for g in signs], 2 / 36, Y

    def grad(self, X):
        g = [0, 0, 0]
        for c, w, Y in self.neighbours(X):
            for a in range(3):
                if c[a]:
                    g[a] = g[a] + 6 * w * c[a] * Y
        return g

    def lap(self, X):
        return sum(12 * w * (Y - X) for _, w, Y in self.neighbours(X))

    def force(self, rho):
        """g of the momentum-conserving formulation, eta = 1/2."""
        mu, F = self.fluid(rho)
        gr = self.grad(rho)
        iso = -0.5 * sum(v * v for v in gr) - rho * self.lap(rho)
        gmu, gF, glF = self.grad(mu), self.grad(F), self.grad(self.lap(F))
        out = []
        for a in range(3):
            div = sum(self.grad(gr[a] * gr[b])[b] for b in range(3)) + self.grad(iso)[a]
            g4 = gF[a] - glF[a] / 12
            out.append(-(rho * gmu[a] + mu * gr[a] - 0.5 * gF[a] - 0.5 * g4 + KAPPA * div) / rho)
        return out

    def step(self, f, out):
        if self.mode == "walls":
            rho_w = self.wall_density(f)
        if self.mode == "nonideal":
            rho = torch.stack([torch.cat([self.pull(f, s, a, b).sum(0) for a, b in self.blocks]) for s in (0, 1)])
            force = self.force(rho)
        for s in (0, 1):
            for a, b in self.blocks:
                v = self.pull(f, s, a, b)
                if self.mode == "walls":
                    self.wall_emission(v, s, a, rho_w)
                rho, u, theta = self.moments(v)
                if self.mode == "nonideal":
                    g = [x[s, a:b] for x in force]
                    u = [x + 0.5 * y for x, y in zip(u, g)]
                    fe = self.series(rho, u, torch.full_like(rho, self.th0))
                    Fi = fe * sum(y * (c - x) for x, y, c in zip(u, g, self.c)) / self.th0
                    out[s, :, a:b] = v + 2 * self.beta * (fe - v) + (1 - self.beta) * Fi
                    continue
                fe = self.equilibrium(rho, u, theta)
                k = 2.0 if self.mode != "entropic_path" else self.path_length(v, fe)
                out[s, :, a:b] = v + k * self.beta * (fe - v)
        return out

    def stored(self, f, prec):
        """The storage's number of f, in place: f itself or (f / w - 1) times the scale."""
        if prec == "f64":
            return f
        for s in (0, 1):
            f[s].div_(self.w).sub_(1).mul_(SCALE[prec])
        return f

    def totals(self, f):
        tot = []
        for wgt in (torch.ones_like(self.w), *self.c, 0.5 * self.csq):
            tot.append(sum((f[s, :, a:b] * wgt).sum() for s in (0, 1) for a, b in self.blocks))
        return torch.stack(tot)


def _populations(nx, ny, nz, seed):
    """Populations near rest, off equilibrium: w_i (1 + smooth + noise)."""
    c = np.array(_velocities(), dtype=np.float64) / 2
    e = _Exact(1, 1, 1, 1.0)
    g = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.empty((2, 41, nz, ny, nx), dtype=F64, device="cuda")
    X = wl.node_positions(nx, ny, nz, "cuda")[0]
    for i in range(41):
        wave = 5e-3 * torch.sin(2 * math.pi * X / nx + float(c[i, 0]))
        noise = 2e-3 * (2 * torch.rand((2, nz, ny, nx), generator=g, device="cuda", dtype=F64) - 1)
        f[:, i] = float(e.w[i]) * (1 + wave + noise)
    return f


def _conv(x, w, bias, xper):
    """Periodic 3x3x3 convolution of a d-layout volume: segments of xper voxels along x."""
    B, nz, ny, nx, ci = x.shape
    v = x.reshape(B, nz, ny, nx // xper, xper, ci)
    out = torch.zeros(v.shape[:-1] + (w.shape[0],), dtype=F64, device=x.device)
    for tap in range(27):
        dz, dy, dx = tap // 9 - 1, (tap // 3) % 3 - 1, tap % 3 - 1
        out += torch.roll(v, (-dz, -dy, -dx), (1, 2, 4)) @ w[:, tap].T
    return out.reshape(B, nz, ny, nx, -1) + (0 if bias is None else bias)


def _gelu(z):
    return 0.5 * z * (1 + torch.erf(z / math.sqrt(2.0)))


def exact(case, seed):
    kind = case["kind"]
    if kind == "layer":
        x, w, bias, z, dy = (t.to(F64) for t in _layer_inputs(case, seed))
        xper, cin, cout = 64 // case["dilation"], case["cin"], case["cout"]
        gelu = cout == 32
        pre = _conv(x, w, bias, xper)
        y = (_gelu(pre) if gelu else pre) + (x if cin == cout else 0)
        pdf = torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi)
        dz = dy * (0.5 * (1 + torch.erf(z / math.sqrt(2.0))) + z * pdf) if gelu else dy
        B, nz, ny, nx, _ = x.shape
        v = x.reshape(B, nz, ny, nx // xper, xper, cin)
        dw = torch.empty((cout, 27, cin), dtype=F64, device="cuda")
        for tap in range(27):
            s = torch.roll(v, (1 - tap // 9, 1 - (tap // 3) % 3, 1 - tap % 3), (1, 2, 4))
            dw[:, tap] = dz.reshape(-1, cout).T @ s.reshape(-1, cin)
        wt = w.flip(1).permute(2, 1, 0).contiguous()
        dx = _conv(dz, wt, None, xper) + (dy if cin == cout else 0)
        return [y, pre, dz, dw, dz.reshape(-1, cout).sum(0), dx]
    if kind == "apply":
        ws, bs, x = _network_inputs(case, seed)
        h = x = x.to(F64)
        for k, (w, b, d) in enumerate(zip(ws, bs, (1, 2, 4, 8, 8, 8))):
            w, b = w.to(torch.bfloat16).to(F64), b.to(F64)
            z = torch.zeros(h.shape[:-1] + (w.shape[0],), dtype=F64, device="cuda")
            for tap in range(27):
                sh = (-d * (tap // 9 - 1), -d * ((tap // 3) % 3 - 1), -d * (tap % 3 - 1))
                z += torch.roll(h, sh, (1, 2, 3)) @ w[:, tap].T
            z += b
            h = (x + z) if k == 5 else _gelu(z) + (h if k else 0)
        return h
    th0 = 0.2948964908710634
    if kind == "batch":
        n, tau, amp = _batch_members(case, seed)
        outs = []
        for e, t, A in zip(n, tau, amp):
            m = _Exact(e, e, e, t)
            fl = wl.standing_wave(e, e, e, th0, amplitude=float(A), device="cuda")
            f = m.init(fl["rho"], fl["u"], fl["theta"])
            g = torch.empty_like(f)
            for _ in range(case["steps"]):
                f, g = m.step(f, g), f
            outs.append(m.stored(f, case["prec"]))
        return outs
    nx, ny, nz, prec = case["nx"], case["ny"], case["nz"], case["prec"]
    if kind == "snapshot":
        m = _Exact(nx, ny, nz, 1.0)
        rho, u, theta = _fields(nx, ny, nz, th0, seed)
        f = m.init(rho, u, theta)
        g = _populations(nx, ny, nz, seed)
        sums = m.totals(g)
        return [m.totals(f), rho, u, theta, f, m.stored(g, prec), sums]
    m = _Exact(nx, ny, nz, case["tau"], case["mode"], case["eos"])
    f = m.init(*_fields(nx, ny, nz, th0, seed))
    torch.cuda.empty_cache()
    if case["mode"] == "walls":
        m.set_walls(_walls(th0))
    elif case["mode"] == "nonideal":
        # constants at the critical point theta_c = theta_0 / 1.1, rho_c = 1
        m.set_fluid(*_fluid_constants(case["eos"], th0 / THETA_STAR))
    g = torch.empty_like(f)
    for _ in range(case["steps"]):
        f, g = m.step(f, g), f
    del g
    return m.stored(f, prec)


def _fluid_constants(eos, theta_c):
    if eos == "vdw":
        return 27 / 3 * theta_c / 8, 1 / 3
    if eos == "peng_robinson":
        return 1.851427622 * theta_c, 0.353748714
    lo, hi = 0.01, 0.5  # Carnahan-Starling: critical packing fraction by bisection

    def h(p):
        return (1 + 4 * p + 4 * p ** 2 - 4 * p ** 3 + p ** 4) * (1 - p) - p * (8 + 20 * p - 4 * p ** 2)

    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if h(mid) > 0 else (lo, mid)
    p = 0.5 * (lo + hi)
    return 0.5 * (1 + 4 * p + 4 * p ** 2 - 4 * p ** 3 + p ** 4) / (1 - p) ** 4 * theta_c, 4 * p
