"""The work that is measured: what users of this library have it do, through its public entry points.

Three kinds of case:
  cavity   one lid-driven cavity (``Cavity``): the field is set, some steps are taken, and what a
           program reads back is read back (moments, the Eq. 6 residual, probe series, stream function)
  batch    a Re x Ar sweep (``lbm_batch_*``): all cavities advance together, then every cavity's
           moments and residual are read
  predict  the learned warm start: network forward, smoothing, fine fields
  train    one optimiser step of that network: several backward passes and Adam

Fields leave the library in FP64 whatever the storage; ``run`` hands them on in the type that the
case computes in (FP64, FP32, binary16, bfloat16), which is what its accuracy can be held to.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2211_05009_gb300 import Cavity
from paper_2211_05009_gb300 import binding as B

RESULT = {"f64": torch.float64, "f32": torch.float32, "f32s": torch.float32, "f16s": torch.float16,
          "bf16s": torch.bfloat16, "q16s": torch.float16}
BYTES = {"f64": 8, "f32": 4, "f32s": 4, "f16s": 2, "bf16s": 2, "q16s": 2}
FLOPS = 100  # arithmetic operations of one lattice update (moments, equilibrium, relaxation)
MODES = 5


def listed():
    return [
        # the paper's validation cavity at Re 100: FP64, small, the launches count
        dict(name="f64_128x128", kind="cavity", nx=128, ny=128, Re=100.0, U=0.1, dtype="f64", steps=100, every=0,
             psi=True, tune=False),
        # a program that looks at the field every few steps; odd sizes, no whole checkpoint interval
        dict(name="f32_133x77", kind="cavity", nx=133, ny=77, Re=400.0, U=0.1, dtype="f32", steps=37, every=0,
             psi=False, tune=False),
        # the paper's survey width with its observing point; fits the L2 cache
        dict(name="f32s_500x500", kind="cavity", nx=500, ny=500, Re=4000.0, U=0.1, dtype="f32s", steps=100, every=2,
             psi=False, tune=False),
        # the paper's deep cavity on unshifted FP32, two and a half checkpoint intervals
        dict(name="f32_500x1000", kind="cavity", nx=500, ny=1000, Re=8000.0, U=0.1, dtype="f32", steps=250, every=100,
             psi=True, tune=False),
        # the same cavity as an FP64 reference run
        dict(name="f64_500x1000", kind="cavity", nx=500, ny=1000, Re=6000.0, U=0.1, dtype="f64", steps=100, every=0,
             psi=False, tune=False),
        # the benchmark's cavity: Re 8000 at 2048 x 2048, tuned, probe and stream function
        dict(name="f32s_2048x2048", kind="cavity", nx=2048, ny=2048, Re=8000.0, U=0.05, dtype="f32s", steps=100,
             every=2, psi=True, tune=True),
        # 16-bit storage at the size it is meant for
        dict(name="f16s_4096x4096", kind="cavity", nx=4096, ny=4096, Re=8000.0, U=0.05, dtype="f16s", steps=100,
             every=0, psi=False, tune=True),
        # the 16-bit format that holds 1e-3 U, on the cavity of the precision study
        dict(name="q16s_2048x2048", kind="cavity", nx=2048, ny=2048, Re=8000.0, U=0.05, dtype="q16s", steps=100,
             every=0, psi=False, tune=False),
        # the survey of Sec. 3.3: 45 cavities 500 wide, Ar 0.4..2.0, Re 4000..8000
        dict(name="batch_f32s_45x500", kind="batch", nx=500, count=45, dtype="f32s", U=0.1, re_lo=4000.0, re_hi=8000.0,
             steps=200, pick=0),
        # targets of the warm-start network: 48 FP64 cavities 128 wide
        dict(name="batch_f64_48x128", kind="batch", nx=128, count=48, dtype="f64", U=0.1, re_lo=100.0, re_hi=1000.0,
             steps=200, pick=1),
        # a warm start predicted for one fine cavity
        dict(name="predict_256x256", kind="predict", nx=256, ny=250, width=20, Re=700.0, smooth=4),
        # one optimiser step over a mini-batch of 128-wide samples of uneven heights
        dict(name="train_128_x8", kind="train", nx=128, count=8, width=20, lr=1e-3, pick=2),
    ]


def draw(rng):
    """One more case of the same ranges."""
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    kind = rng.choice(["cavity"] * 5 + ["batch"] * 2 + ["predict", "train"])
    if kind == "cavity":
        dtype = rng.choice(["f64", "f32", "f32s", "f16s", "bf16s", "q16s"])
        nx = int(log(40, 3000 if BYTES[dtype] < 8 else 1200))
        ny = max(16, round(nx * rng.uniform(0.4, 1.8 if nx < 1500 else 1.1)))
        U = rng.choice([0.05, 0.1])
        re = log(max(100.0, 3.0 * U * nx), max(200.0, min(8000.0, 16.0 * nx)))
        return dict(kind=kind, nx=nx, ny=ny, Re=round(re, 1), U=U, dtype=dtype, steps=int(log(20, 320)),
                    every=rng.choice([0, 2, 5, 100]), psi=rng.random() < 0.4, tune=rng.random() < 0.3)
    if kind == "batch":
        nx = int(log(64, 500))
        return dict(kind=kind, nx=nx, count=rng.randint(4, 45), dtype=rng.choice(["f64", "f32s", "f32s", "f16s"]) if nx < 300 else "f32s",
                    U=0.1, re_lo=100.0, re_hi=float(min(8000, 8 * nx)), steps=rng.choice([100, 150, 200]), pick=rng.randint(3, 10**6))
    if kind == "predict":
        nx = rng.choice([128, 256, 384, 512])
        return dict(kind=kind, nx=nx, ny=int(nx * rng.uniform(0.4, 1.4)), width=rng.choice([8, 12, 16, 20, 24]),
                    Re=round(log(100, 4000), 1), smooth=rng.randint(0, 5))
    return dict(kind=kind, nx=rng.choice([128, 256]), count=rng.randint(2, 8), width=rng.choice([8, 12, 16, 20]), lr=1e-3,
                pick=rng.randint(3, 10**6))


# ------------------------------------------------------------------ inputs
def field(nx, ny, U, seed):
    """(rho, ux, uy) of a cavity flow in motion: a few no-slip vortices, a pressure field, the lid."""
    r = np.random.RandomState(seed % (1 << 31))
    x = torch.linspace(0, 1, nx, dtype=torch.float64, device="cuda")
    y = torch.linspace(0, 1, ny, dtype=torch.float64, device="cuda")
    h = ny / nx
    rho = torch.ones((ny, nx), dtype=torch.float64, device="cuda")
    ux, uy = torch.zeros_like(rho), torch.zeros_like(rho)
    pi = math.pi
    for _ in range(MODES):
        m, n = r.randint(1, 5, 2)
        a = r.uniform(-1, 1) * 0.25 * U / (pi * (m + n))
        # psi = a sin(pi x) sin(m pi x) sin(pi y) sin(n pi y): zero with its slope on every wall
        sx, sy = torch.sin(pi * x) * torch.sin(m * pi * x), torch.sin(pi * y) * torch.sin(n * pi * y)
        dx = pi * torch.cos(pi * x) * torch.sin(m * pi * x) + m * pi * torch.sin(pi * x) * torch.cos(m * pi * x)
        dy = pi * torch.cos(pi * y) * torch.sin(n * pi * y) + n * pi * torch.sin(pi * y) * torch.cos(n * pi * y)
        ux += a * dy[:, None] / h * sx[None, :]
        uy -= a * sy[:, None] * dx[None, :]
        m, n = r.randint(1, 4, 2)
        rho += r.uniform(-1, 1) * 0.1 * U * U * torch.cos(n * pi * y)[:, None] * torch.cos(m * pi * x)[None, :]
    ux[-1, 1:-1] = U
    return rho, ux, uy


def sweep(case):
    """(nx, ny, Re) of every cavity of a batch."""
    n, nx = case["count"], case["nx"]
    if case["pick"] == 0:  # the survey's grid
        ars = [0.4 + 0.2 * i for i in range(9)]
        res = [case["re_lo"] + (case["re_hi"] - case["re_lo"]) * i / 4 for i in range(5)]
        return [(nx, round(nx * ar), re) for re in res for ar in ars][:n]
    r = np.random.RandomState(case["pick"])
    return [(nx, max(3, round(nx * r.uniform(0.4, 2.0))), float(r.uniform(case["re_lo"], case["re_hi"]))) for _ in range(n)]


def heights(case):
    """Valid rows of every sample of a training step."""
    r = np.random.RandomState(case["pick"])
    return [max(16, round(case["nx"] * r.uniform(0.4, 1.9))) for _ in range(case["count"])]


def pad16(n):
    return (n + 15) // 16 * 16


def channels(width):
    ch = [width * k for k in (1, 2, 4, 8, 8)]
    io, prev = [], 7
    for c in ch:
        io += [(prev, c), (c, c)]
        prev = c
    for lv in (3, 2, 1, 0):
        io += [(ch[lv + 1] + ch[lv], ch[lv]), (ch[lv], ch[lv])]
    return io + [(ch[0], 3)]


def parameters(width, seed):
    """Network parameters as a trained file holds them: He-scaled weights, small biases."""
    r = np.random.RandomState(seed % (1 << 31))
    out = []
    for k, (ci, co) in enumerate(channels(width)):
        out += [r.uniform(-1, 1, ci * co * 9) * math.sqrt(6.0 / (9 * ci)), r.uniform(-0.05, 0.05, co)]
    return np.concatenate(out).astype(np.float32)


def sample(nx, ny, Re, seed):
    """Network input [7][H][nx] and target [3][H][nx] of one cavity, laid out as the library's own."""
    U, H = 0.1, pad16(ny)
    rho, ux, uy = field(nx, ny, U, seed)
    t_rho, t_ux, t_uy = field(nx, ny, U, seed + 7919)
    inp = torch.zeros((7, H, nx), dtype=torch.float32, device="cuda")
    tgt = torch.zeros((3, H, nx), dtype=torch.float32, device="cuda")
    scale = B.LBM_WARM_RHO_SCALE
    for k, (a, b) in enumerate((((rho - 1) * scale, (t_rho - 1) * scale), (ux / U, t_ux / U), (uy / U, t_uy / U))):
        inp[k, :ny] = a
        tgt[k, :ny] = 0.5 * (a + b)
    inp[3, :ny], inp[4, :ny], inp[6, :ny] = Re / 4000.0, ny / nx / 2.0, 1.0
    inp[5, 0], inp[5, ny - 1], inp[5, :ny, 0], inp[5, :ny, -1] = 1.0, 1.0, 1.0, 1.0
    return inp, tgt


class Held:
    """A library handle given back when the state goes."""

    def __init__(self, handle, release):
        self.handle, self._release = handle, release

    def __del__(self):
        if self.handle:
            self._release(self.handle)
            self.handle = None


# ------------------------------------------------------------------ what a program has in hand
def prepare(case, seed):
    kind = case["kind"]
    if kind == "cavity":
        cav = Cavity(case["nx"], case["ny"], Re=case["Re"], U=case["U"], dtype=case["dtype"])
        if case["tune"]:
            B.lbm_autotune(cav.ctx, 20)
        s = {"cav": cav, "start": field(case["nx"], case["ny"], case["U"], seed)}
        if case["every"]:
            n = max(1, case["steps"] // case["every"])
            s["series"] = cav.probe(0.5, 0.3 * case["ny"] / case["nx"], every=case["every"], cap=n)[1]
    elif kind == "batch":
        cases = sweep(case)
        b = B.lbm_batch_create([c[0] for c in cases], [c[1] for c in cases], [c[2] for c in cases],
                               [case["U"]] * len(cases), case["dtype"])
        s = {"b": Held(b, B.lbm_batch_destroy), "cases": cases}
        B.lbm_batch_set_stream(b, torch.cuda.current_stream().cuda_stream)
        for i, (nx, ny, _) in enumerate(cases):
            B.lbm_batch_set_moments(b, i, *field(nx, ny, case["U"], seed + i))
        B.lbm_batch_autotune(b, 20)
        s["out"] = torch.zeros((3, sum(c[0] * c[1] for c in cases)), dtype=torch.float64, device="cuda")
    else:
        net = B.lbm_net_create(case["width"], 0)
        s = {"net": Held(net, B.lbm_net_destroy)}
        B.lbm_net_set_stream(net, torch.cuda.current_stream().cuda_stream)
        B.lbm_net_set_params(net, parameters(case["width"], seed))
        if kind == "predict":
            s["inp"] = sample(case["nx"], case["ny"], case["Re"], seed)[0]
        else:
            s["samples"] = [sample(case["nx"], ny, 500.0, seed + i) for i, ny in enumerate(heights(case))]
            s["n"] = B.lbm_net_param_count(net)
    s["case"] = case
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    return {"cavity": run_cavity, "batch": run_batch, "predict": run_predict, "train": run_train}[s["case"]["kind"]](s)


def run_cavity(s):
    case, cav = s["case"], s["cav"]
    t = RESULT[case["dtype"]]
    cav.set_moments(*s["start"])
    cav.step(case["steps"])
    rho, ux, uy = cav.moments()
    out = {"rho": rho.to(t), "ux": ux.to(t), "uy": uy.to(t)}
    if case["steps"] >= 100:
        out["residual"] = torch.tensor(cav.residual(), dtype=t)
    if case["psi"]:
        psi_min, _, _, psi = cav.stream_function(psi=True)
        out["psi"], out["psi_min"] = psi.to(t), torch.tensor(psi_min, dtype=t)
    if case["every"] and case["steps"] >= case["every"]:
        out["series"] = s["series"].to(t)
    return out


def run_batch(s):
    case, b = s["case"], s["b"].handle
    t = RESULT[case["dtype"]]
    B.lbm_batch_step(b, case["steps"])
    residual, _ = B.lbm_batch_residual(b, len(s["cases"]))
    at = 0
    for i, (nx, ny, _) in enumerate(s["cases"]):
        B.lbm_batch_moments(b, i, *(o[at:at + nx * ny] for o in s["out"]))
        at += nx * ny
    return {"rho": s["out"][0].to(t), "u": s["out"][1:].to(t), "residual": torch.from_numpy(residual).to(t)}


def run_predict(s):
    case, inp, st = s["case"], s["inp"], torch.cuda.current_stream().cuda_stream
    nx, ny, H = case["nx"], case["ny"], inp.shape[1]
    out = torch.empty((3, H, nx), dtype=torch.float32, device="cuda")
    B.lbm_net_forward(s["net"].handle, inp, H, nx, out)
    raw = out.to(torch.bfloat16)  # BF16 operands: the prediction holds no more than that
    if case["smooth"]:
        B.lbm_warm_smooth(out, ny, H, nx, case["smooth"], torch.empty_like(out), st)
    f = [torch.empty((ny, nx), dtype=torch.float64, device="cuda") for _ in range(3)]
    B.lbm_warm_output(inp, out, nx, ny, H, 0.1, *f, st)
    return {"correction": raw, "p": (f[0] - 1.0).to(torch.bfloat16), "ux": f[1].to(torch.bfloat16), "uy": f[2].to(torch.bfloat16)}


def run_train(s):
    case, net = s["case"], s["net"].handle
    B.lbm_net_zero_grads(net)
    losses = [B.lbm_net_backward(net, inp, inp[:3], tgt, inp[6], inp.shape[1], case["nx"]) for inp, tgt in s["samples"]]
    grads, params = (torch.empty(s["n"], dtype=torch.float32, device="cuda") for _ in range(2))
    B.lbm_net_get_grads(net, grads)
    B.lbm_net_adam_step(net, case["lr"], grad_scale=1.0 / len(losses))
    B.lbm_net_get_params(net, params)
    return {"loss": torch.tensor(losses, dtype=torch.bfloat16), "grads": grads.to(torch.bfloat16), "params": params.to(torch.bfloat16)}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    if case["kind"] in ("cavity", "batch"):
        nodes = case["nx"] * case["ny"] if case["kind"] == "cavity" else sum(c[0] * c[1] for c in sweep(case))
        # the start or the old state in, the new state kept, moments out in the result type
        moved = nodes * (3 * 8 * (case["kind"] == "cavity") + 18 * BYTES[case["dtype"]] + 3 * BYTES[case["dtype"]])
        return {"bytes": float(moved), "flops": float(FLOPS) * nodes * case["steps"]}
    lv = [0, 0, 1, 1, 2, 2, 3, 3, 4, 4, 3, 3, 2, 2, 1, 1, 0, 0, 0]
    io = channels(case["width"])
    mac = sum(ci * co * 9 / 4 ** k for (ci, co), k in zip(io, lv))
    par = sum(ci * co * 9 + co for ci, co in io)
    if case["kind"] == "predict":
        px = case["nx"] * pad16(case["ny"])
        return {"bytes": float(4 * par + px * (7 * 4 + 3 * 2) + case["nx"] * case["ny"] * 3 * 2), "flops": 2.0 * mac * px}
    px = sum(case["nx"] * pad16(ny) for ny in heights(case))
    return {"bytes": float(7 * 4 * par + px * 10 * 4), "flops": 6.0 * mac * px}


# ------------------------------------------------------------------ the same in 64 bits
C = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
WEIGHT = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


def equilibrium(rho, ux, uy):
    sq = 1.5 * (ux * ux + uy * uy)
    out = []
    for (cx, cy), w in zip(C, WEIGHT):
        cu = cx * ux + cy * uy
        out.append(w * rho * (1 + 3 * cu + 4.5 * cu * cu - sq))
    return torch.stack(out)


def advance(start, tau, U, steps, point=None, every=0):
    """Fields after `steps` steps, the last Eq. 6 residual and the samples at `point`."""
    rho, ux, uy = start
    f = equilibrium(rho, ux, uy)
    last, residual, series = (ux, uy), None, []
    for t in range(1, steps + 1):
        # populations streamed to the inner nodes, their moments and non-equilibrium part
        ny, nx = f.shape[1:]
        g = torch.stack([f[j, 1 - cy:ny - 1 - cy, 1 - cx:nx - 1 - cx] for j, (cx, cy) in enumerate(C)])
        r = g.sum(0)
        vx = (g[1] - g[3] + g[5] - g[6] - g[7] + g[8]) / r
        vy = (g[2] - g[4] + g[5] + g[6] - g[7] - g[8]) / r
        neq = g - equilibrium(r, vx, vy)
        # walls: density and non-equilibrium part of the inner neighbour, the wall's own velocity
        rho = F.pad(r[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
        neq = F.pad(neq[None], (1, 1, 1, 1), mode="replicate")[0]
        ux, uy = F.pad(vx, (1, 1, 1, 1)), F.pad(vy, (1, 1, 1, 1))
        ux[-1, 1:-1] = U
        f = equilibrium(rho, ux, uy) + (1 - 1 / tau) * neq
        if t % 100 == 0:
            num = ((ux - last[0]) ** 2 + (uy - last[1]) ** 2).sum()
            residual, last = torch.sqrt(num / (last[0] ** 2 + last[1] ** 2).sum()), (ux, uy)
        if every and t % every == 0:
            series.append(torch.stack([ux[point], uy[point]]))
    return rho, ux, uy, residual, series


def network(p, inp, width):
    at, k = 0, 0
    io = channels(width)

    def conv(x):
        nonlocal at, k
        ci, co = io[k]
        w = p[at:at + ci * co * 9].view(co, ci, 3, 3)
        b = p[at + ci * co * 9:at + ci * co * 9 + co]
        at, k = at + ci * co * 9 + co, k + 1
        y = F.conv2d(x, w, b, padding=1)
        return y if k == len(io) else F.leaky_relu(y, 0.1)

    x, skips = inp[None], []
    for lv in range(5):
        x = conv(conv(F.avg_pool2d(x, 2) if lv else x))
        skips.append(x)
    for lv in (3, 2, 1, 0):
        x = conv(conv(torch.cat([F.interpolate(x, scale_factor=2, mode="nearest"), skips[lv]], 1)))
    return conv(x)[0]


def exact(case, seed):
    kind = case["kind"]
    if kind == "cavity":
        nx, ny, U = case["nx"], case["ny"], case["U"]
        point = (min(ny - 1, int(math.floor(0.3 * ny / nx * nx + 0.5))), min(nx - 1, int(math.floor(0.5 * nx + 0.5))))
        rho, ux, uy, residual, series = advance(field(nx, ny, U, seed), 3 * U * nx / case["Re"] + 0.5, U, case["steps"],
                                                point, case["every"])
        out = {"rho": rho, "ux": ux, "uy": uy}
        if residual is not None:
            out["residual"] = residual
        if case["psi"]:
            psi = torch.cumsum(ux, 0) - 0.5 * ux[:1] - 0.5 * ux
            out["psi"], out["psi_min"] = psi, psi.min()
        if series:
            out["series"] = torch.stack(series)
        return out
    if kind == "batch":
        got = [advance(field(nx, ny, case["U"], seed + i), 3 * case["U"] * nx / re + 0.5, case["U"], case["steps"])
               for i, (nx, ny, re) in enumerate(sweep(case))]
        flat = [torch.cat([g[k].reshape(-1) for g in got]) for k in range(3)]
        return {"rho": flat[0], "u": torch.stack(flat[1:]), "residual": torch.stack([g[3] for g in got])}
    p = torch.from_numpy(parameters(case["width"], seed)).to("cuda", torch.float64)
    if kind == "predict":
        nx, ny = case["nx"], case["ny"]
        inp = sample(nx, ny, case["Re"], seed)[0].double()
        raw = network(p, inp, case["width"])
        out = raw[:, :ny]
        for _ in range(case["smooth"]):
            out = F.avg_pool2d(F.pad(out[None], (1, 1, 1, 1), mode="replicate"), 3, stride=1)[0]
        f = inp[:3, :ny] + out
        return {"correction": raw, "p": f[0] / B.LBM_WARM_RHO_SCALE, "ux": f[1] * 0.1, "uy": f[2] * 0.1}
    p.requires_grad_(True)
    losses = []
    for i, ny in enumerate(heights(case)):
        inp, tgt = (t.double() for t in sample(case["nx"], ny, 500.0, seed + i))
        e = (inp[:3] + network(p, inp, case["width"]) - tgt) * inp[6]
        n = inp[6].sum()
        mean = torch.zeros(3, 1, 1, dtype=torch.float64, device="cuda")
        mean[0] = (e[0].sum() / n).detach()
        losses.append((((e - mean) * inp[6]) ** 2).sum() / (3 * n))
        losses[-1].backward()
    g = p.grad / len(losses)
    m, v = 0.1 * g, 0.001 * g * g
    new = p.detach() - case["lr"] * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8)
    return {"loss": torch.stack([x.detach() for x in losses]), "grads": p.grad, "params": new}
