"""Performance cases: the work a program using this package has it do.

Every case goes through the public Python entry points (`lb`, `unet`) and
returns what such a program reads back.  Kinds of work:

* ``lattice``: a periodic lattice advanced by the fused thermal step, then its
  moments.  64^2 and 512^2 droplets and the 4096^2 quench are the sizes of the
  package's own workloads; the ragged ones are generic.
* ``fd``: the same with the finite-difference temperature treatment.
* ``cavity`` / ``channel``: the wall-bounded validation runs (Tables I and II).
* ``sweep``: a batch of uneven domains advanced towards its steady state.
* ``predict``: the warm-start network on new cases and the handoff of its
  prediction to the solver; ``train``: one training step of the network.

The fields of the FP32 storage mode are kept in float32, those of the 16-bit
modes in the mode's own type, those of the FP64 parity mode in float64.
"""
import math

import numpy as np
import torch

from paper_1405_2232_gb300 import lb, unet
from paper_1405_2232_gb300 import inputs as I

STORE = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}
STATE_BYTES = {"fp64": 144, "fp32": 72, "fp16": 40, "bf16": 40}  # f and g of one site
FLOPS = 330  # one site and step: moments, EOS, force stencil, both collisions
THERMAL = {"eq7": lb.LB_THERMAL_EQ7, "eq24": lb.LB_THERMAL_EQ24, "heun": lb.LB_THERMAL_FD26,
           "printed": lb.LB_THERMAL_FD26_PRINTED}


def listed():
    return [
        # the smallest lattice: the sweep's smallest domain on its own, in the default storage; launches count
        dict(name="droplet64_fp32", kind="lattice", nx=64, ny=64, precision="fp32", thermal="eq24",
             start="droplet", beta=1.0, steps=100),
        # the 512^2 droplet (the paper-scale single run): fits the L2 cache
        dict(name="droplet512_fp32", kind="lattice", nx=512, ny=512, precision="fp32", thermal="eq24",
             start="droplet", beta=1.0, steps=100),
        # FP64 parity mode of the same kind of run, not square
        dict(name="droplet384_fp64", kind="lattice", nx=384, ny=320, precision="fp64", thermal="eq24",
             start="droplet", beta=1.3, steps=40),
        # ragged sizes, 16-bit storage, the uncorrected thermal equation
        dict(name="quench1016_fp16_eq7", kind="lattice", nx=1016, ny=765, precision="fp16", thermal="eq7",
             start="quench", beta=1.3, steps=60),
        # the benchmark's lattice, in its storage mode
        dict(name="quench4096_fp32", kind="lattice", nx=4096, ny=4096, precision="fp32", thermal="eq24",
             start="quench", beta=1.3, steps=50),
        # the same in 16-bit storage
        dict(name="quench4096_bf16", kind="lattice", nx=4096, ny=4096, precision="bf16", thermal="eq24",
             start="quench", beta=1.3, steps=50),
        # finite-difference temperature treatment on a large lattice
        dict(name="fd2048_fp32", kind="fd", nx=2048, ny=1600, precision="fp32", thermal="heun", start="quench",
             beta=1.3, steps=50),
        # Table II: natural convection at Ra = 1e4, run in FP64
        dict(name="cavity150_fp64", kind="cavity", nx=150, ny=150, precision="fp64", thermal="eq24", steps=60),
        # Table I: flow between parallel plates on the paper's 500 x 60 nodes, run in FP64
        dict(name="channel500_fp64", kind="channel", nx=500, ny=60, precision="fp64", thermal="eq24", steps=60),
        # part of the parameter sweep: uneven domains of 64..512 nodes a side
        dict(name="sweep28_fp32", kind="sweep", domains=28, lo=64, hi=512, precision="fp32", thermal="eq24",
             steps=400),
        # warm start of a few new cases: network and handoff
        dict(name="predict256", kind="predict", H=256, W=256, N=8),
        # a training step at the package's training size
        dict(name="train256", kind="train", H=256, W=256, N=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice"] * 6 + ["fd", "cavity", "channel", "sweep", "predict", "train"])
    if kind == "lattice":
        prec = rng.choice(["fp32", "fp32", "fp32", "fp16", "bf16", "fp64"])
        hi = 400 if prec == "fp64" else 4000
        nx, ny = _log(rng, 40, hi), _log(rng, 40, hi)
        if prec in ("fp16", "bf16"):
            nx -= nx % 8
        big = nx * ny >= 1 << 19
        return dict(kind=kind, nx=nx, ny=ny, precision=prec, thermal=rng.choice(["eq24", "eq24", "eq7"]),
                    start="quench" if big or prec in ("fp16", "bf16") else "droplet",
                    beta=1.3 if big or prec in ("fp16", "bf16") else rng.choice([1.0, 1.3]),
                    steps=50 if big else rng.choice([40, 60, 101]))
    if kind == "fd":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        hi = 300 if prec == "fp64" else 3000
        return dict(kind=kind, nx=_log(rng, 48, hi), ny=_log(rng, 48, hi), precision=prec,
                    thermal=rng.choice(["heun", "printed"]), start="quench", beta=1.3, steps=40)
    if kind == "cavity":
        n = _log(rng, 40, 250)
        return dict(kind=kind, nx=n, ny=n, precision=rng.choice(["fp64", "fp32"]),
                    thermal="eq24", steps=rng.choice([40, 61]))
    if kind == "channel":
        ny = _log(rng, 20, 100)
        return dict(kind=kind, nx=_log(rng, 4 * ny, 10 * ny), ny=ny, precision="fp64", thermal="eq24",
                    steps=rng.choice([40, 61]))
    if kind == "sweep":
        lo = rng.choice([48, 64, 100])
        return dict(kind=kind, domains=rng.randint(4, 28), lo=lo, hi=rng.randint(2 * lo, 400),
                    precision="fp32", thermal="eq24", steps=200)
    H, W = 8 * _log(rng, 8, 32), 8 * _log(rng, 8, 32)
    return dict(kind=kind, H=H, W=W, N=rng.randint(1, 8) if kind == "predict" else rng.randint(2, 16))


# ------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1234567 + 7919 * int(seed))


def _noise(shape, amp, gen):
    return amp * (2.0 * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64) - 1.0)


def _fields(case, gen):
    """Initial density and temperature of a lattice and the constant T that psi takes."""
    nx, ny = case["nx"], case["ny"]
    x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :]
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None]
    if case["start"] == "quench":
        T0 = 0.75 * I.CS_TC
        rho = 0.12 + _noise((ny, nx), 0.01, gen)
    else:
        T0 = 0.85 * I.CS_TC
        rg, rl = I.coexistence_densities(0.85)
        inside = (x - nx / 2 + 0.5) ** 2 + (y - ny / 2 + 0.5) ** 2 < (min(nx, ny) / 4) ** 2
        rho = torch.where(inside, rl, rg) + _noise((ny, nx), 1e-3, gen)
    return rho.contiguous(), torch.full((ny, nx), T0, device="cuda", dtype=torch.float64), T0


def _wall_params(case):
    """Parameters of the cavity (Ra = 1e4 as in Table II) or the channel (Case A of Table I)."""
    nu, Pr = 0.1, 0.71
    p = dict(nx=case["nx"], ny=case["ny"], precision=case["precision"], thermal=THERMAL[case["thermal"]],
             eos=lb.LB_EOS_IDEAL, a=0.0, b=0.0, R=1.0 / 3.0, cv=1.0, G=1.0, beta=0.0, psi_uses_local_T=1,
             tau_f=0.5 + 3.0 * nu, tau_g=0.5 + 3.0 * nu / Pr)
    if case["kind"] == "cavity":
        p.update(walls=lb.LB_WALLS_CAVITY, T_hot=1.03, T_cold=0.97,
                 g_grav=1e4 * nu * nu / Pr / (0.06 * case["nx"] ** 3))
    else:
        p.update(walls=lb.LB_WALLS_CHANNEL, T_in=1.03, T_w=0.97, U_in=0.05, adiabatic_bottom=0)
    return p


def _lattice_setup(case, seed):
    """(lb_params fields, rho0, T0) of a single-lattice case."""
    gen = _gen(seed)
    if case["kind"] in ("cavity", "channel"):
        shape = (case["ny"], case["nx"])
        return _wall_params(case), 1.0 + _noise(shape, 1e-2, gen), 1.0 + _noise(shape, 1e-2, gen)
    rho, T, T_psi = _fields(case, gen)
    p = dict(nx=case["nx"], ny=case["ny"], precision=case["precision"], thermal=THERMAL[case["thermal"]],
             tau_f=1.0, tau_g=0.8, G=-1.0, beta=case["beta"], psi_uses_local_T=0, T_psi=T_psi)
    if case["precision"] in ("fp16", "bf16"):
        p.update(rho0=0.12, T0=T_psi)
    return p, rho, T


def _sides(case):
    return np.random.default_rng(case["domains"]).integers(case["lo"], case["hi"] + 1, case["domains"]).tolist()


def _sweep_setup(case, seed):
    """Domains of the sweep recipe: side, EOS temperature, G and tau_f vary, droplets and slabs."""
    rng = np.random.default_rng(99991 + int(seed))
    gen = _gen(seed)
    params, rhos, Ts = [], [], []
    for L in _sides(case):
        t = float(rng.uniform(0.78, 0.95))
        rg, rl = I.coexistence_densities(t)
        xy = torch.arange(L, device="cuda", dtype=torch.float64) - L / 2 + 0.5
        if rng.random() < 0.5:
            inside = xy[None, :] ** 2 + xy[:, None] ** 2 < (L * rng.uniform(0.125, 0.25)) ** 2
        else:
            inside = (xy.abs() < L * rng.uniform(0.125, 0.25))[None, :].expand(L, L)
        params.append(dict(nx=L, ny=L, precision=case["precision"], thermal=THERMAL[case["thermal"]],
                           tau_f=float(rng.uniform(0.7, 1.2)), tau_g=0.8, G=float(rng.uniform(-1.2, -0.8)),
                           beta=1.3, psi_uses_local_T=0, T_psi=t * I.CS_TC))
        rhos.append((torch.where(inside, rl, rg) + _noise((L, L), 1e-4, gen)).contiguous())
        Ts.append(torch.full((L, L), t * I.CS_TC, device="cuda", dtype=torch.float64))
    return params, rhos, Ts


def _net_arch(base=32):
    """(input channels as stored, output channels, kernel, real fan-in) in the flat parameter order."""
    enc = [(32, base, 3, 3), (base, base, 3, base)]
    for l in range(1, 4):
        w = base << l
        enc += [(w // 2, w, 3, w // 2), (w, w, 3, w)]
    dec = []
    for l in (2, 1, 0):
        w = base << l
        dec += [(3 * w, w, 3, 3 * w), (w, w, 3, w)]
    return enc + dec + [(base, 2, 1, base)]


def _net_params(gen):
    out = []
    for ci, co, k, real in _net_arch():
        std = math.sqrt((2.0 if k == 3 else 1.0) / (k * k * real))
        W = torch.randn((co, k, k, ci), generator=gen, device="cuda") * std
        W[..., real:] = 0.0
        out += [W.reshape(-1), 0.02 * torch.randn(co, generator=gen, device="cuda")]
    return torch.cat(out)


def _net_inputs(case, gen):
    """Input planes of N cases (T/T_c, G, mask) and their initial fields."""
    N, H, W = case["N"], case["H"], case["W"]
    u = torch.rand((N, 3), generator=gen, device="cuda", dtype=torch.float64)
    t, g = 0.7 + 0.25 * u[:, 0], -1.2 + 0.4 * u[:, 1]
    x = torch.arange(W, device="cuda", dtype=torch.float64)[None, None, :] - W / 2 + 0.5
    y = torch.arange(H, device="cuda", dtype=torch.float64)[None, :, None] - H / 2 + 0.5
    radius = min(H, W) * (0.125 + 0.125 * u[:, 2])
    mask = (x * x + y * y < (radius * radius)[:, None, None]).double()
    planes = torch.stack([((t - 0.775) / 0.1)[:, None, None].expand(N, H, W),
                          ((g + 1.0) / 0.2)[:, None, None].expand(N, H, W), 2.0 * mask - 1.0], dim=3)
    dens = [I.coexistence_densities(float(v)) for v in t.cpu()]
    rg, rl = (torch.tensor([d[k] for d in dens], device="cuda", dtype=torch.float64)[:, None, None] for k in (0, 1))
    T0 = (t * I.CS_TC)[:, None, None].expand(N, H, W)
    return planes.float().contiguous(), (rg + (rl - rg) * mask).contiguous(), T0.contiguous()


# ------------------------------------------------------- prepare, run, work
_stream = None  # one stream for all states: a program that runs one simulation after the other


def prepare(case, seed):
    global _stream
    stream = _stream = _stream or torch.cuda.Stream()
    state = dict(kind=case["kind"], stream=stream)
    if case["kind"] in ("lattice", "fd", "cavity", "channel"):
        p, rho, T = _lattice_setup(case, seed)
        torch.cuda.synchronize()
        L = lb.Lattice(rho, T, stream=stream, device_inputs=True, **p)
        out = [torch.empty((case["ny"], case["nx"]), device="cuda", dtype=torch.float64) for _ in range(4)]
        state.update(L=L, out=out, steps=case["steps"], store=STORE[case["precision"]])
    elif case["kind"] == "sweep":
        params, rhos, Ts = _sweep_setup(case, seed)
        torch.cuda.synchronize()
        B = lb.Batch([lb.lb_params_default(**p) for p in params], rhos, Ts, stream=stream, device_inputs=True)
        state.update(B=B, n=case["domains"], steps=case["steps"])
    else:
        gen = _gen(seed)
        N, H, W = case["N"], case["H"], case["W"]
        weights = _net_params(gen)
        x, rho0, T0 = _net_inputs(case, gen)
        net = unet.UNet(H, W, N, stream=stream)
        torch.cuda.synchronize()
        net.set_params(weights)
        state.update(net=net, x=x, N=N, shape=(H, W))
        if case["kind"] == "predict":
            state.update(rho0=rho0, T0=T0, y=torch.empty((N, H, W, 2), device="cuda"),
                         rho=torch.empty_like(rho0), T=torch.empty_like(T0))
        else:
            state.update(target=_target(case, gen, x))
    torch.cuda.synchronize()
    return state


def _target(case, gen, x):
    """Training targets: a smooth response to the mask plane, of the size real targets have."""
    blur = x[..., 2:3]
    for _ in range(3):
        blur = sum(torch.roll(blur, (dy, dx), (1, 2)) for dy in (-1, 0, 1) for dx in (-1, 0, 1)) / 9.0
    amp = 0.5 + torch.rand((case["N"], 1, 1, 2), generator=gen, device="cuda")
    return (amp * (blur - x[..., 2:3])).contiguous()


def run(state):
    kind, s = state["kind"], state["stream"]
    with torch.cuda.stream(s):
        if kind in ("lattice", "fd", "cavity", "channel"):
            state["L"].step(state["steps"])
            rho, ux, uy, T = state["out"]
            lb.lb_moments_device(state["L"].ctx, rho, ux, uy, T)
            return {k: v.to(state["store"]) for k, v in zip(("rho", "ux", "uy", "T"), (rho, ux, uy, T))}
        if kind == "sweep":
            B = state["B"]
            steps, resid, status = B.run(1e-8, K=100, max_steps=state["steps"])
            fields = [B.fields(d) for d in range(state["n"])]
            return {"steps": steps, "status": status, "residual": resid.astype(np.float32),
                    "rho": [r.astype(np.float32) for r, _ in fields],
                    "T": [t.astype(np.float32) for _, t in fields]}
        net = state["net"]
        if kind == "predict":
            H, W = state["shape"]
            net.forward(state["x"], state["y"], state["N"])
            unet.warm_fields(state["N"], H, W, state["y"], I.UNET_NORM, state["rho0"], state["T0"], state["rho"],
                             state["T"], stream=s)
            return {"y": state["y"], "rho": state["rho"], "T": state["T"]}
        loss = net.train_step(state["x"], state["target"], state["N"], 1e-3)
        return {"loss": loss, "grads": net.grads()}


def work(case):
    """Bytes and operations of one pass: each step reads and writes every population of every site once."""
    kind = case["kind"]
    if kind in ("lattice", "cavity", "channel", "fd"):
        n = case["nx"] * case["ny"]
        word = torch.empty(0, dtype=STORE[case["precision"]]).element_size()
        site = 10 * word if kind == "fd" else STATE_BYTES[case["precision"]]
        return {"bytes": n * (2 * site * case["steps"] + 4 * word), "flops": n * FLOPS * case["steps"]}
    if kind == "sweep":
        n = sum(v * v for v in _sides(case))
        return {"bytes": n * (2 * 72 * case["steps"] + 16), "flops": n * FLOPS * case["steps"]}
    px, par, mac = case["N"] * case["H"] * case["W"], 0, 0.0
    levels = [0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0, 0]
    act = 0.0  # BF16 activations: each layer's output written and read once
    for (ci, co, k, real), l in zip(_net_arch(), levels):
        par += ci * co * k * k + co
        mac += px / 4 ** l * real * co * k * k
        act += 4.0 * px / 4 ** l * co
    if kind == "predict":
        return {"bytes": px * (12 + 8 + 32) + act + 2 * par, "flops": 2 * mac}
    first = px * 3 * 32 * 9  # no input gradient at the first layer
    return {"bytes": px * (12 + 8) + 3 * act + 28 * par, "flops": 2 * (3 * mac - first)}


# ----------------------------------------------------------- 64-bit results
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


class _Reference:
    """The method in plain 64-bit torch over a flat list of sites (one lattice, or several side by side)."""

    def __init__(self, p, shapes, rho, T):
        self.p = p  # parameters: numbers, or one value per site
        self.walls = p.get("walls", 0)
        nb, inside, at, first = [[] for _ in range(9)], [[] for _ in range(9)], [], 0
        for ny, nx in shapes:
            y, x = torch.meshgrid(torch.arange(ny, device="cuda"), torch.arange(nx, device="cuda"), indexing="ij")
            for i in range(9):
                xn, yn = x + EX[i], y + EY[i]
                inside[i].append(torch.stack([(xn >= 0) & (xn < nx), (yn >= 0) & (yn < ny)]).reshape(2, -1))
                xn, yn = (xn.clamp(0, nx - 1), yn.clamp(0, ny - 1)) if self.walls else (xn % nx, yn % ny)
                nb[i].append((first + yn * nx + xn).reshape(-1))
            at.append(torch.stack([x, y]).reshape(2, -1))
            first += ny * nx
        self.nb = [torch.cat(v) for v in nb]
        self.inside = [torch.cat(v, 1) for v in inside] if self.walls else None
        self.x, self.y = torch.cat(at, 1)
        self.shape = shapes[0]
        self.fd = p["thermal"] >= 2
        self.f = torch.stack([w * rho for w in WT])
        self.T = T
        self.g = None if self.fd else p["cv"] * T * self.f

    def psi_sq(self, rho, T):
        p = self.p
        Te = T if p["psi_uses_local_T"] else p["T_psi"]
        if p["eos"] == lb.LB_EOS_IDEAL:
            pr = rho * p["R"] * Te
        else:
            eta = p["b"] * rho / 4
            pr = rho * p["R"] * Te * (1 + eta + eta ** 2 - eta ** 3) / (1 - eta) ** 3 - p["a"] * rho ** 2
        return 2 * (pr - rho / 3) / p["G"]

    def macro(self):
        p = self.p
        rho = self.f.sum(0)
        T = self.T if self.fd else self.g.sum(0) / (rho * p["cv"])
        q = self.psi_sq(rho, T)
        psi = None if p["beta"] == 0.0 else q.sqrt()
        Fx, Fy = torch.zeros_like(rho), torch.zeros_like(rho)
        for v, c in ((psi, p["beta"]), (q, 0.5 * (1 - p["beta"]))):
            if v is None or c == 0.0:
                continue
            sx, sy = torch.zeros_like(rho), torch.zeros_like(rho)
            for i in range(1, 9):
                n = v[self.nb[i]] * (1 / 3 if i < 5 else 1 / 12)
                if EX[i]:
                    sx += EX[i] * n
                if EY[i]:
                    sy += EY[i] * n
            k = -p["G"] * c
            Fx += k * (v * sx if v is psi else sx)
            Fy += k * (v * sy if v is psi else sy)
        if self.walls == lb.LB_WALLS_CAVITY:
            Fy -= rho * p["g_grav"]
        mx = sum(EX[i] * self.f[i] for i in range(9) if EX[i])
        my = sum(EY[i] * self.f[i] for i in range(9) if EY[i])
        return rho, (mx + Fx / 2) / rho, (my + Fy / 2) / rho, T, Fx, Fy

    def grad(self, v):
        gx, gy, lap = torch.zeros_like(v), torch.zeros_like(v), torch.zeros_like(v)
        for i in range(1, 9):
            n = v[self.nb[i]]
            gx += 3 * WT[i] * EX[i] * n
            gy += 3 * WT[i] * EY[i] * n
            lap += 6 * WT[i] * (n - v)
        return gx, gy, lap

    def step(self):
        p = self.p
        rho, ux, uy, T, Fx, Fy = self.macro()
        if self.fd:
            chi = (p["tau_g"] - 0.5) / 3
            rx, ry, _ = self.grad(rho)

            def K(v):
                gx, gy, lap = self.grad(v)
                return -(ux * gx + uy * gy) + chi * (lap + (rx * gx + ry * gy) / rho)

            h1 = K(T)
            self.T = T + 0.5 * (h1 + K(T + (1.0 if p["thermal"] == lb.LB_THERMAL_FD26 else 0.5) * h1))
        usq, cvT, uF = ux * ux + uy * uy, p["cv"] * T, ux * Fx + uy * Fy
        of, og = 1 / p["tau_f"], 1 / p["tau_g"]
        fs, gs = torch.empty_like(self.f), None if self.fd else torch.empty_like(self.g)
        for i in range(9):
            eu, eF = EX[i] * ux + EY[i] * uy, EX[i] * Fx + EY[i] * Fy
            feq = WT[i] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * usq)
            fs[i] = self.f[i] - of * (self.f[i] - feq) + (1 - 0.5 * of) * WT[i] * (3 * (eF - uF) + 9 * eu * eF)
            if not self.fd:
                gs[i] = self.g[i] - og * (self.g[i] - cvT * feq)
                if p["thermal"] == lb.LB_THERMAL_EQ24:
                    gs[i] += (1 - 0.5 * og) * WT[i] * 3 * cvT * eF
        fn, gn = torch.empty_like(fs), None if self.fd else torch.empty_like(gs)
        for i in range(9):
            o = OPP[i]  # what arrives along i comes from the neighbour at e_o, or back from a wall there
            fn[i] = fs[i][self.nb[o]]
            if not self.fd:
                gn[i] = gs[i][self.nb[o]]
            if self.walls and i:
                self.bounce(i, o, fs, gs, fn, gn, rho, ux, uy)
        if self.walls == lb.LB_WALLS_CHANNEL:
            ny, nx = self.shape
            for i in (3, 6, 7):
                rows = slice(max(0, EY[i]), ny + min(0, EY[i]))
                v = gn[i].view(ny, nx)
                v[rows, nx - 1] = v[rows, nx - 2]
        self.f, self.g = fn, gn

    def bounce(self, i, o, fs, gs, fn, gn, rho, ux, uy):
        p, w = self.p, WT[i]
        in_x, in_y = self.inside[o]
        iso = lambda Tw: -gs[o] + 2 * w * p["cv"] * Tw * rho  # noqa: E731
        if self.walls == lb.LB_WALLS_CAVITY:
            fn[i] = torch.where(in_x & in_y, fn[i], fs[o])
            side = iso(p["T_hot"] if EX[o] < 0 else p["T_cold"])
            gn[i] = torch.where(in_x & in_y, gn[i], torch.where(in_x, gs[o], side))
            return
        if EX[o] < 0:
            eu = EX[o] * p["U_in"]
            f_end = fs[o] - 6 * w * rho * eu
            g_end = iso(p["T_in"] * (1 + 4.5 * eu * eu - 1.5 * p["U_in"] ** 2))
        else:
            eu = EX[o] * ux + EY[o] * uy
            f_end = -fs[o] + 2 * w * (1 + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy))
            g_end = gn[i]
        fn[i] = torch.where(in_y, torch.where(in_x, fn[i], f_end), fs[o])
        gn[i] = torch.where(in_y, torch.where(in_x, gn[i], g_end), iso(p["T_w"]))


_DEFAULTS = dict(eos=lb.LB_EOS_CS, a=1.0, b=4.0, R=1.0, cv=1.0)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("lattice", "fd", "cavity", "channel"):
        p, rho, T = _lattice_setup(case, seed)
        ref = _Reference({**_DEFAULTS, **p}, [(case["ny"], case["nx"])], rho.reshape(-1), T.reshape(-1))
        for _ in range(case["steps"]):
            ref.step()
        out = ref.macro()[:4]
        return {k: v.reshape(case["ny"], case["nx"]) for k, v in zip(("rho", "ux", "uy", "T"), out)}
    if kind == "sweep":
        params, rhos, Ts = _sweep_setup(case, seed)
        shapes = [tuple(r.shape) for r in rhos]
        sizes = torch.tensor([r.numel() for r in rhos], device="cuda")
        per_site = {k: torch.repeat_interleave(torch.tensor([q[k] for q in params], device="cuda",
                                                            dtype=torch.float64), sizes)
                    for k in ("tau_f", "G", "T_psi")}
        ref = _Reference({**_DEFAULTS, **params[0], **per_site}, shapes, torch.cat([r.reshape(-1) for r in rhos]),
                         torch.cat([t.reshape(-1) for t in Ts]))
        n = sizes.tolist()
        for k in range(case["steps"]):
            if k == case["steps"] - 100:
                before = [v.split(n) for v in (ref.macro()[0], ref.macro()[3])]
            ref.step()
        now = [v.split(n) for v in (ref.macro()[0], ref.macro()[3])]
        resid = [max(float((b - a).norm() / (100.0 * b.norm())) for a, b in zip(va, vb))
                 for va, vb in zip(zip(*before), zip(*now))]
        return {"steps": None, "status": None, "residual": torch.tensor(resid, dtype=torch.float64),
                "rho": [v.reshape(s) for v, s in zip(now[0], shapes)],
                "T": [v.reshape(s) for v, s in zip(now[1], shapes)]}
    return _net_exact(case, seed)


def _net_exact(case, seed):
    gen = _gen(seed)
    flat = _net_params(gen).double().requires_grad_(case["kind"] == "train")
    x, rho0, T0 = _net_inputs(case, gen)
    P, o = [], 0
    for ci, co, k, _ in _net_arch():
        n = co * k * k * ci
        P.append((flat[o:o + n].view(co, k, k, ci), flat[o + n:o + n + co]))
        o += n + co

    def conv(v, layer):
        W, b = P[layer]
        c = v.shape[3]  # the padding channels of the first layer hold zeros
        taps = [torch.roll(v, (-dy, -dx), (1, 2)) @ W[:, dy + 1, dx + 1, :c].T
                for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
        return torch.relu(sum(taps) + b)

    v, skips = x.double(), []
    for l in range(4):
        v = conv(conv(v, 2 * l), 2 * l + 1)
        if l < 3:
            skips.append(v)
            n, h, w, c = v.shape
            v = v.reshape(n, h // 2, 2, w // 2, 2, c).mean((2, 4))
    for k, l in enumerate((2, 1, 0)):
        v = torch.cat([v.repeat_interleave(2, 1).repeat_interleave(2, 2), skips[l]], 3)
        v = conv(conv(v, 8 + 2 * k), 9 + 2 * k)
    y = v @ P[14][0].view(2, -1).T + P[14][1]
    if case["kind"] == "train":
        loss = ((y - _target(case, gen, x).double()) ** 2).mean()
        loss.backward()
        return {"loss": float(loss), "grads": flat.grad}
    norm = I.UNET_NORM
    r = (rho0 + norm["rho_dev_scale"] * y[..., 0]).clamp(min=1e-4)
    Th = T0 * (1 + norm["t_dev_scale"] * y[..., 1])
    total = lambda a: a.sum((1, 2), keepdim=True)  # noqa: E731
    lo, hi = r.amin((1, 2), keepdim=True), r.amax((1, 2), keepdim=True)
    wgt = (r - lo) * (hi - r)
    lam = (total(rho0) - total(r)) / total(wgt)
    lam = torch.minimum(torch.maximum(lam, -1 / (hi - lo)), 1 / (hi - lo))
    r = r + lam * wgt
    r = r * total(rho0) / total(r)
    return {"y": y, "rho": r, "T": Th * total(rho0 * T0) / total(r * Th)}
