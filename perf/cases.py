"""Timed workloads of the vielbein lattice-Boltzmann + Cahn-Hilliard framework.

Each case is one call as a user's program makes it, on a state that stands for a run under way: phase
domains with tanh walls, a smooth flow of a few per cent of the thermal speed and a density near 1.
The families are

  step      ``vlb.Solver.step``: a torus or flat grid, FP32 or FP64, UW3 or WENO5, hydrodynamic or
            diffusive, explicit or stabilised Cahn-Hilliard, axisymmetric (n_phi = 1) or not
  ensemble  ``vlb.Ensemble.step``: many tori of uneven grids in one call
  measure   the sampling of a coarsening run: conserved totals, interface length, structure length
  layer     one periodic 3 x 3 convolution of the surrogate network, forward and backward
  network   one training iteration, or one prediction, of the whole surrogate network

``exact`` restates every family in plain FP64 torch from the definitions (arXiv:1904.10070, Secs. 2-4).
"""
import math
import random

import numpy as np
import torch

from paper_1904_10070_gb300 import surrogate, vlb

DEV = "cuda"
F64 = torch.float64

COARSEN = dict(R=2.0, r=1.0, tau=0.6, M=2.5e-3, A=0.5, kappa=5e-4)  # the coarsening workload's fluid
PAPER = dict(R=2.5, r=1.0, tau=2.5e-3, M=2.5e-3, A=0.5, kappa=5e-4)  # the paper's phase-separation fluid
STEP = dict(family="step", fp64=False, weno=False, diffusive=False, flat=False, stab=False)


def listed():
    return [
        # a small FP64 reference run (32 x 64 drop torus): every launch is latency
        dict(STEP, name="drop_fp64_32x64", fp64=True, n_theta=32, n_phi=64, steps=10, R=2.5, r=1.0, tau=0.8, M=0.1,
             A=0.04, kappa=0.04),
        # the stripe-oscillation grid in both precisions (tens of thousands of steps each)
        dict(STEP, name="stripe_fp32_128x384", n_theta=128, n_phi=384, steps=20, R=3.0, r=1.0, tau=2.5e-3, M=2.5e-3,
             A=0.5, kappa=1.25e-3),
        dict(STEP, name="stripe_fp64_128x384", fp64=True, n_theta=128, n_phi=384, steps=4, R=3.0, r=1.0, tau=2.5e-3,
             M=2.5e-3, A=0.5, kappa=1.25e-3),
        # the headline coarsening run: state larger than L2
        dict({**STEP, **COARSEN}, name="coarsen_fp32_1024x2048", n_theta=1024, n_phi=2048, steps=4),
        # the other advection scheme, on a flat periodic domain
        dict({**STEP, **PAPER}, name="weno5_fp32_256x512", weno=True, flat=True, n_theta=256, n_phi=512, steps=4),
        # a grid nobody chose for the machine: odd n_phi, rows that are no multiple of a tile; the
        # diffusive regime (no flow in Cahn-Hilliard, no force)
        dict({**STEP, **PAPER}, name="diffusive_fp32_250x501", diffusive=True, n_theta=250, n_phi=501, steps=8),
        # the paper's axisymmetric stripe study: one varphi column of 320 rows, millions of steps
        dict(STEP, name="axisymmetric_fp32_320x1", n_theta=320, n_phi=1, steps=64, R=2.0, r=0.8, tau=2.5e-3, M=2.5e-3,
             A=0.5, kappa=5e-4),
        # long coarsening runs: large steps through the Fourier-stabilised Cahn-Hilliard stages
        dict({**STEP, **COARSEN}, name="stabilised_fp32_1024x2048", stab=True, n_theta=1024, n_phi=2048, steps=2),
        # parameter studies: tori of uneven size advanced together
        dict(family="ensemble", name="ensemble_24_tori", count=24, pick=4, odd=False, steps=8),
        # what a coarsening run samples between blocks of steps
        dict(COARSEN, family="measure", name="measure_fp32_1024x2048", fp64=False, flat=False, n_theta=1024, n_phi=2048),
        # the layer that dominates the surrogate network, in training
        dict(family="layer", name="layer_64_64_256x512", H=256, W=512, cin=64, cout=64),
        # one training iteration of the surrogate at its working grid
        dict(family="network", name="network_train_256x512", H=256, W=512, mode="train"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["step"] * 7 + ["ensemble", "measure", "layer", "network"])
    if family == "layer":
        cin, cout = rng.choice([(16, 64), (64, 64), (64, 16)])
        return dict(family=family, H=2 * _log_int(rng, 4, 128), W=128 * rng.randint(1, 4), cin=cin, cout=cout)
    if family == "network":
        return dict(family=family, H=2 * _log_int(rng, 8, 128), W=128 * rng.randint(1, 4),
                    mode=rng.choice(["train", "predict"]))
    if family == "ensemble":
        return dict(family=family, count=rng.randint(2, 24), pick=rng.randrange(1 << 20), odd=rng.random() < 0.5,
                    steps=rng.randint(1, 8))
    fluid = dict(R=round(rng.uniform(1.5, 4.0), 3), r=1.0, tau=rng.choice([2.5e-3, 0.1, 0.6]), M=2.5e-3, A=0.5,
                 kappa=rng.choice([5e-4, 1.25e-3]))
    if family == "measure":
        return dict(fluid, family=family, fp64=rng.random() < 0.3, flat=rng.random() < 0.3,
                    n_theta=2 ** rng.randint(4, 10), n_phi=2 ** rng.randint(5, 11))
    c = {**STEP, **fluid}
    kind = rng.choice(["plain", "plain", "plain", "odd", "axisymmetric", "stab"])
    c["fp64"] = rng.random() < 0.3
    c["diffusive"] = rng.random() < 0.25
    c["flat"] = rng.random() < 0.25
    c["weno"] = rng.random() < 0.25
    if kind == "axisymmetric":
        return dict(c, n_theta=_log_int(rng, 64, 768 if not c["fp64"] else 384), n_phi=1, steps=rng.randint(4, 64))
    if kind == "stab":
        return dict(c, weno=False, stab=True, n_theta=2 ** rng.randint(5, 9), n_phi=2 ** rng.randint(6, 10),
                    steps=rng.randint(1, 4))
    slow = c["fp64"] or c["weno"]
    nt, ns = _log_int(rng, 16, 256 if slow else 768), _log_int(rng, 32, 512 if slow else 1536)
    if kind == "plain":
        nt, ns = 8 * max(2, nt // 8), 8 * max(4, ns // 8)
    else:
        nt, ns = nt | 1, ns | 1
    return dict(c, n_theta=nt, n_phi=ns, steps=max(1, min(10, int(2e6 / (nt * ns)))))


# ------------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------------

def _smooth(gen, nt, ns, cells):
    """A periodic Gaussian random field of zero mean and unit variance, correlated over `cells` nodes."""
    x = torch.randn((nt, ns), generator=gen, device=DEV, dtype=F64)
    ft = torch.fft.fftfreq(nt, device=DEV, dtype=F64)[:, None]
    fs = torch.fft.fftfreq(ns, device=DEV, dtype=F64)[None, :]
    cells = min(cells, nt / 6.0)
    g = torch.fft.ifft2(torch.fft.fft2(x) * torch.exp(-2.0 * (math.pi * cells) ** 2 * (ft * ft + fs * fs))).real
    g = g - g.mean()
    return g / g.std()


def _fields(seed, nt, ns):
    """(rho, u_theta, u_phi, phi) of a run under way, on the GPU in FP64."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    rho = 1.0 + 0.005 * _smooth(gen, nt, ns, 8.0)
    ut = 0.03 * _smooth(gen, nt, ns, 10.0)
    up = 0.03 * _smooth(gen, nt, ns, 10.0)
    phi = torch.tanh(2.5 * _smooth(gen, nt, ns, 6.0))
    return rho, ut, up, phi


def _dt(c):
    """Half the smaller of the advection-plus-relaxation and the Cahn-Hilliard stability limits."""
    ht = c["r"] * 2.0 * math.pi / c["n_theta"]
    hp = (c["R"] if c.get("flat") else c["R"] - c["r"]) * 2.0 * math.pi / c["n_phi"]
    wide = c["n_phi"] > 1
    rate = math.sqrt(3.0 + math.sqrt(6.0)) * (1.0 / ht + (1.0 / hp if wide else 0.0)) + 0.5 / c["tau"]
    if c.get("stab"):
        ch = c["A"] ** 2 * c["M"] / (6.25 * c["kappa"])
    else:
        lam = 4.0 / ht ** 2 + (4.0 / hp ** 2 if wide else 0.0)
        ch = c["M"] * lam * (c["kappa"] * lam + 2.0 * c["A"]) / 2.5
    return 0.5 / max(rate, ch)


def _params(c):
    return vlb.make_params(R=c["R"], r=c["r"], n_theta=c["n_theta"], n_phi=c["n_phi"], dt=_dt(c), tau=c["tau"], M=c["M"],
                           A=c["A"], kappa=c["kappa"], geometry=vlb.FLAT if c.get("flat") else vlb.TORUS,
                           precision=vlb.FP64 if c.get("fp64") else vlb.FP32,
                           advection=vlb.WENO5 if c.get("weno") else vlb.UW3,
                           ch_mode=vlb.DIFFUSIVE if c.get("diffusive") else vlb.HYDRO, ch_stab=1 if c.get("stab") else 0)


def _members(c):
    """The ensemble's member cases: R spread over [1.3, 5], grids of the batched workload or odd ones."""
    rng, out = random.Random(c["pick"]), []
    for i in range(c["count"]):
        nt, ns = rng.choice([(64, 128), (128, 256), (256, 512), (512, 1024)])
        if c["odd"]:
            nt, ns = rng.randint(40, 320), rng.randint(60, 640)
        R = 1.3 + 3.7 * i / max(c["count"] - 1, 1)
        out.append(dict(PAPER, R=R, n_theta=nt, n_phi=ns))
    return out


def _state_views(handle, workspace, nt, ns, fp64):
    """The resident state as tensors: the 16 population deviations and phi (FP32: its high word)."""
    ptr, stride = vlb.vlb_state_device(handle)
    size, dtype = (8, F64) if fp64 else (4, torch.float32)
    at = ptr - workspace.data_ptr()
    flat = workspace[at:at + 17 * stride * size].view(dtype)
    return {"g": flat.as_strided((16, nt, ns), (stride, ns, 1)), "phi": flat[16 * stride:].as_strided((nt, ns), (ns, 1))}


def _set(handle, fields):
    vlb.vlb_set_fields(handle, *[x.cpu().numpy() for x in fields])


def _layer_inputs(c, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    H, W, cin, cout = c["H"], c["W"], c["cin"], c["cout"]
    x = torch.relu(torch.randn((H, W, cin), generator=gen, device=DEV)).to(torch.bfloat16)
    dy = (1e-3 * torch.randn((H, W, cout), generator=gen, device=DEV)).to(torch.bfloat16)
    w = (math.sqrt(2.0 / (9 * cin)) * torch.randn((cout, 3, 3, cin), generator=gen, device=DEV)).to(torch.bfloat16)
    b = 0.1 * torch.randn((cout,), generator=gen, device=DEV)
    return x, dy, w, b


RATIOS, SCALE_N, SCALE_U, NET_R, LR = (0.05, 0.2, 0.3, 0.3), 0.005, 0.03, 2.5, 1e-3
ADAM_T, ADAM_V = 1000, 1e-6  # a training under way: steps taken, second moment of every parameter


def _network_inputs(c, seed):
    """Snapshots (phi, n, u_theta, u_phi) before and after a window, He-initialised weights and biases."""
    H, W = c["H"], c["W"]

    def snap(s):
        rho, ut, up, phi = _fields(s, H, W)
        return torch.stack([phi, rho, ut, up], dim=-1).reshape(H * W, 4)

    before = snap(seed)
    after = (before + 0.05 * (snap(seed + 1) - before)).to(torch.float32).contiguous()
    gen = torch.Generator(device=DEV).manual_seed(seed + 2)
    ws, bs = [], []
    for k, (cin, cout) in enumerate([(16, 64)] + [(64, 64)] * 6 + [(64, 16)]):
        w = torch.randn((cout, 3, 3, cin), generator=gen, device=DEV) * math.sqrt(2.0 / (9 * (10 if k == 0 else cin)))
        b = 0.1 * torch.randn((cout,), generator=gen, device=DEV)
        if k == 0:
            w[..., 10:] = 0.0
        if k == 7:
            w *= 0.1
            w[4:] = 0.0
            b[4:] = 0.0
        ws.append(w)
        bs.append(b)
    return before.to(torch.float32).contiguous(), after, ws, bs


def prepare(case, seed):
    fam = case["family"]
    if fam in ("step", "measure"):
        s = vlb.Solver(_params(case))
        _set(s.h, _fields(seed, case["n_theta"], case["n_phi"]))
        if fam == "measure":
            return dict(case=case, solver=s)
        return dict(case=case, solver=s, out=_state_views(s.h, s.workspace, *s.shape, case["fp64"]))
    if fam == "ensemble":
        ms = _members(case)
        ens = vlb.Ensemble([_params(m) for m in ms])
        for k, (v, m) in enumerate(zip(ens.views, ms)):
            _set(v, _fields(seed + 1000 * k, m["n_theta"], m["n_phi"]))
        out = [_state_views(v, ens.workspace, m["n_theta"], m["n_phi"], False) for v, m in zip(ens.views, ms)]
        return dict(case=case, ens=ens, out=out)
    if fam == "layer":
        x, dy, w, b = _layer_inputs(case, seed)
        H, W, cin, cout = case["H"], case["W"], case["cin"], case["cout"]
        like = lambda shape, dt: torch.empty(shape, dtype=dt, device=DEV)  # noqa: E731
        ws = like((vlb.vlb_conv3x3_wgrad_workspace_bytes(H, W, cin, cout),), torch.uint8)
        out = dict(y=like((H, W, cout), torch.bfloat16), dx=like((H, W, cin), torch.bfloat16),
                   dw=like((cout, 3, 3, cin), torch.float32), db=like((cout,), torch.float32))
        return dict(case=case, x=x, dy=dy, w=w, b=b, wf=like((cin, 3, 3, cout), torch.bfloat16), ws=ws, out=out)
    H, W = case["H"], case["W"]
    before, after, weights, biases = _network_inputs(case, seed)
    net = surrogate.SurrogateNet(H, W, seed=0)
    net.t = ADAM_T
    for k, (w, b) in enumerate(zip(weights, biases)):
        net.w32[k].copy_(w)
        net.wb[k].copy_(w)
        net.b32[k].copy_(b)
        net.vw[k].fill_(ADAM_V)
        net.vb[k].fill_(ADAM_V)
    tr = surrogate.Trainer(net, RATIOS, SCALE_N, SCALE_U)
    if case["mode"] == "predict":
        return dict(case=case, tr=tr, snap=before, norm8=torch.empty(8, device=DEV), pred=torch.empty_like(before))
    ds = surrogate.Dataset([before], [after], [NET_R], [(1.0, 1.0, SCALE_N, SCALE_U)])
    tr.prepare(ds)
    return dict(case=case, tr=tr, ds=ds)


# ------------------------------------------------------------------------------------------------
# One pass
# ------------------------------------------------------------------------------------------------

def run(state):
    case = state["case"]
    fam = case["family"]
    if fam == "step":
        state["solver"].step(case["steps"])
        return state["out"]
    if fam == "ensemble":
        state["ens"].step(case["steps"])
        return state["out"]
    if fam == "measure":
        s = state["solver"]
        return dict(totals=s.totals(), interface=s.interface_length(), structure=s.structure_length())
    if fam == "layer":
        H, W, cin, cout = case["H"], case["W"], case["cin"], case["cout"]
        st, out = torch.cuda.current_stream().cuda_stream, state["out"]
        x, dy, w, wf = state["x"], state["dy"], state["w"], state["wf"]
        vlb.vlb_conv3x3_fwd(H, W, cin, cout, x, w, state["b"], None, 1, out["y"], None, st)
        vlb.vlb_conv3x3_bwd_weight(H, W, cin, cout, x, dy, out["dw"], out["db"], state["ws"], st)
        vlb.vlb_conv3x3_flip(cin, cout, w, wf, st)
        vlb.vlb_conv3x3_fwd(H, W, cout, cin, dy, wf, None, x, 0, out["dx"], None, st)
        return out
    tr = state["tr"]
    if case["mode"] == "predict":
        tr.predict(state["snap"], NET_R, state["norm8"], state["pred"])
        return dict(pred=state["pred"])
    loss = tr.sample_loss(state["ds"], 0, True, LR)
    net = tr.net
    return dict(loss=loss, out=net.out, dw=list(net.dw), db=list(net.db), w=list(net.w32), b=list(net.b32))


# ------------------------------------------------------------------------------------------------
# Work that no implementation can do without
# ------------------------------------------------------------------------------------------------

def _step_work(c, steps):
    """The state read and written once; per node and stage about 880 flops with UW3 (16 populations x
    7 taps, the velocity-space kernels, equilibrium, update), about 3000 with WENO5; the stabilised
    stages add a real transform and its inverse."""
    n = c["n_theta"] * c["n_phi"]
    word = 8 if c.get("fp64") else 4
    flops = 3.0 * n * steps * (3000 if c.get("weno") else 880)
    if c.get("stab"):
        flops += 3.0 * steps * 2 * 2.5 * n * math.log2(n)
    return {"bytes": 2.0 * n * word * (17 if c.get("fp64") else 18), "flops": flops}


def work(case):
    fam = case["family"]
    if fam == "step":
        return _step_work(case, case["steps"])
    if fam == "ensemble":
        each = [_step_work(m, case["steps"]) for m in _members(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    if fam == "measure":
        n = case["n_theta"] * case["n_phi"]
        return {"bytes": n * (17 * 8.0 if case["fp64"] else 18 * 4.0), "flops": n * (90.0 + 2.5 * math.log2(n))}
    n = case["H"] * case["W"]
    if fam == "layer":
        cin, cout = case["cin"], case["cout"]
        return {"bytes": 2.0 * n * (2 * cin + 2 * cout) + 6.0 * 9 * cin * cout, "flops": 3.0 * 2 * 9 * cin * cout * n}
    train = case["mode"] == "train"
    macs = n * 9.0 * (6 * 64 * 64 + 2 * 16 * 64)
    params = 9 * (6 * 64 * 64 + 2 * 16 * 64)
    return {"bytes": 16.0 * n * 2 + (params * 30.0 if train else params * 2.0),
            "flops": 2.0 * macs * 3 - 2.0 * n * 9 * 16 * 64 if train else 2.0 * macs}


# ------------------------------------------------------------------------------------------------
# The same results in plain 64-bit torch
# ------------------------------------------------------------------------------------------------

def _velocity_set():
    """Gauss-Hermite roots, weights and the derivative kernel K of Sec. 2.3 (Q = 4)."""
    s6 = math.sqrt(6.0)
    v = np.array([-math.sqrt(3 + s6), -math.sqrt(3 - s6), math.sqrt(3 - s6), math.sqrt(3 + s6)])
    he = [np.ones(4), v, v ** 2 - 1, v ** 3 - 3 * v, v ** 4 - 6 * v ** 2 + 3, v ** 5 - 10 * v ** 3 + 15 * v]
    w = 24.0 / he[5] ** 2
    K = -w[:, None] * sum(np.outer(he[k + 1], he[k]) / math.factorial(k) for k in range(4))
    return v, w, K


V, WT, KERNEL = _velocity_set()


def _at(x, k, axis):
    """x at node + k along axis (periodic)."""
    return torch.roll(x, -k, dims=axis)


class _Torus:
    """The semi-discrete system of Sec. 2 on one grid and its SSP-RK3 step, in FP64."""

    def __init__(self, c):
        self.c, self.dt = c, _dt(c)
        nt, ns = c["n_theta"], c["n_phi"]
        self.dth, self.dph = 2 * math.pi / nt, 2 * math.pi / ns
        a = 0.0 if c.get("flat") else c["r"] / c["R"]
        th = torch.arange(nt, device=DEV, dtype=F64)[:, None] * self.dth
        self.J, self.Jp, self.Jm = (1 + a * torch.cos(th + d * self.dth) for d in (0.0, 0.5, -0.5))
        self.gam = torch.zeros_like(th) if c.get("flat") else torch.sin(th) / (c["R"] * self.J)
        self.K = torch.tensor(KERNEL, device=DEV)
        if c.get("stab"):
            h_t = c["r"] * self.dth
            h_p = (c["R"] if c.get("flat") else c["R"] - c["r"]) * self.dph
            m = torch.arange(nt, device=DEV, dtype=F64)[:, None]
            n = torch.arange(ns, device=DEV, dtype=F64)[None, :]
            lap = 4 / h_t ** 2 * torch.sin(math.pi * m / nt) ** 2 + 4 / h_p ** 2 * torch.sin(math.pi * n / ns) ** 2
            self.damp = 1.0 / (1.0 + self.dt * c["M"] * c["kappa"] * lap * lap)

    def laplace(self, x):
        c = self.c
        lt = (self.Jp * (_at(x, 1, 0) - x) - self.Jm * (x - _at(x, -1, 0))) / (c["r"] ** 2 * self.J * self.dth ** 2)
        return lt + (_at(x, 1, 1) - 2 * x + _at(x, -1, 1)) / (c["R"] ** 2 * self.J ** 2 * self.dph ** 2)

    def flux(self, g, axis, positive):
        """Difference of the upwind face values on the two sides of a node."""
        s = 1 if positive else -1
        p = [_at(g, s * k + (0 if positive else 1), axis) for k in (-2, -1, 0, 1, 2)]
        if not self.c.get("weno"):
            F = (-p[1] + 5 * p[2] + 2 * p[3]) / 6
        else:
            q = [(2 * p[0] - 7 * p[1] + 11 * p[2]) / 6, (-p[1] + 5 * p[2] + 2 * p[3]) / 6, (2 * p[2] + 5 * p[3] - p[4]) / 6]
            b = [13 / 12 * (p[0] - 2 * p[1] + p[2]) ** 2 + 0.25 * (p[0] - 4 * p[1] + 3 * p[2]) ** 2,
                 13 / 12 * (p[1] - 2 * p[2] + p[3]) ** 2 + 0.25 * (p[1] - p[3]) ** 2,
                 13 / 12 * (p[2] - 2 * p[3] + p[4]) ** 2 + 0.25 * (3 * p[2] - 4 * p[3] + p[4]) ** 2]
            al = [d / (1e-6 + bk) ** 2 for d, bk in zip((0.1, 0.6, 0.3), b)]
            F = (al[0] * q[0] + al[1] * q[1] + al[2] * q[2]) / (al[0] + al[1] + al[2])
        return F - _at(F, -1, axis)

    def equilibrium(self, n, ut, up, i, j):
        xi, usq = V[i] * ut + V[j] * up, ut * ut + up * up
        return n * WT[i] * WT[j] * (1 + xi + 0.5 * (xi * xi - usq) + xi * (xi * xi - 3 * usq) / 6)

    def moments(self, f):
        n = f.sum(dim=(0, 1))
        ut = sum(V[i] * f[i].sum(dim=0) for i in range(4)) / n
        return n, ut, sum(V[j] * f[:, j].sum(dim=0) for j in range(4)) / n

    def rhs(self, f, phi):
        c, J, gam = self.c, self.J, self.gam
        n, ut, up = self.moments(f)
        mu = -c["A"] * phi * (1 - phi * phi) - c["kappa"] * self.laplace(phi)
        Ft = Fp = torch.zeros_like(phi)
        Lphi = c["M"] * self.laplace(mu)
        if not c.get("diffusive"):
            Ft = -phi * (_at(mu, 1, 0) - _at(mu, -1, 0)) / (2 * c["r"] * self.dth) / n
            Fp = -phi * (_at(mu, 1, 1) - _at(mu, -1, 1)) / (2 * c["R"] * J * self.dph) / n
            gt, gp = J * ut * phi, up * phi
            Lphi = Lphi - (_at(gt, 1, 0) - _at(gt, -1, 0)) / (2 * c["r"] * J * self.dth) \
                - (_at(gp, 1, 1) - _at(gp, -1, 1)) / (2 * c["R"] * J * self.dph)
        Lf = torch.empty_like(f)
        for i in range(4):
            for j in range(4):
                dvt = sum(KERNEL[i, m] * f[m, j] for m in range(4))
                dvp = sum(KERNEL[j, m] * f[i, m] for m in range(4))
                dfv = sum(KERNEL[j, m] * V[m] * f[i, m] for m in range(4))
                Lf[i, j] = (-V[i] * self.flux(J * f[i, j], 0, V[i] > 0) / (c["r"] * J * self.dth)
                            - V[j] * self.flux(f[i, j], 1, V[j] > 0) / (c["R"] * J * self.dph)
                            - Ft * dvt - Fp * dvp + gam * (V[j] ** 2 * dvt - V[i] * dfv)
                            - (f[i, j] - self.equilibrium(n, ut, up, i, j)) / c["tau"])
        Lphi = self.dt * Lphi
        if c.get("stab"):
            Lphi = torch.fft.ifft2(torch.fft.fft2(J * Lphi) * self.damp).real / J
        return self.dt * Lf, Lphi

    def step(self, f, phi):
        a, b = self.rhs(f, phi)
        f1, p1 = f + a, phi + b
        a, b = self.rhs(f1, p1)
        f1, p1 = 0.75 * f + 0.25 * (f1 + a), 0.75 * phi + 0.25 * (p1 + b)
        a, b = self.rhs(f1, p1)
        return f / 3 + 2 / 3 * (f1 + a), phi / 3 + 2 / 3 * (p1 + b)

    def reference_density(self, rho):
        """The area-weighted mean density rounded to 20 significant bits."""
        mean = float((self.J * rho).sum() / (self.J.sum() * rho.shape[1]))
        m, e = math.frexp(mean)
        return math.ldexp(round(math.ldexp(m, 20)), e - 20)

    def run(self, seed, steps):
        nt, ns = self.c["n_theta"], self.c["n_phi"]
        rho, ut, up, phi = _fields(seed, nt, ns)
        f = torch.stack([torch.stack([self.equilibrium(rho, ut, up, i, j) for j in range(4)]) for i in range(4)])
        n0 = self.reference_density(rho)
        for _ in range(steps):
            f, phi = self.step(f, phi)
        g = f - n0 * torch.tensor(np.outer(WT, WT), device=DEV)[:, :, None, None]
        return {"g": g.reshape(16, nt, ns), "phi": phi}

    def measure(self, seed):
        c, (nt, ns) = self.c, (self.c["n_theta"], self.c["n_phi"])
        rho, ut, up, phi = _fields(seed, nt, ns)
        dA = c["r"] * c["R"] * self.J * self.dth * self.dph
        gt = (_at(phi, 1, 0) - _at(phi, -1, 0)) / (2 * c["r"] * self.dth)
        gp = (_at(phi, 1, 1) - _at(phi, -1, 1)) / (2 * c["R"] * self.J * self.dph)
        psi = (0.25 * c["A"] * (1 - phi * phi) ** 2 + 0.5 * c["kappa"] * (gt * gt + gp * gp)) * dA
        totals = torch.stack([(rho * dA).sum(), (phi * dA).sum(), psi.sum(), torch.sqrt(ut * ut + up * up).max()])
        edge = c["R"] * self.Jp * self.dph
        length = ((phi * _at(phi, 1, 1) < 0) * (c["r"] * self.dth)).sum() + ((phi * _at(phi, 1, 0) < 0) * edge).sum()
        S = torch.fft.fft2(phi).abs() ** 2
        m = torch.fft.fftfreq(nt, 1.0 / nt, device=DEV, dtype=F64)[:, None] / c["r"]
        n = torch.fft.fftfreq(ns, 1.0 / ns, device=DEV, dtype=F64)[None, :] / c["R"]
        S[0, 0] = 0.0
        ls = 2 * math.pi * S.sum() / (torch.sqrt(m * m + n * n) * S).sum()
        return dict(totals=totals.cpu().numpy(), interface=float(length), structure=float(ls))


def _shift(x, t):
    """x at (row + t // 3 - 1, column + t % 3 - 1), periodic, of an [H][W][C] tensor."""
    return torch.roll(x, (1 - t // 3, 1 - t % 3), dims=(0, 1))


def _conv(x, w, b=None):
    y = sum(_shift(x, t) @ w[:, t // 3, t % 3, :].T for t in range(9))
    return y if b is None else y + b


def _conv_grads(x, w, dy):
    """(gradient of the input, of the weights, of the bias) of _conv."""
    dx = sum(_shift(dy, 8 - t) @ w[:, t // 3, t % 3, :] for t in range(9))
    flat = dy.reshape(-1, dy.shape[-1])
    dw = torch.stack([flat.T @ _shift(x, t).reshape(-1, x.shape[-1]) for t in range(9)], dim=1)
    return dx, dw.reshape(dy.shape[-1], 3, 3, x.shape[-1]), flat.sum(dim=0)


def _exact_network(case, seed):
    H, W = case["H"], case["W"]
    before, after, weights, biases = _network_inputs(case, seed)
    before, after = before.to(F64), after.to(F64)
    biases = [b.to(F64) for b in biases]
    ws = [w.to(torch.bfloat16).to(F64) for w in weights]
    n_mean, s_phi = before[:, 1].mean(), before[:, 0].square().mean().sqrt()
    one = torch.ones((), device=DEV, dtype=F64)
    sc = torch.stack([s_phi, SCALE_N * one, SCALE_U * one, SCALE_U * one])
    shift = torch.stack([0 * one, n_mean, 0 * one, 0 * one])
    th = torch.arange(H, device=DEV, dtype=F64) * (2 * math.pi / H)
    a = 1.0 / NET_R
    J = 1 + a * torch.cos(th)
    geo = torch.stack([J, torch.sin(th) / J, torch.sin(th), torch.cos(th), 1 / J, a + 0 * J], dim=-1)
    x = torch.cat([((before - shift) / sc).reshape(H, W, 4), geo[:, None, :].expand(H, W, 6),
                   torch.zeros((H, W, 6), device=DEV, dtype=F64)], dim=-1)
    acts = [x]
    for k in range(8):
        y = _conv(acts[-1], ws[k], biases[k])
        acts.append(torch.relu(y) if k < 7 else y)
    out = acts[-1]
    ratio = torch.tensor(RATIOS, device=DEV, dtype=F64) * sc
    if case["mode"] == "predict":
        return dict(pred=before + ratio * out[..., :4].reshape(-1, 4))
    diff = out[..., :4] - ((after - before) / ratio).reshape(H, W, 4)
    dz = torch.zeros_like(out)
    dz[..., :4] = 2 * diff / (4 * H * W)
    dws, dbs = [None] * 8, [None] * 8
    for k in range(7, -1, -1):
        dx, dws[k], dbs[k] = _conv_grads(acts[k], ws[k], dz)
        dz = dx * (acts[k] > 0)
    def adam(p, g):  # first moment zero before the step
        m, v = 0.1 * g, 0.999 * ADAM_V + 0.001 * g * g
        return p - LR * (m / (1 - 0.9 ** (ADAM_T + 1))) / ((v / (1 - 0.999 ** (ADAM_T + 1))).sqrt() + 1e-8)

    return dict(loss=(diff * diff).mean().reshape(1), out=out, dw=dws, db=dbs,
                w=[adam(w.to(F64), g) for w, g in zip(weights, dws)], b=[adam(b, g) for b, g in zip(biases, dbs)])


def exact(case, seed):
    fam = case["family"]
    if fam == "step":
        return _Torus(case).run(seed, case["steps"])
    if fam == "ensemble":
        return [_Torus(m).run(seed + 1000 * k, case["steps"]) for k, m in enumerate(_members(case))]
    if fam == "measure":
        return _Torus(case).measure(seed)
    if fam == "layer":
        x, dy, w, b = (t.to(F64) for t in _layer_inputs(case, seed))
        dx, dw, db = _conv_grads(x, w, dy)
        return dict(y=torch.relu(_conv(x, w, b)), dx=dx * (x > 0), dw=dw, db=db)
    return _exact_network(case, seed)
