"""The workloads of this framework as performance cases.

A user of the library does a handful of things: advance one lattice (short and long
runs, every size from a microchannel to the two-bubble channel, FP32 or FP16
storage), run one to steady state, advance an ensemble, read out the state of a run,
and train or apply the warm-start network.  Each case below is one of them, through
the calls that program makes: paper_2306_11320_gb300.tpflbm, .unet, .warmstart and the
two C ABIs behind them.

A case is a dict of plain values; "kind" selects the workload:

  run       Lattice.init, step(steps), fields(device=True): a simulation from given fields
  steady    init, then one chunk of the time-to-steady loop: step(steps), residual
  ensemble  Batch.step(steps), then every member's fields into device memory
  monitor   diagnostics, bubbles and fields of a state: what a run records between chunks
  conv      one 3x3 layer of the network, forward and backward (tpfnet_*)
  predict   UNet.forward on a batch of channels (the trained network)
  train     UNet.train_step

`exact` restates the method in 64 bits with plain torch: the lattice Boltzmann step
(class Ref64) and the network (torch.nn.functional).
"""
import ctypes as C
import math

import numpy as np
import torch

from paper_2306_11320_gb300 import warmstart as WS
from paper_2306_11320_gb300 import workloads as WL
from paper_2306_11320_gb300.tpflbm import Batch, Lattice
from paper_2306_11320_gb300.unet import net_library

FIELDS = ("phi", "ux", "uy", "p", "T")
PLANE_BYTES = (232, 172)  # populations, (phi u) and FP16 records of one node, read and written once


def listed():
    return [
        # the heated microchannel of Sec. 4.1 (20k steps in full): the smallest lattice
        # in use, where a step is a few microseconds of launch and latency
        dict(name="microchannel_128x32", kind="run", flow="microchannel", nx=128, ny=32, storage=0, steps=1000),
        # the warm-start channel's time-to-steady loop, of which a run has hundreds of chunks
        dict(name="steady_512x128", kind="steady", flow="microchannel", nx=512, ny=128, storage=0, steps=1000),
        # the migrating drop of Sec. 4.2, periodic in x
        dict(name="drop_256x1024", kind="run", flow="drop", nx=256, ny=1024, storage=0, steps=200),
        # the two bubbles of Sec. 4.3, inlet and outflow: the largest single lattice
        dict(name="bubbles_2048x512", kind="run", flow="bubbles", nx=2048, ny=512, storage=0, steps=100),
        # the same with float16 deviation storage
        dict(name="bubbles_2048x512_f16", kind="run", flow="bubbles", nx=2048, ny=512, storage=1, steps=100),
        # odd rows (no 16-byte multiple): a two-phase state between walls
        dict(name="ragged_331x117", kind="run", flow="random", nx=331, ny=117, storage=0, steps=200),
        # the parameter sweep: 256 lattices of uneven sizes
        dict(name="ensemble_256", kind="ensemble", n=256, storage=0, steps=100),
        # a quarter of it with float16 storage
        dict(name="ensemble_64_f16", kind="ensemble", n=64, storage=1, steps=100),
        # reading out the two-bubble channel: conserved sums, bubbles, fields
        dict(name="monitor_2048x512", kind="monitor", flow="bubbles", nx=2048, ny=512, storage=0),
        # a layer of the network's second level, forward and backward
        dict(name="conv_4x64x256_64", kind="conv", N=4, H=64, W=256, cin=64, cout=64),
        # the network's prediction for one channel (every warm start)
        dict(name="predict_1", kind="predict", n=1),
        # one training step at the batch size the network is trained with
        dict(name="train_4", kind="train", n=4),
    ]


def _logu(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["run"] * 9 + ["steady"] * 2 + ["ensemble"] * 2 + ["monitor"] * 2 + ["conv"] * 3 +
                      ["predict", "train"])
    if kind in ("run", "steady", "monitor"):
        # 2^11 to 2^20 nodes, aspect 1/4 to 8; a third of the rows odd
        nodes = _logu(rng, 2 ** 11, 2 ** 20)
        aspect = _logu(rng, 0.25, 8.0)
        nx = max(24, int(round(math.sqrt(nodes * aspect))))
        ny = max(16, int(round(nodes / nx)))
        if rng.random() < 0.67:
            nx = -(-nx // 8) * 8
        nx, ny = min(nx, 2048), min(ny, 1024)
        flow = rng.choice(["microchannel", "drop", "bubbles", "random"])
        if kind == "steady":
            flow = "microchannel"
        if kind == "monitor":
            return dict(kind=kind, flow=flow, nx=nx, ny=ny, storage=rng.randrange(2))
        # no more node updates than the two-bubble case
        steps = int(min(_logu(rng, 10, 1000), 100 * 2 ** 20 / (nx * ny)))
        case = dict(kind=kind, flow=flow, nx=nx, ny=ny, storage=rng.randrange(2), steps=max(10, steps))
        if kind == "run" and rng.random() < 0.15:
            case["collision"] = 1  # two-relaxation-time
        if kind == "run" and rng.random() < 0.15:
            case["normal_law"] = 1  # local interface normal
        return case
    if kind == "ensemble":
        return dict(kind=kind, n=int(round(_logu(rng, 4, 256))), storage=rng.randrange(2),
                    steps=rng.randrange(10, 100))
    if kind == "conv":
        # the network's levels, other pixel widths, wider and narrower layers
        lvl = rng.randrange(4)
        W, H = 512 >> lvl, 128 >> lvl
        if rng.random() < 0.3:
            W, H = rng.randrange(9, W + 1), rng.randrange(8, H + 1)
        ch = 32 << lvl
        cin = rng.choice([ch, ch, 3 * ch, max(32, ch // 2)])
        return dict(kind=kind, N=rng.randrange(1, 9), H=H, W=W, cin=cin, cout=ch)
    if kind == "predict":
        return dict(kind=kind, n=rng.randrange(1, 21))
    return dict(kind=kind, n=rng.randrange(1, 9))


# ------------------------------------------------------------------ inputs

def _flow(case, rng):
    """(params, fields) of a lattice: the workload's own initial state, placed and stirred
    by the seed (a smooth flow of the size the workload develops, vanishing at the walls)."""
    nx, ny = case["nx"], case["ny"]
    if case["flow"] == "microchannel":
        p, f, _ = WL.microchannel(nx=nx, ny=ny, lam_r=float(rng.uniform(0.2, 5.0)), k=int(rng.integers(1, 5)))
    elif case["flow"] == "drop":
        R = max(4.0, min(nx, ny) / 8.0)
        p, f, _ = WL.drop_migration(nx=nx, ny=ny, R=R, Ma=float(rng.choice([0.1, 10.0])))
        shift = int(rng.integers(0, nx))  # periodic in x
        f = {k: np.roll(v, shift, axis=1) for k, v in f.items()}
    elif case["flow"] == "bubbles":
        s = min(nx / 2048.0, ny / 512.0)
        p, f, _ = WL.bubbles(nx=nx, ny=ny, R1=max(4.0, 40.0 * s), R2=max(3.0, 32.0 * s), spacing=max(20.0, 150.0 * s),
                             lead_x_frac=float(rng.uniform(0.6, 0.9)))
    else:
        p, f, _ = WL.random_state(nx, ny, seed=int(rng.integers(1 << 30)), bc_x=0, bc_y=0, sigma_law=1, amp_u=0.0)
        # temperature differences independent of the length (sigma is quadratic in them)
        f["T"] = f["T"] + (0.4 / nx - 0.01) * np.arange(nx)
        p.update(T_bot_slope=0.2 / nx, T_top_slope=-0.1 / nx)
    p.update(collision=case.get("collision", 0), normal_law=case.get("normal_law", 0), trt_lambda=0.25)
    x, y = (np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny
    f = dict(f)
    # u = (d psi / dy, -d psi / dx) of a stream function flat at the walls
    for m in range(1, 4):
        a, ph = 2e-3 * min(nx, ny) * rng.normal() / (2 * math.pi * m), rng.uniform(0, 2 * math.pi)
        f["ux"] = f["ux"] + np.outer(2 * math.pi / ny * np.sin(2 * math.pi * y), a * np.cos(2 * math.pi * m * x + ph))
        f["uy"] = f["uy"] + np.outer(1 - np.cos(2 * math.pi * y),
                                     a * 2 * math.pi * m / nx * np.sin(2 * math.pi * m * x + ph))
        f["p"] = f["p"] + 1e-4 * rng.normal() * np.cos(2 * math.pi * m * x + ph)[None]
    return p, {k: f[k].astype(np.float32) for k in FIELDS}


def _members(case, rng):
    """The parameter sweep's lattices and initial fields."""
    out = []
    for p, f, m in WL.ensemble(n=case["n"], seed=0):
        nx, ny = m["nx"], m["ny"]
        x, y = (np.arange(nx, dtype=np.float32) + 0.5) / nx, (np.arange(ny, dtype=np.float32) + 0.5) / ny
        f = {k: f[k].astype(np.float32) for k in FIELDS}
        a, ph = 1e-3 * min(nx, ny) * rng.normal() / (2 * math.pi), rng.uniform(0, 2 * math.pi)
        f["ux"] += np.outer(2 * math.pi / ny * np.sin(2 * math.pi * y),
                            a * np.cos(2 * math.pi * x + ph)).astype(np.float32)
        f["uy"] += np.outer(1 - np.cos(2 * math.pi * y),
                            a * 2 * math.pi / nx * np.sin(2 * math.pi * x + ph)).astype(np.float32)
        f["p"] += (1e-4 * rng.normal() * np.cos(2 * math.pi * x + ph))[None].astype(np.float32)
        out.append((nx, ny, p, f))
    return out


def _ptr(t):
    return C.c_void_p(t.data_ptr())


def _net_targets(n, seed):
    """Smooth normalised target fields, as the channels' departures from their cold start are."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    t = torch.randn((n, len(WS.OUT_FIELDS), WS.NY // 8, WS.NX // 8), device="cuda", generator=g)
    t = torch.nn.functional.interpolate(t, scale_factor=8, mode="bilinear")
    return t.permute(0, 2, 3, 1).contiguous()


def _net_maps(n, seed):
    return torch.from_numpy(np.stack([WS.features(i) for i in WS.sample_instances(n, seed)])).cuda()


def _conv_inputs(case, seed):
    N, H, W, ci, co = case["N"], case["H"], case["W"], case["cin"], case["cout"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    rnd = lambda *s: torch.randn(s, device="cuda", generator=g)  # noqa: E731
    x = rnd(N, H, W, ci).relu().to(torch.bfloat16)  # an activation: half of it zero
    wt = (rnd(9, co, ci) * math.sqrt(2.0 / (9 * ci))).to(torch.bfloat16)
    b = 0.01 * rnd(co)
    dy = (1e-3 * rnd(N, H, W, co)).to(torch.bfloat16)
    return x, wt, b, dy


# ----------------------------------------------------------- the cases' passes

def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind in ("run", "steady", "monitor"):
        p, f = _flow(case, rng)
        # a stream of the lattice's own, as the warm-start comparison and the benchmark use
        lat = Lattice(case["nx"], case["ny"], p, storage=case["storage"], stream=torch.cuda.Stream())
        dev = {k: torch.from_numpy(v).cuda() for k, v in f.items()}
        torch.cuda.synchronize()
        if kind == "monitor":
            lat.init(**dev)
        return dict(kind=kind, lat=lat, fields=dev, steps=case.get("steps", 0))
    if kind == "ensemble":
        mem = _members(case, rng)
        b = Batch([(nx, ny, p) for nx, ny, p, _ in mem], storage=case["storage"])
        b.tune(steps=10)  # once per ensemble
        offs, tot = [], 0
        for k, (nx, ny, _, f) in enumerate(mem):
            b.init(k, **f)
            offs.append(tot)
            tot += nx * ny
        out = torch.empty((5, tot), device="cuda")
        return dict(kind=kind, batch=b, offs=offs, out=out, steps=case["steps"])
    if kind == "conv":
        x, wt, b, dy = _conv_inputs(case, seed)
        st = dict(kind=kind, lib=net_library(), x=x, wt=wt, b=b, dy=dy, dims=tuple(case[k] for k in "NHW"),
                  cin=case["cin"], cout=case["cout"], y=torch.empty_like(dy), dz=torch.empty_like(dy),
                  dx=torch.empty_like(x), dw=torch.empty(wt.shape, device="cuda"), db=torch.empty_like(b),
                  wflip=torch.empty_like(wt))
        return st
    if kind == "predict":
        net, _, _ = WS.load(WS.WEIGHTS)
        return dict(kind=kind, net=net, x=WS.pack_inputs(net, _net_maps(case["n"], seed)))
    net = WS.make_net(seed=seed)
    return dict(kind=kind, net=net, x=WS.pack_inputs(net, _net_maps(case["n"], seed)),
                y=_net_targets(case["n"], seed))


def run(state):
    kind = state["kind"]
    if kind == "run":
        lat = state["lat"]
        lat.init(**state["fields"])
        lat.step(state["steps"])
        return lat.fields(device=True)
    if kind == "steady":
        lat = state["lat"]
        lat.init(**state["fields"])
        lat.residual(WS.DT_SCALE)  # the loop's first snapshot
        lat.step(state["steps"])
        ru, rT, k = lat.residual(WS.DT_SCALE)
        return dict(lat.fields(device=True), converged=max(ru, rT) < 1e-8, window=k)
    if kind == "ensemble":
        b, out = state["batch"], state["out"]
        b.step(state["steps"])
        for k, o in enumerate(state["offs"]):
            rc = b.lib.tpflbm_batch_get_fields(b.h, k, *[C.c_void_p(out.data_ptr() + 4 * (j * out.shape[1] + o))
                                                         for j in range(5)])
            b._check(rc)
        return dict(zip(FIELDS, out))
    if kind == "monitor":
        lat = state["lat"]
        d = lat.diagnostics()
        rows = lat.bubbles()
        return dict(lat.fields(device=True), sums=np.array([d[k] for k in ("sum_phi", "sum_rcpT", "sum_T")]),
                    nonfinite=d["nonfinite"], regions=len(rows),
                    bubbles=np.array([[r[k] for k in Lattice.BUBBLE_KEYS] for r in rows]))
    if kind == "conv":
        s, lib = state, state["lib"]
        (N, H, W), ci, co = s["dims"], s["cin"], s["cout"]
        cs = C.c_void_p(torch.cuda.current_stream().cuda_stream)
        s["dw"].zero_()
        s["db"].zero_()
        s["dz"].copy_(s["dy"])  # the mask below works in place
        rc = lib.tpfnet_conv3x3(_ptr(s["x"]), N, H, W, ci, _ptr(s["wt"]), _ptr(s["b"]), co, 1, _ptr(s["y"]), cs)
        rc |= lib.tpfnet_relu_mask(_ptr(s["dz"]), _ptr(s["y"]), s["dz"].numel(), cs)
        rc |= lib.tpfnet_conv3x3_wgrad(_ptr(s["x"]), _ptr(s["dz"]), N, H, W, ci, co, _ptr(s["dw"]), _ptr(s["db"]), cs)
        rc |= lib.tpfnet_conv3x3_dgrad(_ptr(s["dz"]), N, H, W, co, _ptr(s["wt"]), ci, _ptr(s["wflip"]), _ptr(s["dx"]),
                                       cs)
        if rc:
            raise RuntimeError("tpfnet call failed")
        return [s["y"], s["dx"], s["dw"], s["db"]]
    if kind == "predict":
        return state["net"].forward(state["x"])
    net = state["net"]
    loss = net.train_step(state["x"], state["y"])
    return dict(loss=loss, grads=[net.G[k] for k in sorted(net.G)], params=[net.P[k] for k in sorted(net.P)])


# -------------------------------------------------------------------- work

def _ensemble_nodes(n):
    """Nodes of the parameter sweep (sizes as workloads.ensemble draws them)."""
    return sum(m["nx"] * m["ny"] for _, _, m in WL.ensemble(n=n, seed=0))


def _net_layers():
    """(Cin, Cout, level) of the network's 3x3 layers."""
    c = (WS.C_IN,) + WS.CHANNELS
    enc = [(c[0], c[1], 0), (c[1], c[1], 0), (c[1], c[2], 1), (c[2], c[2], 1), (c[2], c[3], 2), (c[3], c[3], 2),
           (c[3], c[4], 3), (c[4], c[4], 3)]
    dec = [(c[4] + c[3], c[3], 2), (c[3], c[3], 2), (c[3] + c[2], c[2], 1), (c[2], c[2], 1), (c[2] + c[1], c[1], 0),
           (c[1], c[1], 0)]
    return enc + dec


def work(case):
    """Bytes and floating-point operations a pass cannot do without.  A lattice step reads
    and writes its state once (232 bytes per node, 172 with float16 storage) and does about
    300 operations per node; initialising and reading out move the five fields."""
    kind = case["kind"]
    if kind in ("run", "steady"):
        n = case["nx"] * case["ny"]
        return dict(bytes=n * (case["steps"] * PLANE_BYTES[case["storage"]] + 40), flops=n * case["steps"] * 300)
    if kind == "monitor":
        n = case["nx"] * case["ny"]
        return dict(bytes=n * (PLANE_BYTES[case["storage"]] // 2 + 20), flops=n * 300)
    if kind == "ensemble":
        n = _ensemble_nodes(case["n"])
        return dict(bytes=n * (case["steps"] * PLANE_BYTES[case["storage"]] + 20), flops=n * case["steps"] * 300)
    if kind == "conv":
        px = case["N"] * case["H"] * case["W"]
        ci, co = case["cin"], case["cout"]
        # x, dy in; y, dx out (bf16); weights in, their gradients out
        return dict(bytes=px * 4 * (ci + co) + 9 * ci * co * 6, flops=3 * 2 * px * 9 * ci * co)
    px = case["n"] * WS.NX * WS.NY
    flops = sum(2 * (px >> (2 * lvl)) * 9 * a * b for a, b, lvl in _net_layers())
    weights = sum(9 * a * b for a, b, _ in _net_layers())
    if kind == "predict":
        return dict(bytes=px * (2 * 32 + 4 * 5) + 2 * weights, flops=flops)
    # training: the activations are written forward and read backward, as their gradients are
    acts = sum((px >> (2 * lvl)) * b for _, b, lvl in _net_layers())
    return dict(bytes=8 * acts + px * 84 + 28 * weights, flops=3 * flops)


# ----------------------------------------------------- the method in 64 bits

CX, CY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
WQ = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


class Ref64:
    """The three coupled lattice Boltzmann equations in float64 (plain torch, whole-array
    operations, pull streaming)."""

    def __init__(self, nx, ny, p, fields):
        kw = dict(dtype=torch.float64, device="cuda")
        self.p, self.nx, self.ny = p, nx, ny
        self.cx = torch.tensor(CX, **kw).view(9, 1, 1)
        self.cy = torch.tensor(CY, **kw).view(9, 1, 1)
        self.w = torch.tensor(WQ, **kw).view(9, 1, 1)
        self.x = torch.arange(nx, **kw)
        self.y = torch.arange(ny, **kw)
        f = {k: torch.as_tensor(v, **kw) for k, v in fields.items()}
        rho = self.prop("rho", f["phi"].clamp(-1, 1))
        self.f, self.g, self.h = self.equilibria(f["phi"], rho, f["ux"], f["uy"], f["p"], f["T"])
        self.pu = (f["phi"] * f["ux"], f["phi"] * f["uy"])

    def prop(self, name, pc):
        lo, hi = (self.p[name + "_l"], self.p[name + "_h"]) if name != "rcp" else (
            self.p["rho_l"] * self.p["cp_l"], self.p["rho_h"] * self.p["cp_h"])
        return 0.5 * (lo + hi) + 0.5 * (hi - lo) * pc

    def equilibria(self, phi, rho, ux, uy, p, T):
        w = self.w
        cu = self.cx * ux + self.cy * uy
        s = w * (3 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy))
        feq, heq, geq = w * phi * (1 + 3 * cu), w * T, 3 * p * w + rho * s
        geq[0] -= 3 * p
        return feq, geq, heq

    def wall(self, top, x):
        p = self.p
        if top:
            return p["T_top"] + p["T_top_slope"] * x
        return p["T_bot"] + p["T_bot_amp"] * torch.cos(2 * math.pi * p["T_bot_k"] * x / self.nx) + p["T_bot_slope"] * x

    def padded(self, phi, T):
        p = self.p
        if p["bc_x"] == 0:
            px = [torch.cat((a[:, -1:], a, a[:, :1]), 1) for a in (phi, T)]
        else:
            px = [torch.cat((phi[:, :1], phi, phi[:, -1:]), 1),
                  torch.cat((2 * p["T_in"] - T[:, :1], T, T[:, -1:]), 1)]
        if p["bc_y"] == 1:
            return [torch.cat((a[-1:], a, a[:1]), 0) for a in px]
        xg = torch.arange(-1, self.nx + 1, dtype=torch.float64, device="cuda")
        a, t = px
        return [torch.cat((a[:1], a, a[-1:]), 0),
                torch.cat((2 * self.wall(False, xg)[None] - t[:1], t, 2 * self.wall(True, xg)[None] - t[-1:]), 0)]

    def grad(self, q):
        """isotropic gradient of a padded field"""
        a = lambda i: q[1 + CY[i]:1 + CY[i] + self.ny, 1 + CX[i]:1 + CX[i] + self.nx]  # noqa: E731
        return (3 * sum(WQ[i] * CX[i] * a(i) for i in range(1, 9) if CX[i]),
                3 * sum(WQ[i] * CY[i] * a(i) for i in range(1, 9) if CY[i]),
                6 * sum(WQ[i] * (a(i) - a(0)) for i in range(1, 9)))

    def macro(self):
        p = self.p
        m = dict(phi=self.f.sum(0), T=self.h.sum(0))
        phi, T = m["phi"], m["T"]
        qp, qt = self.padded(phi, T)
        gx, gy, lap = self.grad(qp)
        tx, ty, _ = self.grad(qt)
        pc = phi.clamp(-1, 1)
        m["rho"], m["rcp"] = self.prop("rho", pc), self.prop("rcp", pc)
        m["og"] = 1 / (3 * self.prop("mu", pc) / m["rho"] + 0.5)
        m["oh"] = 1 / (3 * self.prop("lambda", pc) + 0.5)
        dT = T - p["T_ref"]
        if p["sigma_law"] == 1:
            sig, ds = p["sigma_ref"] + 0.5 * p["sigma_TT"] * dT * dT, p["sigma_TT"] * dT
        else:
            sig, ds = p["sigma_ref"] + p["sigma_T"] * dT, p["sigma_T"]
        W = p["W"]
        mu = phi ** 3 - phi - W * W * lap
        sx, sy = ds * tx, ds * ty
        g2, sp = gx * gx + gy * gy, sx * gx + sy * gy
        k = 3 * math.sqrt(2) * W / 4
        m["Fx"] = k * (g2 * sx - sp * gx + sig * mu * gx / (W * W)) + p["Gx"]
        m["Fy"] = k * (g2 * sy - sp * gy + sig * mu * gy / (W * W)) + p["Gy"]
        ux = m["ux"] = ((self.cx * self.g).sum(0) + 0.5 * m["Fx"]) / m["rho"]
        uy = m["uy"] = ((self.cy * self.g).sum(0) + 0.5 * m["Fy"]) / m["rho"]
        dr = 0.5 * (p["rho_h"] - p["rho_l"])
        m["rx"], m["ry"] = dr * gx, dr * gy
        uu = ux * ux + uy * uy
        m["p"] = (1 / 3) / (5 / 9) * (self.g[1:].sum(0) + 0.5 * (ux * m["rx"] + uy * m["ry"]) - m["rho"] * uu * 2 / 3)
        m["ax"], m["ay"] = phi * ux - self.pu[0], phi * uy - self.pu[1]
        tau = 3 * p["M_phi"] + 0.5
        nx, ny, thr = gx, gy, 1e-10
        if p.get("normal_law", 0) == 1:
            nx = -((self.cx * self.f).sum(0) - phi * ux + 0.5 * m["ax"])
            ny = -((self.cy * self.f).sum(0) - phi * uy + 0.5 * m["ay"])
            thr = 1e-10 * tau / 3
        nn = torch.sqrt(nx * nx + ny * ny)
        inv = torch.where(nn > thr, 1 / nn.clamp_min(1e-300), torch.zeros_like(nn))
        m["nx"], m["ny"] = nx * inv, ny * inv
        m["Fh"] = 3 * m["rcp"] * m["oh"] * (ux * (self.cx * self.h).sum(0) + uy * (self.cy * self.h).sum(0))
        return m

    def fields(self):
        m = self.macro()
        return {k: m[k] for k in FIELDS}

    def step(self):
        p, w, cx, cy = self.p, self.w, self.cx, self.cy
        m = self.macro()
        phi, T, rho, ux, uy = m["phi"], m["T"], m["rho"], m["ux"], m["uy"]
        feq, geq, heq = self.equilibria(phi, rho, ux, uy, m["p"], T)
        op = 1 / (3 * p["M_phi"] + 0.5)
        th = (1 - phi * phi) / (math.sqrt(2) * p["W"])
        f = self.f + op * (feq - self.f) + (1 - 0.5 * op) * w * (cx * (3 * m["ax"] + m["nx"] * th) +
                                                                 cy * (3 * m["ay"] + m["ny"] * th))
        G = w * (3 * (cx * m["Fx"] + cy * m["Fy"]) + 3 * (cx * ux + cy * uy) * (cx * m["rx"] + cy * m["ry"]))
        if p.get("collision", 0) == 1:
            o = list(OPP)
            ev = lambda q: 0.5 * (q + q[o])  # noqa: E731
            od = lambda q: 0.5 * (q - q[o])  # noqa: E731
            lam = p["trt_lambda"]
            other = lambda om: 1 / (0.5 + lam / (1 / om - 0.5))  # noqa: E731
            gp, gm = m["og"], other(m["og"])
            hm, hp = m["oh"], other(m["oh"])
            g = self.g + gp * ev(geq - self.g) + gm * od(geq - self.g) + (1 - 0.5 * gp) * ev(G) + (1 - 0.5 * gm) * od(G)
            h = self.h + hp * ev(heq - self.h) + hm * od(heq - self.h) + w * m["Fh"]
        else:
            g = self.g + m["og"] * (geq - self.g) + (1 - 0.5 * m["og"]) * G
            h = self.h + m["oh"] * (heq - self.h) + w * m["Fh"]
        nf, ng, nh = (torch.empty_like(q) for q in (f, g, h))
        for i in range(9):
            for new, q in ((nf, f), (ng, g), (nh, h)):
                new[i] = torch.roll(q[i], (CY[i], CX[i]), (0, 1))
            o = OPP[i]
            if p["bc_x"] == 1 and CX[i] == 1:  # inlet
                u = 6 * p["u_ave"] * (yc := self.y + 0.5 - 0.5 * CY[i]) * (self.ny - yc) / self.ny ** 2
                nf[i][:, 0] = f[o][:, 0] + 6 * WQ[i] * p["phi_in"] * u
                ng[i][:, 0] = g[o][:, 0] + 6 * WQ[i] * rho[:, 0] * u
                nh[i][:, 0] = -h[o][:, 0] + 2 * WQ[i] * p["T_in"]
            if p["bc_x"] == 1 and CX[i] == -1:  # outflow
                cu = (CX[i] * ux + CY[i] * uy)[:, -1]
                uu = (ux * ux + uy * uy)[:, -1]
                ng[i][:, -1] = -g[o][:, -1] + 2 * WQ[i] * (3 * p["p_out"] + rho[:, -1] * (4.5 * cu * cu - 1.5 * uu))
                nf[i][:, -1] = torch.roll(f[i][:, -1], CY[i], 0)
                nh[i][:, -1] = torch.roll(h[i][:, -1], CY[i], 0)
            if p["bc_y"] == 0 and CY[i]:  # walls
                r = 0 if CY[i] == 1 else -1
                nf[i][r], ng[i][r] = f[o][r], g[o][r]
                nh[i][r] = -h[o][r] + 2 * WQ[i] * self.wall(CY[i] == -1, self.x - 0.5 * CX[i])
        nh = self.h + (nh - self.h) / m["rcp"]
        self.f, self.g, self.h = nf, ng, nh
        self.pu = (phi * ux, phi * uy)


def _net64(params, x, grads=False):
    """The network in float64 on NCHW input; params: the masters' float64 copies."""
    import torch.nn.functional as F

    def conv(name, v, relu=True):
        W = params[name + ".W"]
        k = W.view(3, 3, W.shape[1], W.shape[2]).permute(2, 3, 0, 1)
        v = F.conv2d(v, k[:, :v.shape[1]], params[name + ".b"], padding=1)
        return F.relu(v) if relu else v

    two = lambda a, b, v: conv(b, conv(a, v))  # noqa: E731
    e0 = two("e0a", "e0b", x)
    e1 = two("e1a", "e1b", F.avg_pool2d(e0, 2))
    e2 = two("e2a", "e2b", F.avg_pool2d(e1, 2))
    d = two("b_a", "b_b", F.avg_pool2d(e2, 2))
    for lvl, skip in ((2, e2), (1, e1), (0, e0)):
        up = d.repeat_interleave(2, 2).repeat_interleave(2, 3)
        d = two("d%da" % lvl, "d%db" % lvl, torch.cat((up, skip), 1))
    return torch.einsum("nchw,co->nhwo", d, params["head.W"]) + params["head.b"]


def exact(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind in ("run", "steady", "monitor"):
        p, f = _flow(case, rng)
        steps = case.get("steps", 0)
        # a float64 step is about 250 whole-array operations
        if steps * (4e-3 + case["nx"] * case["ny"] * 2e-8) > 15:
            return None
        ref = Ref64(case["nx"], case["ny"], p, f)
        for _ in range(steps):
            ref.step()
        out = ref.fields()
        if kind == "steady":
            out.update(converged=None, window=None)
        if kind == "monitor":
            m = ref.macro()
            sums = torch.stack([m["phi"].sum(), (m["rcp"] * m["T"]).sum(), m["T"].sum()])
            out.update(sums=sums, nonfinite=None, regions=None, bubbles=None)
        return out
    if kind == "ensemble":
        if case["n"] * case["steps"] * 5e-3 > 15:
            return None
        refs = [Ref64(nx, ny, p, f) for nx, ny, p, f in _members(case, rng)]
        for r in refs:
            for _ in range(case["steps"]):
                r.step()
        fl = [r.fields() for r in refs]
        return {k: torch.cat([a[k].reshape(-1) for a in fl]) for k in FIELDS}
    if kind == "conv":
        import torch.nn.functional as F

        x, wt, b, dy = (t.double() for t in _conv_inputs(case, seed))
        ci, co = case["cin"], case["cout"]
        k = wt.view(3, 3, co, ci).permute(2, 3, 0, 1).contiguous().requires_grad_()
        xi = x.permute(0, 3, 1, 2).contiguous().requires_grad_()
        bi = b.requires_grad_()
        y = F.relu(F.conv2d(xi, k, bi, padding=1))
        y.backward(dy.permute(0, 3, 1, 2))
        return [y.detach().permute(0, 2, 3, 1).contiguous(), xi.grad.permute(0, 2, 3, 1).contiguous(),
                k.grad.permute(2, 3, 0, 1).reshape(9, co, ci).contiguous(), bi.grad]
    if kind == "predict":
        d = np.load(WS.WEIGHTS, allow_pickle=False)
        par = {}
        for key in d.files:
            if key.endswith(":bf16"):
                par[key[:-5]] = torch.from_numpy((d[key].astype(np.uint32) << 16).view(np.float32)).cuda().double()
            elif key != "__norm__":
                par[key] = torch.from_numpy(d[key]).cuda().double()
        x = _net_maps(case["n"], seed).to(torch.bfloat16).double()
        return torch.cat([_net64(par, x[i:i + 1]) for i in range(case["n"])])
    net = WS.make_net(seed=seed)  # its initial weights only
    # the convolutions use the bfloat16 copies of the weights
    par = {k: (net.P[k].bfloat16() if net.Pb[k] is not None else net.P[k]).double().requires_grad_() for k in net.P}
    x = _net_maps(case["n"], seed).to(torch.bfloat16).double()
    y = _net_targets(case["n"], seed).double()
    loss = torch.zeros((), dtype=torch.float64, device="cuda")
    for i in range(case["n"]):
        part = ((_net64(par, x[i:i + 1]) - y[i:i + 1]) ** 2).sum() / y.numel()
        part.backward()
        loss += part.detach()
    g = {k: v.grad for k, v in par.items()}
    # Adam's first step on the float32 masters
    new = {k: net.P[k].double() - 1e-3 * g[k] / (g[k].abs() + 1e-8) for k in g}
    return dict(loss=loss, grads=[g[k] for k in sorted(g)], params=[new[k] for k in sorted(new)])
