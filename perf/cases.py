"""The work a user has this framework do, as measurable cases.

Every case is one pass through the public entry points of the Python binding:
a solver (``mdf.Solver``) stepped and read back, a batch of problems
(``mdf.Batch``) stepped and read back, or the warm-start network
(``warmstart.Net``) applied or trained.  Sizes and parameters are those of the
repository's benchmark, tests and training program.

A time step reads the state and writes it, so ``work`` counts, for every step
of a pass, the state once in and once out (with the force, metric and alpha = 0
planes the step reads) and, once per pass, the copy the caller asks for.

``exact`` restates the method (arXiv:2306.08216, Sec. 2.2 Steps (1)-(4)) and
the network in plain FP64 torch, from the paper and the network's
specification alone.
"""
import math
import os

import numpy as np
import torch

from paper_2306_08216_gb300 import mdf
from paper_2306_08216_gb300 import warmstart as WS

U_LID = 0.1
WEIGHTS = os.path.join(WS.WEIGHTS_DIR, "warmstart_cavity_R128.npy")
TWO_PI = 2.0 * math.pi
CHECKED = 16  # problems of a sweep that exact() marches
SIDES = (65, 129, 257, 513)  # grid sides of the cavity sweep


def listed():
    return [
        # A time-dependent force is set before every step of a small periodic
        # grid, and the velocity and pressure are read after ten steps: the
        # smallest calls a user makes, all latency and launches.
        dict(name="forced_64_call_by_call", kind="solver", flow="periodic", nx=64, ny=64, fluid="newton",
             storage="fp32", rho0=False, force="time", nu=0.01, u0=0.1, steps=1, calls=10, read="fields"),
        # Decaying Taylor-Green vortex, 64^2 for 1000 steps: the accuracy
        # configuration, a small problem stepped for long.
        dict(name="taylor_green_64", kind="solver", flow="periodic", nx=64, ny=64, fluid="newton", storage="fp32",
             rho0=False, force="none", nu=0.01, u0=0.01, steps=1000, calls=1, read="state"),
        # Lid-driven cavity at Re 1000 marched towards its steady state: 100
        # steps between residual checks.
        dict(name="cavity_257", kind="solver", flow="cavity", nx=257, ny=257, fluid="newton", storage="fp32",
             rho0=False, force="none", nu=1e-4, u0=U_LID, steps=100, calls=1, read="residual"),
        # Channel flow between tanh-stretched walls driven by a force field,
        # sides that are no multiple of any tile.
        dict(name="channel_1000x385", kind="solver", flow="channel", nx=1000, ny=385, fluid="newton",
             storage="fp32", rho0=False, force="field", nu=1e-3, u0=0.1, steps=48, calls=1, read="state"),
        # Power-law cavity on the body-fitted trapezoid grid, 513^2.
        dict(name="trapezoid_513", kind="solver", flow="trapezoid", nx=513, ny=513, fluid="power", storage="fp32",
             rho0=False, force="none", re=400.0, n=0.7, u0=U_LID, steps=48, calls=1, read="state"),
        # Taylor-Green on 4096^2: the bandwidth run.
        dict(name="taylor_green_4096", kind="solver", flow="periodic", nx=4096, ny=4096, fluid="newton",
             storage="fp32", rho0=False, force="none", nu=0.01, u0=0.01, steps=20, calls=1, read="state"),
        # Forced periodic flow kept in BF16 deviations, twice the nodes per
        # byte, on a grid that is not square.
        dict(name="forced_2048x1536_bf16", kind="solver", flow="periodic", nx=2048, ny=1536, fluid="newton",
             storage="bf16", rho0=False, force="field", nu=0.01, u0=0.1, steps=32, calls=1, read="state"),
        # The density-like distribution evolved beside the velocity.
        dict(name="density_2048", kind="solver", flow="periodic", nx=2048, ny=2048, fluid="newton", storage="fp32",
             rho0=True, force="none", nu=0.01, u0=0.1, steps=32, calls=1, read="state"),
        # The sweep of 512 power-law cavities, every one stepped by the same
        # launch.
        dict(name="sweep_512", kind="batch", count=512, storage="fp32", steps=32),
        # A smaller sweep kept in FP16 deviations.
        dict(name="sweep_96_fp16", kind="batch", count=96, storage="fp16", steps=32),
        # The trained warm-start network on a full batch.
        dict(name="network_forward_16", kind="forward", R=128, batch=16),
        # Four Adam steps of its training, then the parameters.
        dict(name="network_train_16", kind="train", R=128, batch=16, steps=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solver"] * 7 + ["batch"] * 2 + ["forward", "train"])
    if kind == "batch":
        return dict(kind="batch", count=_log_int(rng, 8, 256), storage=rng.choice(["fp32", "fp32", "fp16", "bf16"]),
                    steps=rng.choice([20, 32, 50]))
    if kind in ("forward", "train"):
        c = dict(kind=kind, R=rng.choice([64, 96, 128]), batch=rng.randint(1, 16))
        if kind == "train":
            c["steps"] = rng.randint(2, 4)
        return c
    flow = rng.choice(["periodic", "periodic", "periodic", "cavity", "cavity", "channel", "trapezoid"])
    top = 3000 if flow == "periodic" else 1200
    nx = _log_int(rng, 48, top)
    ny = max(48, min(top, int(nx * math.exp(rng.uniform(-0.7, 0.7)))))
    c = dict(kind="solver", flow=flow, nx=nx, ny=ny, fluid="newton", storage="fp32", rho0=False, force="none",
             u0=U_LID, steps=0, calls=1, read="state")
    if flow == "periodic":
        c["storage"] = rng.choice(["fp32", "fp32", "fp32", "fp16", "bf16"])
        c["rho0"] = c["storage"] == "fp32" and rng.random() < 0.25
        c["force"] = rng.choice(["none", "none", "const", "field"])
        c["nu"] = math.exp(rng.uniform(math.log(2e-3), math.log(2e-2)))
    elif flow == "channel":
        c["force"] = rng.choice(["const", "field"])
        c["nu"] = 1e-3
    else:
        c["fluid"] = "power" if flow == "trapezoid" else rng.choice(["newton", "power"])
        if c["fluid"] == "power":
            c["re"] = math.exp(rng.uniform(math.log(100.0), math.log(1000.0)))
            c["n"] = rng.choice([rng.uniform(0.5, 0.95), rng.uniform(1.05, 1.5)])
        else:
            c["nu"] = U_LID / math.exp(rng.uniform(math.log(100.0), math.log(1000.0)))
        c["read"] = rng.choice(["state", "residual"])
    c["steps"] = max(16, min(500, int(1.5e8 / (nx * ny))))
    return c


# ------------------------------------------------------------------- inputs


def _power_law(re, n, u0=U_LID):
    """(K, n, nu_min, nu_max) and nu_ref of a cavity with a lid of length 1."""
    K = u0 ** (2.0 - n) / re
    nu_ref = K * u0 ** (n - 1.0)
    return (K, n, nu_ref / 20.0, nu_ref * 20.0), nu_ref


# Power-law cavities are cold starts: from rest and, in FP32, marched for a
# while before the pass so that the whole cavity moves (a node at rest has no
# viscosity to solve for).  The seed draws their Reynolds numbers.
def _marched(case):
    return 96 if case["storage"] == "fp32" else 0



def _problem(case, seed):
    """Keywords of mdf.Solver / mdf.Batch for a single problem."""
    nx, ny, flow = case["nx"], case["ny"], case["flow"]
    kw = dict(nx=nx, ny=ny, storage=case["storage"], rho0=case["rho0"])
    if flow == "periodic":
        kw.update(nu=case["nu"], lx=TWO_PI, ly=TWO_PI * ny / nx)
    elif flow == "channel":
        s = np.arange(ny) / (ny - 1.0)
        y = 0.5 * (1.0 + np.tanh(1.5 * (2.0 * s - 1.0)) / math.tanh(1.5))
        lx = nx / ny
        kw.update(nu=case["nu"], grid="separable", x=np.arange(nx) * (lx / nx), y=y, lx=lx, ly=1.0,
                  walls=(False, True))
    else:
        kw.update(walls=(True, True), u_wall=(0.0, 0.0, 0.0, case["u0"]), lx=1.0, ly=(ny - 1.0) / (nx - 1.0))
        if flow == "trapezoid":  # lid of length 1, bottom 0.5, height 1
            XI, ET = np.meshgrid(np.arange(nx) / (nx - 1.0), np.arange(ny) / (ny - 1.0))
            half = 0.25 * (1.0 + ET)
            kw.update(grid="curvilinear", x=0.5 - half + 2.0 * half * XI, y=ET)
        if case["fluid"] == "power":
            re = case["re"] * np.random.default_rng(seed).uniform(0.9, 1.1)
            kw["power_law"], kw["nu"] = _power_law(re, case["n"])
        else:
            kw["nu"] = case["nu"]
    return kw


def _modes(g, shape, device, count=3):
    """A smooth random stream function and its derivatives, periodic with
    period 2 pi on both axes, of order one."""
    ny, nx = shape
    x = torch.arange(nx, device=device, dtype=torch.float64) * (TWO_PI / nx)
    y = torch.arange(ny, device=device, dtype=torch.float64).unsqueeze(1) * (TWO_PI / ny)
    psi = torch.zeros(shape, device=device, dtype=torch.float64)
    dx, dy = torch.zeros_like(psi), torch.zeros_like(psi)
    for _ in range(count):
        kx, ky = int(g.integers(1, 4)), int(g.integers(1, 4))
        px, py, a = g.uniform(0, TWO_PI), g.uniform(0, TWO_PI), g.uniform(0.2, 0.5)
        sx, cx = torch.sin(kx * x + px), torch.cos(kx * x + px)
        sy, cy = torch.sin(ky * y + py), torch.cos(ky * y + py)
        psi += a * sx * sy
        dx += a * kx * cx * sy
        dy += a * ky * sx * cy
    return psi, dx, dy


def _fields(case, seed, device):
    """Initial u, v, p and, where the case has them, force and density fields
    (FP32 tensors): a Taylor-Green vortex with random phases and modes, a
    channel profile with a perturbation, a vortex that meets the walls of a
    cavity at rest, or rest."""
    g = np.random.default_rng(seed)
    nx, ny, u0 = case["nx"], case["ny"], case["u0"]
    psi, dx, dy = _modes(g, (ny, nx), device)
    x = torch.arange(nx, device=device, dtype=torch.float64)
    y = torch.arange(ny, device=device, dtype=torch.float64).unsqueeze(1)
    p = torch.zeros((ny, nx), device=device, dtype=torch.float64)
    if case["flow"] == "periodic":
        X, Y = x * (TWO_PI / nx) + g.uniform(0, TWO_PI), y * (TWO_PI / ny) + g.uniform(0, TWO_PI)
        u = u0 * (-torch.cos(X) * torch.sin(Y) + 0.1 * dy)
        v = u0 * (torch.sin(X) * torch.cos(Y) - 0.1 * dx)
        p = -(u0 * u0 / 4.0) * (torch.cos(2.0 * X) + torch.cos(2.0 * Y))
    elif case["flow"] == "channel":
        s = torch.linspace(-1.0, 1.0, ny, device=device, dtype=torch.float64).unsqueeze(1)
        Y = 0.5 * (1.0 + torch.tanh(1.5 * s) / math.tanh(1.5))
        w = 4.0 * Y * (1.0 - Y)
        u = u0 * w * (1.0 + 0.1 * dy)
        v = -0.1 * u0 * w * dx
    else:
        xi, et = x / (nx - 1.0), y / (ny - 1.0)
        wx, wy = torch.sin(math.pi * xi), torch.sin(math.pi * et)
        q = 1.0 + 0.3 * psi  # psi_wall = wx^2 wy^2 q
        if case["fluid"] == "power":
            q = torch.zeros_like(psi)  # from rest
        u = u0 * (2.0 * wx * wx * wy * torch.cos(math.pi * et) * q)
        v = -u0 * (2.0 * wx * torch.cos(math.pi * xi) * wy * wy * q)
    out = dict(u=u, v=v, p=p)
    if case["force"] == "field":
        k = 8.0 * case["nu"] * u0
        base = 1.0 if case["flow"] == "channel" else 0.0
        out["fx"], out["fy"] = k * (base + 0.2 * dy), -k * 0.2 * dx
    if case["rho0"]:
        out["rho"] = 1.0 + 0.1 * psi
    return {k: t.to(torch.float32).contiguous() for k, t in out.items()}


def _const_force(case, seed):
    a = np.random.default_rng(seed + 1).uniform(0.5, 1.5)
    return a * 8.0 * case["nu"] * case["u0"], 0.25 * a * 8.0 * case["nu"] * case["u0"]


def _time_force(case, seed):
    fx, fy = _const_force(case, seed)
    return [(fx * math.cos(0.1 * k), fy * math.sin(0.1 * k)) for k in range(case["calls"])]


def _sweep(case, seed):
    """Re, power-law index, side of every cavity of a sweep: the sides come in
    equal shares, Re and n are drawn from the ranges in which the flow of
    every side settles."""
    g = np.random.default_rng(seed)
    n = case["count"]
    re = np.exp(g.uniform(math.log(100.0), math.log(1000.0), size=n))
    index = g.uniform(0.5, 1.4, size=n)
    index = np.where(index > 0.95, index + 0.1, index)  # [0.5, 1.5] without the neighbourhood of 1
    return re, index, np.array([SIDES[i % len(SIDES)] for i in range(n)])


def _net_inputs(case, seed, device):
    """Input planes and smooth targets of `batch` square cavities, FP32."""
    g = np.random.default_rng(seed)
    R, B = case["R"], case["batch"]
    x = torch.empty((B, 8, R, R), device=device, dtype=torch.float64)
    s = torch.arange(R, device=device, dtype=torch.float64) / (R - 1.0)
    x[:, 0] = torch.from_numpy(g.uniform(-1, 1, size=B)).to(device).view(B, 1, 1)  # scaled log Re
    x[:, 1] = torch.from_numpy(g.uniform(-1, 1, size=B)).to(device).view(B, 1, 1)  # scaled index
    x[:, 2], x[:, 3] = s, s.unsqueeze(1)                                           # node coordinates
    x[:, 4], x[:, 5], x[:, 6], x[:, 7] = 1.0, 0.0, 0.0, 1.0                         # metric coefficients
    t = torch.empty((B, 3, R, R), device=device, dtype=torch.float64)
    for b in range(B):
        psi, dx, dy = _modes(g, (R, R), device, count=2)
        t[b, 0], t[b, 1], t[b, 2] = 0.5 * dy, -0.5 * dx, 0.2 * psi
    return x.to(torch.float32).contiguous(), t.to(torch.float32).contiguous()


def _net_params(shapes, seed):
    """He initialisation of a stack of 3 x 3 convolutions, zero biases."""
    g = np.random.default_rng(seed + 17)
    parts = []
    for i, (co, ci) in enumerate(shapes):
        std = math.sqrt(2.0 / (9.0 * ci)) * (0.1 if i == len(shapes) - 1 else 1.0)
        parts += [(std * g.standard_normal(co * 9 * ci)).astype(np.float32), np.zeros(co, dtype=np.float32)]
    return np.concatenate(parts)


LEARNING_RATE = 2e-4


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "solver":
        kw = _problem(case, seed)
        s = mdf.Solver(kw.pop("nx"), kw.pop("ny"), **kw)
        f = _fields(case, seed, dev)
        torch.cuda.synchronize()
        s.init(f["u"], f["v"], f["p"])
        if case["rho0"]:
            s.init_rho0(f["rho"])
        if case["force"] == "field":
            s.set_force((f["fx"], f["fy"]))
        elif case["force"] == "const":
            s.set_force(_const_force(case, seed))
        if case["fluid"] == "power":
            s.step(_marched(case))
            s.synchronize()
            if case["read"] == "residual":
                s.residual()
        st = dict(kind="solver", solver=s, steps=case["steps"], calls=case["calls"], read=case["read"], forces=None,
                  rho0=case["rho0"])
        if case["force"] == "time":
            st["forces"] = _time_force(case, seed)
        shape = (case["ny"], case["nx"])
        if case["read"] == "fields":
            st["out"] = {k: torch.empty(shape, device=dev) for k in ("u", "v", "P")}
        else:
            st["out"] = torch.empty((2, 5) + shape, device=dev)
        if case["rho0"]:
            st["rho"] = torch.empty(shape, device=dev)
        return st
    if case["kind"] == "batch":
        re, n, side = _sweep(case, seed)
        probs = []
        for r, k, m in zip(re, n, side):
            pl, nu = _power_law(float(r), float(k))
            probs.append(dict(nx=int(m), ny=int(m), nu=nu, walls=(True, True), u_wall=(0.0, 0.0, 0.0, U_LID),
                              power_law=pl, storage=case["storage"]))
        b = mdf.Batch(probs)
        problems = [b.problem(i) for i in range(len(probs))]
        b.step(_marched(case))
        size = [10 * int(m) * int(m) for m in side]
        k = min(CHECKED, len(size))
        first, rest = torch.empty(sum(size[:k]), device=dev), torch.empty(sum(size[k:]), device=dev)
        outs = [t.view(2, 5, int(m), int(m)) for t, m in zip(first.split(size[:k]) + rest.split(size[k:]), side)]
        torch.cuda.synchronize()
        return dict(kind="batch", batch=b, problems=problems, steps=case["steps"],
                    states=[first, rest], outs=outs)
    net = WS.Net(case["R"], case["batch"])
    x, t = _net_inputs(case, seed, dev)
    if case["kind"] == "forward":
        net.load(WEIGHTS)
        out = torch.empty((case["batch"], 3, case["R"], case["R"]), device=dev)
        torch.cuda.synchronize()
        return dict(kind="forward", net=net, x=x, out=out)
    net.set_params(_net_params(net.layer_shapes(), seed))
    torch.cuda.synchronize()
    return dict(kind="train", net=net, x=x, t=t, steps=case["steps"])


def run(state):
    if state["kind"] == "solver":
        s = state["solver"]
        for k in range(state["calls"]):
            if state["forces"] is not None:
                s.set_force(state["forces"][k])
            s.step(state["steps"])
        if state["read"] == "fields":
            s.fields_device(state["out"])
            return state["out"]
        res = None
        if state["read"] == "residual":
            r, drift = s.residual()
            res = [r, np.array(drift, dtype=np.float32)]
        out = s.state(out=state["out"])
        if state["rho0"]:
            # the density through the C call (the binding returns host arrays)
            mdf.lib().mdf_get_rho0(s.handle, state["rho"].data_ptr(), 1)
            return [out, state["rho"]]
        return out if res is None else [out] + res
    if state["kind"] == "batch":
        state["batch"].step(state["steps"])
        for p, o in zip(state["problems"], state["outs"]):
            p.state(out=o)
        return state["states"]
    if state["kind"] == "forward":
        return state["net"].forward(state["x"], out=state["out"])
    loss = [state["net"].train_step(state["x"], state["t"], LEARNING_RATE) for _ in range(state["steps"])]
    return [loss, state["net"].get_params()]


# --------------------------------------------------------------------- work

# Additions and multiplications of one node update (an FMA counts two): the
# four streamed populations of both distributions in two passes, the moments
# and equilibria of two stages and three relaxations; on top of it the
# power-law rates and the density's own lane.
NODE_FLOPS, POWER_FLOPS, RHO0_FLOPS = 350, 100, 160

CHANNELS = [(8, 32, 1), (32, 32, 1), (32, 64, 2), (64, 64, 2), (64, 128, 4), (128, 128, 4), (128, 256, 8),
            (256, 256, 8), (256, 128, 4), (128, 128, 4), (128, 64, 2), (64, 64, 2), (64, 32, 1), (32, 32, 1),
            (32, 3, 1)]


def work(case):
    if case["kind"] == "solver":
        n, steps = case["nx"] * case["ny"], case["steps"] * case["calls"]
        node = 80 if case["storage"] == "fp32" else 56
        node += 40 if case["rho0"] else 0
        node += 8 if case["force"] == "field" else 0
        node += 16 if case["flow"] == "trapezoid" else 0
        flops = NODE_FLOPS + (POWER_FLOPS if case["fluid"] == "power" else 0) + (RHO0_FLOPS if case["rho0"] else 0)
        read = (node // 2 + 12 if case["read"] == "fields" else 80) + (12 if case["rho0"] else 0)
        return dict(bytes=n * (steps * node + read), flops=n * steps * flops)
    if case["kind"] == "batch":
        n = sum(int(m) ** 2 for m in _sweep(case, 0)[2])
        node = 80 if case["storage"] == "fp32" else 56
        return dict(bytes=n * (case["steps"] * node + 80), flops=n * case["steps"] * (NODE_FLOPS + POWER_FLOPS))
    R, B = case["R"], case["batch"]
    macs = sum(9 * ci * co * (R // d) ** 2 for ci, co, d in CHANNELS)
    params = sum(co * 9 * ci + co for ci, co, _ in CHANNELS)
    io = B * R * R * 4 * 11
    if case["kind"] == "forward":
        return dict(bytes=io + 4 * params, flops=2 * B * macs)
    return dict(bytes=case["steps"] * (io + 24 * params) + 4 * params, flops=case["steps"] * 6 * B * macs)


# -------------------------------------------------------------------- exact


class _Method:
    """One time step of the method in FP64 for problems of one grid; scalars
    of a problem may be tensors [B, 1, 1], planes are [B, ny, nx]."""

    def __init__(self, nx, ny, nu, grid="uniform", lx=1.0, ly=1.0, x=None, y=None, power_law=None,
                 walls=(False, False), u_wall=(0, 0, 0, 0), storage="fp32", rho0=False, c=1.0, cfl=0.5, eta=0.8,
                 s_ratio=1.5, device="cuda"):
        t = lambda a: torch.as_tensor(a, dtype=torch.float64, device=device)  # noqa: E731
        self.nx, self.ny, self.c, self.cs2, self.sr = nx, ny, c, 0.4 * c * c, s_ratio
        self.xw, self.yw, self.uw, self.pl, self.nu = walls[0], walls[1], u_wall, power_law, nu
        self.a1, self.a0, self.a2 = 0.5 * eta, 1.5 * (1.0 - eta), 0.5 * (1.0 - eta)
        self.curvi = grid == "curvilinear"
        if grid == "uniform":
            dx, dy = lx / (nx - 1 if walls[0] else nx), ly / (ny - 1 if walls[1] else ny)
            dmin = min(dx, dy)
            self.kx, self.ky = c / dx, c / dy
        elif grid == "separable":
            x, y = np.asarray(x, dtype=np.float64), np.asarray(y, dtype=np.float64)
            gx, ex = self._diff(x, 0, walls[0], lx)
            gy, ey = self._diff(y, 0, walls[1], ly)
            dmin = min(ex.min(), ey.min())
            self.kx, self.ky = t(c / gx), t(c / gy).unsqueeze(1)
        else:
            x, y = np.asarray(x, dtype=np.float64), np.asarray(y, dtype=np.float64)
            xi, xj = self._diff(x, 1, True, 0)[0], self._diff(x, 0, True, 0)[0]
            yi, yj = self._diff(y, 1, True, 0)[0], self._diff(y, 0, True, 0)[0]
            J = xi * yj - xj * yi
            self.m = [t(c * yj / J), t(c * -xj / J), t(c * -yi / J), t(c * xi / J)]  # xi_x, xi_y, eta_x, eta_y
            dmin = min(np.hypot(np.diff(x, axis=a), np.diff(y, axis=a)).min() for a in (0, 1))
        self.dt = cfl * dmin / c

    @staticmethod
    def _diff(z, axis, wall, period):
        """Second-order differences per node index and the edge lengths."""
        z = np.moveaxis(z, axis, 0)
        d = np.empty_like(z)
        d[1:-1] = 0.5 * (z[2:] - z[:-2])
        edge = np.diff(z, axis=0)
        if wall:
            d[0] = 0.5 * (-3.0 * z[0] + 4.0 * z[1] - z[2])
            d[-1] = 0.5 * (3.0 * z[-1] - 4.0 * z[-2] + z[-3])
        else:
            d[0] = 0.5 * (z[1] - (z[-1] - period))
            d[-1] = 0.5 * ((z[0] + period) - z[-2])
            edge = np.concatenate([edge, [z[0] + period - z[-1]]])
        return np.moveaxis(d, 0, axis), edge

    # A distribution is a list of its five populations, each a tensor with the
    # two velocity components (alpha = u, v) on its first axis.

    def feq(self, u, v, P):
        i = 0.5 / self.c
        w, uv = torch.stack([u, v]) / 5, u * v * i
        x, y = torch.stack([(u * u + P) * i, uv]), torch.stack([uv, (v * v + P) * i])
        return [w, w + x, w + y, w - x, w - y]

    def moments(self, g):
        u, v = g[0] + g[1] + g[2] + g[3] + g[4]
        return u, v, 0.5 * (self.c * ((g[1][0] - g[3][0]) + (g[2][1] - g[4][1])) - u * u - v * v)

    def rates(self, n):
        """First-moment rate s = cs^2 / nu per node."""
        if self.pl is None:
            return self.cs2 / self.nu
        t = lambda z: torch.as_tensor(z, dtype=torch.float64, device=n[0].device)  # noqa: E731
        K, ni, lo, hi = (t(z) for z in self.pl)
        (gx1, gx2), (gy1, gy2) = self.c * (n[1] - n[3]), self.c * (n[2] - n[4])
        sxy = 0.5 * (gy1 + gx2)
        lg = 0.5 * torch.log((2.0 * (gx1 * gx1 + gy2 * gy2 + 2.0 * sxy * sxy)).clamp_min(1e-280))
        a, m = 0.5 * self.cs2 * self.dt, ni - 1.0
        lmin, lmax = torch.log(lo), torch.log(hi)
        k = torch.log(K) + m * lg
        q = torch.minimum(torch.maximum(k / ni, lmin), lmax)
        for _ in range(8):  # Newton on q = ln nu of nu = K (g / (nu + a))^(n-1)
            e = torch.exp(q)
            q = q - (q - k + m * torch.log(e + a)) / (1.0 + m * e / (e + a))
            q = torch.minimum(torch.maximum(q, lmin - 1.0), lmax + 1.0)
        return self.cs2 / torch.minimum(torch.maximum(torch.exp(q), lo), hi)

    def relax(self, g, n, Ap, A):
        """g - n + Ap n + (A - Ap) P_c n, P_c the projector on first moments."""
        x, y, b = 0.5 * (A - Ap) * (n[1] - n[3]), 0.5 * (A - Ap) * (n[2] - n[4]), 1 - Ap
        return [g[0] - b * n[0], g[1] - b * n[1] + x, g[2] - b * n[2] + y, g[3] - b * n[3] - x, g[4] - b * n[4] - y]

    def grad(self, f, axis, sign):
        """Mixed central/upwind difference per node index along an axis (-1: x,
        -2: y) for a population moving with `sign`, times that sign."""
        f1, fm1, fm2 = (torch.roll(f, sign * k, axis) for k in (-1, 1, 2))
        if (self.xw if axis == -1 else self.yw):
            at = 1 if sign > 0 else f.shape[axis] - 2  # beyond the wall: linear extrapolation
            fm2.select(axis, at).copy_(2.0 * fm1.select(axis, at) - f.select(axis, at))
        return self.a1 * (f1 - fm1) + self.a0 * (f - fm1) + self.a2 * (fm2 - fm1)

    def stream(self, base, f, step):
        """base - step c_j.grad f for the five populations."""
        out = [base[0]]
        for j in (1, 2, 3, 4):
            s, x = (1 if j < 3 else -1), j in (1, 3)
            if not self.curvi:
                out.append(base[j] - step * (self.kx if x else self.ky) * self.grad(f[j], -1 if x else -2, s))
                continue
            xi, eta = (s * self.m[0], s * self.m[2]) if x else (s * self.m[1], s * self.m[3])
            acc = base[j]
            for ct, axis in ((xi, -1), (eta, -2)):
                up = torch.where(ct > 0, self.grad(f[j], axis, 1), self.grad(f[j], axis, -1))
                acc = acc - step * ct.abs() * up
            out.append(acc)
        return out

    def walls(self, g):
        """Non-equilibrium extrapolation onto the wall nodes, in place."""
        def put(dst, src, side):
            nb = [p[src] for p in g]
            u, v = sum(nb)
            z = torch.zeros_like(u)
            e0, e1 = self.feq(u, v, z), self.feq(z + self.uw[side], z, z)
            for j in range(5):
                g[j][dst] = nb[j] + e1[j] - e0[j]
        e, inner = Ellipsis, slice(1, -1)
        if self.xw:
            rows = inner if self.yw else slice(None)
            put((e, rows, 0), (e, rows, 1), 0)
            put((e, rows, -1), (e, rows, -2), 1)
        if self.yw:
            cols = inner if self.xw else slice(None)
            put((e, 0, cols), (e, 1, cols), 2)
            put((e, -1, cols), (e, -2, cols), 3)
        if self.xw and self.yw:
            for dy, sy in ((0, 1), (-1, -2)):
                put((e, dy, 0), (e, sy, 1), 0)
                put((e, dy, -1), (e, sy, -2), 1)

    def init(self, u, v, p):
        u, v, p = (z.to(torch.float64).clone() for z in (u, v, p))
        if self.yw:
            u[..., 0, :], u[..., -1, :] = self.uw[2], self.uw[3]
            v[..., 0, :], v[..., -1, :] = 0.0, 0.0
        if self.xw:
            u[..., :, 0], u[..., :, -1] = self.uw[0], self.uw[1]
            v[..., :, 0], v[..., :, -1] = 0.0, 0.0
        return self.feq(u, v, p)

    def feq0(self, rho, u, v):
        x, y = rho * u * (0.5 / self.c), rho * v * (0.5 / self.c)
        return [rho / 5, rho / 5 + x, rho / 5 + y, rho / 5 - x, rho / 5 - y]

    def step(self, g, F=None, r=None):
        """One step of the distributions g (and of the density's, r) under
        the force F [2, 1, ny, nx]."""
        dt, h = self.dt, 0.5 * self.dt
        u, v, P = self.moments(g)
        n = [x - y for x, y in zip(g, self.feq(u, v, P))]
        s = self.rates(n)
        sp = self.sr * s
        rho = lambda q: (1.0 - 0.5 * dt * q) / (1.0 + 0.5 * dt * q)  # noqa: E731
        plus = self.relax(g, n, rho(sp), rho(s))
        bar = self.relax(g, n, 0.25 + 0.75 * rho(sp), 0.25 + 0.75 * rho(s))
        kp, k = 1.0 / (1.0 + 0.5 * h * sp), 1.0 / (1.0 + 0.5 * h * s)
        if r is not None:
            n0 = [x - y for x, y in zip(r, self.feq0(sum(r), u, v))]
            plus0 = self.relax(r, n0, rho(sp), rho(s))
            bar0 = self.relax(r, n0, 0.25 + 0.75 * rho(sp), 0.25 + 0.75 * rho(s))
        fb = self.stream(bar, bar, h)
        if F is not None:
            fb = [q + h * 0.2 * F for q in fb]
        u, v, P = self.moments(fb)
        f = self.relax(fb, [x - y for x, y in zip(fb, self.feq(u, v, P))], kp, k)
        walls = self.xw or self.yw
        if walls:
            self.walls(f)
        out = self.stream(plus, f, dt)
        if F is not None:
            out = [q + dt * 0.2 * F for q in out]
        if walls:
            self.walls(out)
        if r is None:
            return out, None
        fb0 = self.stream(bar0, bar0, h)
        n0 = [x - y for x, y in zip(fb0, self.feq0(sum(fb0), u, v))]
        return out, self.stream(plus0, self.relax(fb0, n0, kp, k), dt)


def _state(g, k):
    """fhat [2, 5, ny, nx] of problem k."""
    return torch.stack([p[:, k] for p in g], dim=1)


def _exact_solver(case, seed, dev):
    m = _Method(**_problem(case, seed), device=dev)
    f = _fields(case, seed, dev)
    one = lambda t: t.unsqueeze(0)  # noqa: E731
    g = m.init(one(f["u"]), one(f["v"]), one(f["p"]))
    if case["fluid"] == "power":
        for _ in range(_marched(case)):
            g, _r = m.step(g)
    r = m.feq0(one(f["rho"]).double(), *m.moments(g)[:2]) if case["rho0"] else None
    u_start, v_start = m.moments(g)[:2]
    for k in range(case["calls"]):
        F = None
        if case["force"] == "field":
            F = torch.stack([f["fx"], f["fy"]]).double().unsqueeze(1)
        elif case["force"] == "const":
            F = torch.tensor(_const_force(case, seed), dtype=torch.float64, device=dev).view(2, 1, 1, 1)
        elif case["force"] == "time":
            F = torch.tensor(_time_force(case, seed)[k], dtype=torch.float64, device=dev).view(2, 1, 1, 1)
        for _ in range(case["steps"]):
            g, r = m.step(g, F, r)
    u, v, P = m.moments(g)
    if case["read"] == "fields":
        return {"u": u[0], "v": v[0], "P": P[0]}
    state = _state(g, 0)
    if case["read"] == "residual":
        d = ((u - u_start) ** 2 + (v - v_start) ** 2).sum().sqrt()
        res = float(d / (case["steps"] * case["calls"] * (u * u + v * v).sum().sqrt()))
        return [state, res, np.array([float(u.sum()), float(v.sum())])]
    return [state, sum(r)[0]] if case["rho0"] else state


def _exact_batch(case, seed, dev):
    re, n, side = (a[:CHECKED] for a in _sweep(case, seed))
    parts = [None] * len(side)
    for m in sorted(set(side.tolist())):
        part = [i for i in range(len(side)) if side[i] == m]
        pl = [_power_law(float(re[i]), float(n[i]))[0] for i in part]
        pl = tuple(torch.tensor([q[j] for q in pl], dtype=torch.float64, device=dev).view(-1, 1, 1) for j in range(4))
        M = _Method(m, m, 1.0, power_law=pl, walls=(True, True), u_wall=(0.0, 0.0, 0.0, U_LID), device=dev)
        z = torch.zeros((len(part), m, m), device=dev)
        g = M.init(z, z, z)
        for _ in range(_marched(case) + case["steps"]):
            g, _r = M.step(g)
        for j, i in enumerate(part):
            parts[i] = _state(g, j).reshape(-1)
    return [torch.cat(parts), None]


def _net_apply(p, x):
    """The U-Net of the warm start on FP64 tensors (parameters as one flat
    vector: per layer weights [Cout][3][3][Cin], then bias)."""
    F = torch.nn.functional
    w, k = [], 0
    for ci, co, _ in CHANNELS:
        q = p[k:k + co * 9 * ci].view(co, 3, 3, ci).permute(0, 3, 1, 2)
        w.append((q, p[k + co * 9 * ci:k + co * 9 * ci + co]))
        k += co * 9 * ci + co

    def conv(h, l, skip=None, act=True):
        z = F.conv2d(h, w[l][0], w[l][1], padding=1)
        z = z if skip is None else z + skip
        return F.silu(z) if act else z

    up = lambda h: F.interpolate(h, scale_factor=2, mode="nearest")  # noqa: E731
    s0 = conv(conv(x, 0), 1)
    s1 = conv(conv(F.avg_pool2d(s0, 2), 2), 3)
    s2 = conv(conv(F.avg_pool2d(s1, 2), 4), 5)
    h = conv(conv(F.avg_pool2d(s2, 2), 6), 7)
    h = conv(conv(up(h), 8, s2), 9)
    h = conv(conv(up(h), 10, s1), 11)
    h = conv(conv(up(h), 12, s0), 13)
    return conv(h, 14, act=False)


def _exact_net(case, seed, dev):
    x, t = (z.double() for z in _net_inputs(case, seed, dev))
    if case["kind"] == "forward":
        p = torch.from_numpy(np.load(WEIGHTS)).reshape(-1).double().to(dev)
        with torch.no_grad():
            return torch.cat([_net_apply(p, x[i:i + 4]) for i in range(0, len(x), 4)])
    p = torch.from_numpy(_net_params([(co, ci) for ci, co, _ in CHANNELS], seed)).double().to(dev)
    m, v, losses = torch.zeros_like(p), torch.zeros_like(p), []
    b1, b2, eps = 0.9, 0.999, 1e-8
    for k in range(1, case["steps"] + 1):
        q = p.detach().requires_grad_(True)
        total = 0.0
        grad = torch.zeros_like(p)
        for i in range(0, len(x), 4):
            part = ((_net_apply(q, x[i:i + 4]) - t[i:i + 4]) ** 2).sum() / t.numel()
            grad += torch.autograd.grad(part, q)[0]
            total += float(part.detach())
        losses.append(total)
        m, v = b1 * m + (1 - b1) * grad, b2 * v + (1 - b2) * grad * grad
        p = p - LEARNING_RATE * (m / (1 - b1 ** k)) / ((v / (1 - b2 ** k)).sqrt() + eps)
    return [losses, p]


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] == "solver":
        return _exact_solver(case, seed, dev)
    if case["kind"] == "batch":
        return _exact_batch(case, seed, dev)
    return _exact_net(case, seed, dev)
