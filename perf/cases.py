"""Performance cases: what users of this framework have it do, at the sizes they do it.

Five kinds of work, each through the public entry points:
  march    one simulation: clb.Simulation.step, .residual and the fields on the device (clb_macros_device), in the
           three storage forms (f64, f16n, f16s), on cavities, channels and periodic boxes;
  batch    a parameter study: clb.Batch.step, the Nusselt numbers of every case and the fields of some;
  conv     one convolution layer of the warm-start network: forward, input gradient, weight and bias gradient;
  train    the network's forward pass, loss and backward pass (surrogate.Net);
  predict  the network's inference from host features to host fields (surrogate.predict).
"""
import math

import numpy as np
import torch

from paper_2110_05943_gb300 import clb, surrogate
from paper_2110_05943_gb300.inputs import batch_cases

PRECISION = {"f64": clb.CLB_F64, "f16s": clb.CLB_F16S, "f16n": clb.CLB_F16N}
# bytes of one node's state, read and written once a step, and what is read of its porosity
NODE_BYTES = {"f64": 2 * 14 * 8 + 8, "f16s": 2 * 14 * 2 + 4, "f16n": 2 * (14 * 2 + 8) + 4}
NODE_FLOPS = 257           # arithmetic of one node update (both collisions, velocity, force)
WEIGHTS = "paper_2110_05943_gb300/weights/warmstart_128.npz"
CHANNELS = (32, 64, 96, 160, 192, 288)   # of the network's layers, as it carries them


def _march(nx, ny, precision, steps, walls="cavity", porosity="field", residual=False, shift=1, forchheimer=1, Ra=1e6,
           Da=1e-3, Pr=0.71, sigma=1.0, **more):
    return dict(kind="march", nx=nx, ny=ny, precision=precision, steps=steps, walls=walls, porosity=porosity,
                residual=residual, shift=shift, forchheimer=forchheimer, Ra=Ra, Da=Da, Pr=Pr, sigma=sigma, **more)


def listed():
    return [
        # the smallest run: the 64^2 cavity with uniform porosity, between two checks for steadiness
        _march(64, 64, "f64", 100, porosity="uniform", residual=True, Ra=1e4, Da=1e-2, Pr=1.0, name="f64_cavity_64"),
        # the Brinkman channel, periodic along x and driven by a body force
        _march(1024, 256, "f64", 100, walls="channel", porosity="uniform", Ra=1e5, Da=1e-2, name="f64_channel_1024x256"),
        # the MRT limit (unit shifts) on a grid that fits no tile, random porosity
        _march(701, 509, "f64", 100, shift=0, Ra=1e5, Da=1e-2, sigma=0.8, name="f64_mrt_701x509"),
        # the large FP64 run: a seeded random-porosity cavity
        _march(4096, 4096, "f64", 8, name="f64_cavity_4096"),
        # the small cavity in the accurate FP16 form, between two checks for steadiness
        _march(128, 128, "f16n", 1000, residual=True, Ra=1e4, Da=1e-2, name="f16n_cavity_128"),
        # the large run in the accurate FP16 form
        _march(4096, 4096, "f16n", 64, sigma=0.8, name="f16n_cavity_4096"),
        # the largest run, in the fast FP16 form
        _march(8192, 8192, "f16s", 32, sigma=0.8, name="f16s_cavity_8192"),
        # a mid-sized channel with odd sides in the fast FP16 form, Brinkman-Darcy (no Forchheimer term)
        _march(1531, 389, "f16s", 200, walls="channel", forchheimer=0, Ra=1e5, Da=1e-2, name="f16s_channel_1531x389"),
        # a parameter study: 512 cavities with sides from 16 to 1024
        dict(kind="batch", cases=512, shapes=7, side_lo=64, side_hi=1024, precision="f16n", steps=64, every=64,
             name="batch_f16n_512"),
        # a decoder layer of the network at the training batch
        dict(kind="conv", n=16, size=64, cin=160, cout=64, name="conv_64x64_160_64"),
        # one training step's passes, batch 16
        dict(kind="train", n=16, size=128, name="train_16"),
        # the warm start of one cavity
        dict(kind="predict", n=1, size=128, name="predict_1"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    p = rng.random()
    if p < 0.65:
        precision = "f64" if p < 0.35 else rng.choice(("f16n", "f16s"))
        top, budget = (4096, 1.2e8) if precision == "f64" else (8192, 1.6e9)
        nx, ny = _log(rng, 48, top), _log(rng, 48, top)
        steps = int(max(4, min(200, budget / (nx * ny))))
        lo = max(3.0, 2 * math.log10(ny) - 2.8)   # tall grids at low Ra would be all viscosity
        return _march(nx, ny, precision, steps, walls=rng.choice(("cavity", "cavity", "channel", "periodic")),
                      porosity=rng.choice(("field", "field", "uniform")), residual=rng.random() < 0.3,
                      shift=int(rng.random() < 0.8), forchheimer=int(rng.random() < 0.8),
                      Ra=round(10 ** rng.uniform(lo, 6), 1), Da=float("%.2e" % 10 ** rng.uniform(-3.5, -1)),
                      Pr=round(rng.uniform(0.7, 1.0), 2), sigma=round(rng.uniform(0.5, 2.0), 2))
    if p < 0.77:
        n = _log(rng, 8, 256)
        return dict(kind="batch", cases=n, shapes=rng.randrange(1000), side_lo=64, side_hi=_log(rng, 128, 1024),
                    precision=rng.choice(("f64", "f16n", "f16n", "f16s")), steps=rng.choice((32, 33, 64)),
                    every=max(8, n // 8))
    if p < 0.9:
        return dict(kind="conv", n=rng.randint(1, 16), size=rng.choice((16, 32, 64, 128)), cin=rng.choice(CHANNELS),
                    cout=rng.choice(CHANNELS[:-1]))
    if p < 0.96:
        return dict(kind="train", n=rng.randint(1, 16), size=rng.choice((64, 128)))
    return dict(kind="predict", n=rng.randint(1, 16), size=rng.choice((64, 128)))


# ------------------------------------------------------------------ inputs
def _rand(seed, *shape):
    return torch.randn(shape, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda")


def _porosity(nx, ny, seed, ell=32.0):
    """0.3 + 0.6 Phi(g), g a unit Gaussian random field of correlation length ell (or an eighth of the grid)."""
    ell = min(ell, min(nx, ny) / 8.0)
    kx = 2 * math.pi * torch.fft.rfftfreq(nx, device="cuda")
    ky = 2 * math.pi * torch.fft.fftfreq(ny, device="cuda")
    w = torch.fft.rfft2(_rand(seed, ny, nx)) * torch.exp(-0.25 * ell * ell * (ky[:, None] ** 2 + kx[None, :] ** 2))
    g = torch.fft.irfft2(w, s=(ny, nx)).double()
    return 0.3 + 0.6 * torch.special.ndtr((g - g.mean()) / g.std())


WALLS = {"cavity": ("wall",) * 4, "channel": ("periodic", "periodic", "wall", "wall"), "periodic": ("periodic",) * 4}
WALL_T = {"cavity": (1.0, 0.0, None, None), "channel": (None, None, 1.0, 0.0), "periodic": (None,) * 4}
LID = 0.01                # speed of the channel's upper plate
AX = 1e-7                 # body force of channels and periodic boxes


def _start(c, seed):
    """Porosity and a smooth moving state (rho, ux, uy, T) that vanishes at the walls, on the GPU in 64 bits."""
    nx, ny = c["nx"], c["ny"]
    phi = _porosity(nx, ny, seed) if c["porosity"] == "field" else torch.full((ny, nx), 0.6, dtype=torch.float64, device="cuda")
    r = np.random.RandomState(seed)
    x = torch.linspace(0, 1, nx, dtype=torch.float64, device="cuda")[None, :]
    y = torch.linspace(0, 1, ny, dtype=torch.float64, device="cuda")[:, None]
    win = torch.ones((ny, nx), dtype=torch.float64, device="cuda")
    if c["walls"] == "cavity":
        win = win * torch.sin(math.pi * x) ** 2
    if c["walls"] != "periodic":
        win = win * torch.sin(math.pi * y) ** 2

    def mode():
        kx, ky = r.randint(1, 3, 2)
        return torch.cos(2 * math.pi * (int(kx) * x + int(ky) * y) + r.uniform(0, 2 * math.pi))

    T = {"cavity": 1 - x + 0 * y, "channel": 1 - y + 0 * x, "periodic": 0.5 + 0 * (x + y)}[c["walls"]]
    return phi, (1 + 0.003 * mode(), 0.03 * win * mode(), 0.03 * win * mode(), T + 0.1 * win * mode())


def _params(c, nx, ny, **more):
    return clb.clb_params_default(nx=nx, ny=ny, precision=PRECISION[c["precision"]], **more)


def _batch(c, seed):
    shapes = batch_cases(c["cases"], seed=c["shapes"], side_lo=c["side_lo"], side_hi=c["side_hi"])
    return [(s.nx, s.ny, q) for s, q in zip(shapes, batch_cases(c["cases"], seed=seed))]


def prepare(case, seed):
    c = case
    if c["kind"] == "march":
        phi, fields = _start(c, seed)
        p = _params(c, c["nx"], c["ny"], Ra=c["Ra"], Da=c["Da"], Pr=c["Pr"], sigma=c["sigma"], shift=c["shift"],
                    forchheimer=c["forchheimer"], ax=0.0 if c["walls"] == "cavity" else AX)
        bc = clb.clb_bc(WALLS[c["walls"]], u=(0.0, 0.0, 0.0, LID if c["walls"] == "channel" else 0.0), T=WALL_T[c["walls"]])
        sim = clb.Simulation.create(p, phi.cpu().numpy(), bc, stream=torch.cuda.current_stream().cuda_stream)
        sim.set_fields(*[f.cpu().numpy() for f in fields])
        out = [torch.empty((c["ny"], c["nx"]), dtype=torch.float64, device="cuda") for _ in range(4)]
        return {"case": c, "sim": sim, "out": out}
    if c["kind"] == "batch":
        cs = _batch(c, seed)
        b = clb.Batch([_params(c, nx, ny, Ra=q.Ra, Da=q.Da, Pr=q.Pr, sigma=q.sigma) for nx, ny, q in cs],
                      [q.phi for _, _, q in cs], [clb.clb_bc_cavity(1.0, 0.0) for _ in cs],
                      stream=torch.cuda.current_stream().cuda_stream)
        b.set_tiling(9)   # 8 x 16 threads, 4 tiles per block: what tune() finds for such studies
        return {"case": c, "batch": b}
    if c["kind"] == "conv":
        n, s, ci, co = c["n"], c["size"], c["cin"], c["cout"]
        w = (_rand(seed + 1, 9 * ci, co) / math.sqrt(9 * ci)).bfloat16()
        return {"case": c, "lib": surrogate._lib(), "x": _rand(seed, n, s, s, ci).clamp_min(0).bfloat16(), "w": w,
                "wt": w.t().contiguous(), "b": 0.1 * _rand(seed + 2, co), "dy": _rand(seed + 3, n, s, s, co).bfloat16()}
    n, s = c["n"], c["size"]
    net = surrogate.Net.create(torch, seed=0).load(WEIGHTS)
    r = np.random.RandomState(seed)
    X = []
    for i in range(n):
        phi = (r.uniform(0.4, 0.9) + (_porosity(s, s, seed + i, 16.0) - 0.6) / 2).clamp(0.3, 0.95).cpu().numpy()
        X.append(surrogate.features(phi, 10 ** r.uniform(3, 6), 10 ** r.uniform(-4, -1), r.uniform(0.7, 1.0), r.uniform(0.5, 2.0)))
    X = np.stack(X)
    if c["kind"] == "predict":
        return {"case": c, "net": net, "X": X}
    low = torch.nn.functional.avg_pool2d(_rand(seed, n, 4, s, s), 9, 1, 4, count_include_pad=False)
    return {"case": c, "net": net, "x": surrogate.to_bf16(torch, X), "y": (3 * low).permute(0, 2, 3, 1).contiguous()}


# ------------------------------------------------------------------ passes
def run(state):
    c = state["case"]
    if c["kind"] == "march":
        sim, out = state["sim"], state["out"]
        sim.step(c["steps"])
        res = {"fields": out}
        if c["residual"]:
            res["residual"] = list(sim.residual())
        clb.clb_macros_device(sim.handle, *[t.data_ptr() for t in out])
        return res
    if c["kind"] == "batch":
        b = state["batch"]
        b.step(c["steps"])
        # the hot wall's Nusselt number of every case, and the fields of some of the cases
        return {"nu": b.nusselt(clb.W), "fields": [b.macros(k) for k in range(0, c["cases"], c["every"])]}
    if c["kind"] == "conv":
        lib, n, s, ci, co = state["lib"], c["n"], c["size"], c["cin"], c["cout"]
        x, dy = state["x"], state["dy"]
        y = torch.empty((n, s, s, co), dtype=torch.bfloat16, device="cuda")
        dx = torch.empty((n, s, s, ci), dtype=torch.bfloat16, device="cuda")
        dw = torch.empty((9 * ci, co), device="cuda")
        db = torch.empty(co, device="cuda")
        p = torch.Tensor.data_ptr
        rc = [lib.clb_nop_conv_fwd(p(x), p(state["w"]), p(state["wt"]), p(state["b"]), p(y), 0, 1, n, s, s, ci, co, 9, None),
              lib.clb_nop_conv_dgrad(p(dy), p(state["w"]), p(x), p(dx), n, s, s, ci, co, 9, None),
              lib.clb_nop_zero(p(dw), dw.numel() * 4, None), lib.clb_nop_zero(p(db), db.numel() * 4, None),
              lib.clb_nop_conv_wgrad_bias(p(x), p(dy), p(dw), p(db), n, s, s, ci, co, 9, 0, None)]
        if any(rc):
            raise RuntimeError("convolution calls failed: %s" % rc)
        return {"y": y, "dx": dx, "dw": dw, "db": db}
    net, n, s = state["net"], c["n"], c["size"]
    if c["kind"] == "predict":
        return surrogate.predict(net, state["X"])
    out, acts = net.forward(state["x"], n, s, s)
    loss, g = net.loss_and_grad(out, state["y"])
    net.backward(g, acts, n, s, s)
    return {"out": out, "loss": loss, "grads": net.grads}


# (cin, cout, resolution divisor) of the network's layers, real channels; the last is 1x1
LAYERS = ((8, 24, 1), (24, 24, 1), (24, 48, 2), (48, 48, 2), (48, 96, 4), (96, 96, 4), (96, 192, 8), (192, 192, 8),
          (288, 96, 4), (96, 96, 4), (144, 48, 2), (48, 48, 2), (72, 24, 1), (24, 24, 1), (24, 4, 1))


def work(case):
    c = case
    if c["kind"] == "march":
        n = c["nx"] * c["ny"]
        return {"bytes": n * (c["steps"] * NODE_BYTES[c["precision"]] + 32), "flops": n * c["steps"] * NODE_FLOPS}
    if c["kind"] == "batch":
        n = sum(nx * ny for nx, ny, _ in _batch(c, 0))
        return {"bytes": n * c["steps"] * NODE_BYTES[c["precision"]], "flops": n * c["steps"] * NODE_FLOPS}
    if c["kind"] == "conv":
        m, ci, co = c["n"] * c["size"] ** 2, c["cin"], c["cout"]
        return {"bytes": 4 * m * (ci + co) + 9 * ci * co * 6, "flops": 3 * 2 * m * 9 * ci * co}
    m = c["n"] * c["size"] ** 2
    one = [2 * (m // d ** 2) * (9 if i < 14 else 1) * a * b for i, (a, b, d) in enumerate(LAYERS)]
    act = [2 * (m // d ** 2) * (a + b) for a, b, d in LAYERS]
    if c["kind"] == "predict":
        return {"bytes": sum(act), "flops": sum(one)}
    return {"bytes": 3 * sum(act), "flops": 3 * sum(one) - one[0]}


# ------------------------------------------------------------------ the same in plain 64-bit torch
EX, EY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)


def _from_moments(m):
    """Distributions whose raw moments (1, x, y, xx, yy, xy, xxy, xyy, xxyy) are m."""
    a, b = m[3] - m[8], m[4] - m[8]
    c, d = m[1] - m[7], m[2] - m[6]
    return [m[0] - m[3] - m[4] + m[8], (c + a) / 2, (d + b) / 2, (a - c) / 2, (b - d) / 2, (m[8] + m[5] + m[6] + m[7]) / 4,
            (m[8] - m[5] + m[6] - m[7]) / 4, (m[8] + m[5] - m[6] - m[7]) / 4, (m[8] - m[5] - m[6] + m[7]) / 4]


def _moments(f):
    out = []
    for p, q in ((0, 0), (1, 0), (0, 1), (2, 0), (0, 2), (1, 1), (2, 1), (1, 2), (2, 2)):
        out.append(sum(f[i] * (EX[i] ** p * EY[i] ** q) for i in range(9) if EX[i] ** p * EY[i] ** q))
    return out


def _meq(rho, u, v, phi):
    return [rho, rho * u, rho * v, rho / 3 + rho * u * u / phi, rho / 3 + rho * v * v / phi, rho * u * v / phi,
            rho * v / 3 + rho * u * u * v / phi, rho * u / 3 + rho * u * v * v / phi,
            rho / 9 + rho * (u * u + v * v) / (3 * phi) + rho * (u * v / phi) ** 2]


def _geq(T, u, v, sigma, c2):
    return _g_from([sigma * T, u * T, v * T, (c2 + u * u) * T, (c2 + v * v) * T])


def _g_from(n):
    return [n[0] - n[3] - n[4], (n[3] + n[1]) / 2, (n[4] + n[2]) / 2, (n[3] - n[1]) / 2, (n[4] - n[2]) / 2]


def _shift(u, v, p, m, sign):
    """N m of the porous central-moment shift (sign -1) or its inverse (sign +1)."""
    x, y = sign * u, sign * v
    return [m[0], x * m[0] + m[1], y * m[0] + m[2], x * x / p * m[0] + 2 * x / p * m[1] + m[3],
            y * y / p * m[0] + 2 * y / p * m[2] + m[4], (x * y * m[0] + y * m[1] + x * m[2]) / p + m[5],
            (x * x * y * m[0] + 2 * x * y * m[1] + x * x * m[2]) / p + y * m[3] + 2 * x * m[5] + m[6],
            (x * y * y * m[0] + y * y * m[1] + 2 * x * y * m[2]) / p + x * m[4] + 2 * y * m[5] + m[7],
            ((x * y) ** 2 * m[0] + 2 * x * y * y * m[1] + 2 * x * x * y * m[2]) / p ** 2
            + (y * y * m[3] + x * x * m[4] + 4 * x * y * m[5] + 2 * y * m[6] + 2 * x * m[7]) / p + m[8]]


class _Reference:
    def __init__(self, c, phi, fields):
        nx, ny, Ra, Pr = c["nx"], c["ny"], c["Ra"], c["Pr"]
        self.c, self.phi, L = c, phi, ny - 1.0
        inv = 0.5 + 0.1 * L * math.sqrt(3 * Pr / Ra)
        self.sv, self.c2, self.sigma = 1 / inv, 0.125, c["sigma"]
        self.sb = self.sv if self.sv >= 1.2 else 1.2
        self.nu = (inv - 0.5) / 3
        self.za = 1 / (0.5 + self.nu / (self.c2 * Pr))
        self.K = c["Da"] * L * L
        self.gb = Ra * self.nu * (self.nu / Pr) / L ** 3
        self.ax = 0.0 if c["walls"] == "cavity" else AX
        self.l1 = phi * (1.75 / torch.sqrt(150 * phi ** 3)) / (2 * math.sqrt(self.K)) if c["forchheimer"] else 0 * phi
        rho, u, v, T = fields
        self.f, self.g = _from_moments(_meq(rho, u, v, phi)), _geq(T, u, v, self.sigma, self.c2)
        self._macros()

    def _macros(self):
        """(rho, u, v, T) of all nodes; wall nodes are rebuilt by non-equilibrium extrapolation."""
        f, g, phi = self.f, self.g, self.phi
        rho, T = sum(f), sum(g) / self.sigma
        vx = sum(f[i] * EX[i] for i in range(1, 9) if EX[i]) / rho + 0.5 * phi * self.ax
        vy = sum(f[i] * EY[i] for i in range(1, 9) if EY[i]) / rho + 0.5 * phi * self.gb * (T - 0.5)
        l0 = 0.5 * (1 + phi * self.nu / (2 * self.K))
        den = l0 + torch.sqrt(l0 * l0 + self.l1 * torch.sqrt(vx * vx + vy * vy))
        u, v = vx / den, vy / den
        w = self.c["walls"]
        if w != "periodic":
            # sides in turn, corners with the W/E walls (their velocity, an isothermal wall first); sources are interior
            ix = (lambda a, s: a) if w == "channel" else (lambda a, s: a[s])
            todo = [(2, 0), (3, -1)] + ([(0, 0), (1, -1)] if w == "cavity" else [])
            neq = [a - b for a, b in zip(f + g, _from_moments(_meq(rho, u, v, phi)) + _geq(T, u, v, self.sigma, self.c2))]
            rho, u, v, T = rho.clone(), u.clone(), v.clone(), T.clone()
            n = T.shape[1]
            xs = torch.arange(n, device=T.device)
            if w == "cavity":
                xs = xs.clamp(1, n - 2)
            m = T.shape[0]
            ys = torch.arange(1, m - 1, device=T.device)
            T0 = T.clone()
            for side, e in todo:
                s, ss = (1, 2) if e == 0 else (-2, -3)
                tw, lid = WALL_T[w][side], LID if (w == "channel" and side == 3) else 0.0
                if side >= 2:
                    dst, src = (e, slice(None)), (s, xs)
                    xx = xs.clone()
                    if w == "cavity":   # corners: the diagonal neighbour, and T of the W/E walls
                        xx[0], xx[-1] = 2, n - 3
                    Tb = tw if tw is not None else (4 * T0[s][xs] - T0[ss][xx]) / 3
                else:
                    dst, src = (ys, e), (ys, s)
                    Tb = tw if tw is not None else (4 * T0[ys, s] - T0[ys, ss]) / 3
                rho[dst], u[dst], v[dst], T[dst] = rho[src], lid, 0.0, Tb
                if side >= 2 and w == "cavity":
                    T[e, 0], T[e, -1] = WALL_T[w][0], WALL_T[w][1]
                fb = _from_moments(_meq(rho[dst], u[dst], v[dst], phi[dst])) + _geq(T[dst], u[dst], v[dst], self.sigma, self.c2)
                for a, b, d in zip(f + g, fb, neq):
                    a[dst] = b + d[src]
        self.now = (rho, u, v, T)

    def step(self):
        c, p, f, g = self.c, self.phi, self.f, self.g
        rho, u, v, T = self.now
        um = torch.sqrt(u * u + v * v)
        drag = p * self.nu / self.K + 2 * self.l1 * um
        Fx, Fy = -drag * u + p * self.ax, -drag * v + p * self.gb * (T - 0.5)
        m = _moments(f)
        sp, sm = (self.sb + self.sv) / 2, (self.sb - self.sv) / 2
        rates = (1.0, 1.0, 1.0, None, None, self.sv, 1.2, 1.2, 1.8)
        if c["shift"]:
            mt = _shift(u, v, p, m, -1)
            eq = [rho, 0, 0, rho / 3, rho / 3, 0, 0, 0, rho / 9]
            S = [0, rho * Fx, rho * Fy, 0, 0, 0, rho * Fy / 3, rho * Fx / 3, 0]
        else:
            mt, eq = m, _meq(rho, u, v, p)
            S = [0, rho * Fx, rho * Fy, 2 * rho * u * Fx / p, 2 * rho * v * Fy / p, rho * (u * Fy + v * Fx) / p,
                 rho * Fy / 3 + rho * (Fy * u * u + 2 * Fx * u * v) / p, rho * Fx / 3 + rho * (Fx * v * v + 2 * Fy * u * v) / p,
                 2 / 3 * rho * (u * Fx + v * Fy) / p + 2 * rho * u * v * (Fx * v + Fy * u) / p ** 2]
        d = [a - b for a, b in zip(mt, eq)]
        new = [a if r is None else a - r * b + (1 - r / 2) * s for a, b, s, r in zip(mt, d, S, rates)]
        new[3] = mt[3] - sp * d[3] - sm * d[4] + S[3] - (sp * S[3] + sm * S[4]) / 2
        new[4] = mt[4] - sm * d[3] - sp * d[4] + S[4] - (sm * S[3] + sp * S[4]) / 2
        f = _from_moments(_shift(u, v, p, new, +1) if c["shift"] else new)
        n1, n2, c2, k = g[1] - g[3], g[2] - g[4], self.c2, 1 - self.za
        a1, a2 = self.za * u * T + k * n1, self.za * v * T + k * n2
        if c["shift"]:
            n = [sum(g), a1, a2, (c2 - u * u) * T + 2 * u * a1, (c2 - v * v) * T + 2 * v * a2]
        else:
            n = [sum(g), a1, a2, (c2 + u * u) * T, (c2 + v * v) * T]
        roll = lambda a, i: torch.roll(a, (EY[i], EX[i]), (0, 1))   # noqa: E731
        self.f = [roll(a, i) for i, a in enumerate(f)]
        self.g = [roll(a, i) for i, a in enumerate(_g_from(n))]
        self._macros()


def _net64(X, n, s, target=None):
    """The network in 64 bits on its stored weights: output, and with a target the loss and the gradients, laid out as
    Net.grads (channels padded with zeros to multiples of 32, the decoder's two inputs each)."""
    F, z = torch.nn.functional, np.load(WEIGHTS)
    pad = lambda k: (k + 31) // 32 * 32   # noqa: E731
    W, B = [], []
    for i, (a, b, _) in enumerate(LAYERS):
        k = 3 if i < 14 else 1
        w = torch.from_numpy(z["w%d" % i]).view(torch.bfloat16).double().cuda()
        W.append(w.reshape(k, k, a, b).permute(3, 2, 0, 1).contiguous().requires_grad_(target is not None))
        B.append(torch.from_numpy(z["b%d" % i]).double().cuda().requires_grad_(target is not None))
    conv = lambda i, x: F.relu(F.conv2d(x, W[i], B[i], padding=1))   # noqa: E731
    up = lambda x: F.interpolate(x, scale_factor=2, mode="nearest")   # noqa: E731
    e1 = conv(1, conv(0, X.double().permute(0, 3, 1, 2)))
    e2 = conv(3, conv(2, F.avg_pool2d(e1, 2)))
    e3 = conv(5, conv(4, F.avg_pool2d(e2, 2)))
    x = conv(7, conv(6, F.avg_pool2d(e3, 2)))
    x = conv(9, conv(8, torch.cat([up(x), e3], 1)))
    x = conv(11, conv(10, torch.cat([up(x), e2], 1)))
    x = conv(13, conv(12, torch.cat([up(x), e1], 1)))
    out = F.conv2d(x, W[14], B[14]).permute(0, 2, 3, 1)
    if target is None:
        return out
    loss = ((out - target.double()) ** 2).mean()
    loss.backward()
    two = {8: (192, 96), 10: (96, 48), 12: (48, 24)}
    flat = []
    for i, (a, b, _) in enumerate(LAYERS):
        parts = two.get(i, (a,))
        rows = [j + sum(map(pad, parts[:q])) for q, part in enumerate(parts) for j in range(part)]
        bp = pad(b) if i < 14 else b
        w = torch.zeros((9 if i < 14 else 1, sum(map(pad, parts)), bp), dtype=torch.float64, device="cuda")
        w[:, rows, :b] = W[i].grad.permute(2, 3, 1, 0).reshape(-1, a, b)
        flat += [w.reshape(-1), F.pad(B[i].grad, (0, bp - b))]
    return {"out": out.detach(), "loss": loss.detach().reshape(1), "grads": torch.cat(flat)}


def exact(case, seed):
    c = case
    if c["kind"] == "march":
        if c["nx"] * c["ny"] * c["steps"] > 2.5e9:
            return None
        ref = _Reference(c, *_start(c, seed))
        was = [a.clone() for a in ref.now]
        for _ in range(c["steps"]):
            ref.step()
        res = {"fields": list(ref.now)}
        if c["residual"]:
            d = [float((a - b).square().sum()) for a, b in zip(ref.now, was)]
            q = [float(a.square().sum()) for a in ref.now]
            res["residual"] = [math.sqrt((d[1] + d[2]) / (q[1] + q[2])), math.sqrt(d[3] / q[3])]
        return res
    if c["kind"] == "batch":
        return None   # hundreds of small runs one after the other: far over 20 seconds
    if c["kind"] == "conv":
        s = prepare(c, seed)
        x = s["x"].double().permute(0, 3, 1, 2).contiguous()
        w = s["w"].double().reshape(3, 3, c["cin"], c["cout"]).permute(3, 2, 0, 1).contiguous()
        dy = s["dy"].double().permute(0, 3, 1, 2).contiguous()
        y = torch.nn.functional.conv2d(x, w, s["b"].double(), padding=1).clamp_min(0).permute(0, 2, 3, 1)
        dx = torch.nn.functional.conv_transpose2d(dy, w, padding=1).where(x > 0, torch.zeros_like(x))
        dw = torch.stack([torch.einsum("nchw,nohw->co", torch.nn.functional.pad(x, (1, 1, 1, 1))
                                       [:, :, i:i + c["size"], j:j + c["size"]], dy) for i in range(3) for j in range(3)])
        return {"y": y, "dx": dx.permute(0, 2, 3, 1), "dw": dw.reshape(-1, c["cout"]), "db": dy.sum((0, 2, 3))}
    s = prepare(c, seed)
    if c["kind"] == "predict":
        X = torch.from_numpy(s["X"]).cuda().bfloat16()
        return _net64(X, c["n"], c["size"])
    return _net64(s["x"], c["n"], c["size"], s["y"])
