"""Learned warm start for the porous-cavity time march.

A small convolutional neural operator (U-Net-like, four levels, ~1.1 M
parameters) maps the porosity field and (Ra, Da, Pr, sigma) of a cavity to
its steady (u, v, T) and density.  Its prediction initialises the LB time march
(clb_set_fields); the time march itself is unchanged, so the converged
answer is the solver's, and the plain cold start remains the fallback.

Every forward and backward pass runs in the library's kernels
(include/clb_nop.h): implicit-GEMM convolutions on the BF16 tensor cores
with FP32 accumulation, pooling, upsampling, concatenation, loss and Adam.
PyTorch only provides device memory and the stream.

Network (NHWC, BF16 activations, ReLU after every 3x3 convolution):
  enc1 128^2: 8 -> 24 -> 24        enc2 64^2: 24 -> 48 -> 48
  enc3 32^2: 48 -> 96 -> 96        bottom 16^2: 96 -> 192 -> 192
  dec3 32^2: [up 192 | 96] -> 96 -> 96
  dec2 64^2: [up 96 | 48] -> 48 -> 48
  dec1 128^2: [up 48 | 24] -> 24 -> 24       head: 1x1, 24 -> 4 (FP32)
"""
from __future__ import annotations

import ctypes
import math
from dataclasses import dataclass

import numpy as np

from . import clb

U_C = 0.1 / math.sqrt(3.0)     # characteristic velocity Ma c_s of Eq. 46, lattice units
# Boussinesq pressure variation across the cavity ~ g beta dT L = u_c^2, i.e.
# a density variation of ~3 u_c^2 = 0.01.
RHO_SCALE = 0.01
N_IN, N_OUT = 8, 4

_VP = ctypes.c_void_p


class AdamSeg(ctypes.Structure):
    """clb_nop_adam_seg of include/clb_nop.h."""
    _fields_ = [("w", _VP), ("g", _VP), ("m", _VP), ("v", _VP), ("wb", _VP), ("wbt", _VP), ("n", ctypes.c_int64),
                ("rows", ctypes.c_int32), ("cols", ctypes.c_int32)]


class NopLayer(ctypes.Structure):
    """clb_nop_layer of include/clb_nop.h."""
    _fields_ = [("w", _VP), ("wt", _VP), ("bias", _VP), ("cin", ctypes.c_int32), ("cout", ctypes.c_int32),
                ("taps", ctypes.c_int32), ("relu", ctypes.c_int32)]


def _lib():
    L = clb.load()
    if not getattr(L, "_nop_ready", False):
        i32, i64, f32 = ctypes.c_int32, ctypes.c_int64, ctypes.c_float
        L.clb_nop_conv_fwd.argtypes = [_VP, _VP, _VP, _VP, _VP, i32, i32, i32, i32, i32, i32, i32, i32, _VP]
        L.clb_nop_conv_dgrad.argtypes = [_VP, _VP, _VP, _VP, i32, i32, i32, i32, i32, i32, _VP]
        L.clb_nop_conv_wgrad.argtypes = [_VP, _VP, _VP, i32, i32, i32, i32, i32, i32, i32, _VP]
        L.clb_nop_conv_wgrad_bias.argtypes = [_VP, _VP, _VP, _VP, i32, i32, i32, i32, i32, i32, i32, _VP]
        L.clb_nop_bias_grad.argtypes = [_VP, _VP, i64, i32, _VP]
        L.clb_nop_pool2.argtypes = [_VP, _VP, i32, i32, i32, i32, i32, _VP]
        L.clb_nop_up2.argtypes = [_VP, _VP, i32, i32, i32, i32, i32, _VP]
        L.clb_nop_concat.argtypes = [_VP, _VP, _VP, i64, i32, i32, i32, _VP]
        L.clb_nop_mse.argtypes = [_VP, _VP, _VP, i32, _VP, _VP, i64, _VP]
        L.clb_nop_adam.argtypes = [_VP, _VP, _VP, _VP, _VP, i64, f32, f32, f32, f32, i32, _VP]
        L.clb_nop_adam_multi.argtypes = [ctypes.POINTER(AdamSeg), i32, f32, f32, f32, f32, i32, _VP]
        L.clb_nop_cast_bf16.argtypes = [_VP, _VP, i64, _VP]
        L.clb_nop_zero.argtypes = [_VP, i64, _VP]
        L.clb_nop_transpose.argtypes = [_VP, _VP, i32, i32, _VP]
        L.clb_nop_check.argtypes = [_VP]
        L.clb_nop_wait_selftest.argtypes = [i64, _VP]
        L.clb_nop_add_mask.argtypes = [_VP, _VP, _VP, _VP, i64, _VP]
        L.clb_nop_net_acts.argtypes = [ctypes.POINTER(NopLayer), i32, i32, i32, ctypes.POINTER(i64)]
        L.clb_nop_net_acts.restype = i64
        L.clb_nop_net_forward.argtypes = [ctypes.POINTER(NopLayer), _VP, i32, _VP, _VP, i32, i32, i32, _VP]
        L.clb_nop_net_forward.restype = ctypes.c_int
        L.clb_nop_net_scratch.argtypes = [ctypes.POINTER(NopLayer), i32, i32, i32]
        L.clb_nop_net_scratch.restype = i64
        pvp = ctypes.POINTER(_VP)
        L.clb_nop_net_backward.argtypes = [ctypes.POINTER(NopLayer), pvp, pvp, pvp, _VP, _VP, i32, i32, i32, _VP, _VP]
        L.clb_nop_net_backward.restype = ctypes.c_int
        L._nop_ready = True
    return L


def _ok(rc, what):
    if rc != 0:
        raise RuntimeError(f"{what} failed with status {rc}")


def _p(t):
    return None if t is None else t.data_ptr()


# ------------------------------------------------------------------ features
def features(phi: np.ndarray, Ra: float, Da: float, Pr: float, sigma: float) -> np.ndarray:
    """(H, W, 8) network input: normalised porosity, log10 Ra, log10 Da, Pr,
    sigma (broadcast), the two node coordinates and the mean porosity
    (broadcast).  Eight channels keep every layer's channel count a
    multiple of 8, the tensor-core path's granule."""
    phi = np.asarray(phi, dtype=np.float32)
    h, w = phi.shape
    out = np.empty((h, w, N_IN), dtype=np.float32)
    out[..., 0] = (phi - 0.65) / 0.15
    out[..., 1] = (math.log10(Ra) - 4.5) / 0.87
    out[..., 2] = (math.log10(Da) + 2.5) / 0.87
    out[..., 3] = (Pr - 0.85) / 0.087
    out[..., 4] = (sigma - 1.25) / 0.43
    out[..., 5] = np.linspace(-0.5, 0.5, w, dtype=np.float32)[None, :]
    out[..., 6] = np.linspace(-0.5, 0.5, h, dtype=np.float32)[:, None]
    out[..., 7] = (float(phi.mean()) - 0.65) / 0.15
    return out


def conduction_T(h: int, w: int, T_hot: float = 1.0, T_cold: float = 0.0) -> np.ndarray:
    """Pure-conduction temperature between the west (hot) and east (cold)
    wall nodes, x = 0 and x = w - 1: the Ra -> 0 limit of the cavity."""
    x = np.arange(w, dtype=np.float64) / (w - 1)
    return np.broadcast_to(T_hot + (T_cold - T_hot) * x, (h, w))


def _scale_terms(Ra, Da, Pr, sigma, eps_mean):
    a, d = math.log10(Ra), math.log10(Da)
    return np.array([1.0, a, d, math.log10(Pr), math.log10(sigma), eps_mean, a * a, d * d, a * d])


def fit_velocity_scale(params, u_rms):
    """Least-squares fit of log(u_rms / u_c) to a quadratic in (log10 Ra,
    log10 Da) plus linear terms in log10 Pr, log10 sigma and the mean
    porosity, over the training cases; params = [(Ra, Da, Pr, sigma, eps)]."""
    A = np.stack([_scale_terms(*p) for p in params])
    coef, *_ = np.linalg.lstsq(A, np.log(np.asarray(u_rms) / U_C), rcond=None)
    return coef


def velocity_scale(coef, Ra, Da, Pr, sigma, eps_mean) -> float:
    """Predicted RMS speed of the steady flow (lattice units)."""
    return float(U_C * math.exp(float(_scale_terms(Ra, Da, Pr, sigma, eps_mean) @ coef)))


def targets(rho: np.ndarray, ux: np.ndarray, uy: np.ndarray, T: np.ndarray, vscale: float) -> np.ndarray:
    """(H, W, 4) normalised steady fields: u / vscale, v / vscale,
    (T - T_conduction) / 0.5, (rho - mean rho) / RHO_SCALE.  Only density
    differences are learned: the walls' extrapolation leaks mass slowly, so
    the mean density of a converged run depends on its history."""
    Tc = conduction_T(*T.shape)
    return np.stack([ux / vscale, uy / vscale, (T - Tc) / 0.5, (rho - rho.mean()) / RHO_SCALE],
                    axis=-1).astype(np.float32)


def fields_from(pred: np.ndarray, vscale: float):
    """Inverse of targets(): (rho, ux, uy, T) in lattice units, mean density 1
    (the mass of the fluid at rest)."""
    pred = np.asarray(pred, dtype=np.float64)
    Tc = conduction_T(*pred.shape[:2])
    d = pred[..., 3] - pred[..., 3].mean()
    return (1.0 + RHO_SCALE * d, pred[..., 0] * vscale, pred[..., 1] * vscale, Tc + 0.5 * pred[..., 2])


def augment_rot180(X: np.ndarray, Y: np.ndarray):
    """Centro-symmetric copies of (features, targets).  With the hot wall at
    x = 0, the cold one at x = L, adiabatic top and bottom and buoyancy about
    T0 = (T_hot + T_cold) / 2, the Boussinesq Brinkman-Forchheimer equations
    map a solution (u, T, p)(x) on porosity eps(x) to (-u, 1 - T, p)(R x) on
    eps(R x), R the rotation by 180 degrees about the centre: velocities and
    the temperature deviation change sign, the pressure does not."""
    Xr = X.copy()
    Xr[..., 0] = X[:, ::-1, ::-1, 0]
    Yr = Y[:, ::-1, ::-1, :] * np.array([-1.0, -1.0, -1.0, 1.0], dtype=np.float32)
    return Xr, np.ascontiguousarray(Yr)


def peclet(vscale: float, nu: float, Pr: float, L: float) -> float:
    """Peclet number u L / alpha of the predicted flow (alpha = nu / Pr)."""
    return vscale * L * Pr / nu


# ------------------------------------------------------------------ layers
# Activations carry their channels padded with zeros to multiples of 32: the
# TMA-fed convolutions copy 32- or 64-channel boxes, and a box that runs past
# the last channel (24 of 32, say) is filled by the hardware at a large cost
# (a 24 -> 24 layer at 16 x 128^2 takes 55 us, a 32 -> 32 one 27 us).  The
# padding weights and biases are zero and stay zero (their gradients are
# exactly zero), so the padded network computes the same function as the
# real one; saved weights hold the real parts only.
def _pad32(c: int) -> int:
    return (c + 31) // 32 * 32


class Conv:
    """One convolution: FP32 master weights [taps * cin][cout] (cin, cout
    padded), BF16 copy and its transpose, FP32 bias, gradients and Adam
    moments.  rin: the padded positions of the real input channels;
    cout_real: the real outputs (the first ones)."""

    def __init__(self, torch, rin, cin, cout_real, taps, relu, rng, pad_out=True):
        self._torch = torch
        self.rin = np.asarray(list(rin), dtype=np.int64)
        self.cin_real, self.cout_real = len(self.rin), cout_real
        self.cin, self.cout, self.taps, self.relu = cin, (_pad32(cout_real) if pad_out else cout_real), taps, relu
        fan = taps * self.cin_real
        std = math.sqrt((2.0 if relu else 1.0) / fan)
        w = self.embed(rng.standard_normal((taps * self.cin_real, cout_real)).astype(np.float32) * std)
        dev = "cuda"
        self.w = torch.from_numpy(w).to(dev)
        self.wb = torch.empty(w.shape, dtype=torch.bfloat16, device=dev)
        self.b = torch.zeros(self.cout, dtype=torch.float32, device=dev)
        self.gw = torch.zeros_like(self.w)
        self.gb = torch.zeros_like(self.b)
        self.mw, self.vw = torch.zeros_like(self.w), torch.zeros_like(self.w)
        self.mb, self.vb = torch.zeros_like(self.b), torch.zeros_like(self.b)
        self.wbt = torch.empty((self.cout, taps * cin), dtype=torch.bfloat16, device=dev)   # for the forward
        _ok(_lib().clb_nop_cast_bf16(_p(self.w), _p(self.wb), self.w.numel(), None), "cast")
        self.refresh_t()

    def embed(self, real: np.ndarray) -> np.ndarray:
        """[taps * cin_real][cout_real] -> the padded [taps * cin][cout], zeros elsewhere."""
        out = np.zeros((self.taps, self.cin, self.cout), dtype=real.dtype)
        out[:, self.rin, :self.cout_real] = real.reshape(self.taps, self.cin_real, self.cout_real)
        return out.reshape(self.taps * self.cin, self.cout)

    def real(self, t):
        """The real part [taps * cin_real][cout_real] of a padded weight-shaped tensor."""
        idx = self._torch.as_tensor(self.rin, device=t.device)
        v = t.reshape(self.taps, self.cin, self.cout)[:, idx, :self.cout_real]
        return v.reshape(self.taps * self.cin_real, self.cout_real)

    def refresh_t(self):
        """Rebuild the transposed BF16 copy from the BF16 weights."""
        _ok(_lib().clb_nop_transpose(_p(self.wb), _p(self.wbt), self.taps * self.cin, self.cout, None), "transpose")

    @property
    def nparams(self):
        return self.taps * self.cin_real * self.cout_real + self.cout_real


@dataclass
class Net:
    layers: list
    torch: object
    scale_coef: object = None      # velocity-scale fit (fit_velocity_scale), stored with the weights

    @classmethod
    def create(cls, torch, seed=0, width=(24, 48, 96, 192), cin=N_IN, cout=N_OUT):
        rng = np.random.default_rng(seed)
        c1, c2, c3, c4 = width
        P = _pad32
        r = lambda c: range(c)
        cat = lambda a, b: list(range(a)) + [P(a) + j for j in range(b)]   # [up(a) | skip(b)], each padded
        spec = [(r(cin), P(cin), c1), (r(c1), P(c1), c1), (r(c1), P(c1), c2), (r(c2), P(c2), c2),
                (r(c2), P(c2), c3), (r(c3), P(c3), c3), (r(c3), P(c3), c4), (r(c4), P(c4), c4),
                (cat(c4, c3), P(c4) + P(c3), c3), (r(c3), P(c3), c3), (cat(c3, c2), P(c3) + P(c2), c2),
                (r(c2), P(c2), c2), (cat(c2, c1), P(c2) + P(c1), c1), (r(c1), P(c1), c1)]
        layers = [Conv(torch, ri, ci, co, 9, True, rng) for ri, ci, co in spec]
        layers.append(Conv(torch, r(c1), P(c1), cout, 1, False, rng, pad_out=False))
        net = cls(layers, torch)
        net.n_in = cin
        net._flat_grads()
        return net

    def _flat_grads(self):
        """All weight and bias gradients as views of one buffer (cleared by
        one call per backward pass), and the Adam segment table."""
        t = self.torch
        total = sum(l.gw.numel() + l.gb.numel() for l in self.layers)
        self.grads = t.zeros(total, dtype=t.float32, device="cuda")
        off = 0
        for l in self.layers:
            n = l.gw.numel()
            l.gw = self.grads[off:off + n].view(l.w.shape)
            off += n
            l.gb = self.grads[off:off + l.b.numel()]
            off += l.b.numel()
        segs = []
        for l in self.layers:
            segs.append(AdamSeg(_p(l.w), _p(l.gw), _p(l.mw), _p(l.vw), _p(l.wb), _p(l.wbt), l.w.numel(),
                                l.taps * l.cin, l.cout))
            segs.append(AdamSeg(_p(l.b), _p(l.gb), _p(l.mb), _p(l.vb), None, None, l.b.numel(), 1, l.b.numel()))
        self._segs = (AdamSeg * len(segs))(*segs)

    @property
    def nparams(self):
        return sum(l.nparams for l in self.layers)

    # resolution divisor of each layer (forward order)
    RES = (1, 1, 2, 2, 4, 4, 8, 8, 4, 4, 2, 2, 1, 1, 1)

    def train_flops(self, n, h, w):
        """Tensor-core FLOPs of one training step: forward, input gradient
        (all layers but the first) and weight gradient of every convolution."""
        tot = 0
        for i, (l, d) in enumerate(zip(self.layers, self.RES)):
            one = 2.0 * n * (h // d) * (w // d) * l.taps * l.cin_real * l.cout_real   # real channels
            tot += one * (2 if i == 0 else 3)
        return tot

    # activations the forward pass keeps, in the library's order: name (a number:
    # the output of that layer), the layer whose channel count it has (in: its
    # input's), resolution divisor
    ACTS = (("x", 0, True, 1), (1, 0, False, 1), (2, 1, False, 1), ("p1", 1, False, 2), (3, 2, False, 2), (4, 3, False, 2),
            ("p2", 3, False, 4), (5, 4, False, 4), (6, 5, False, 4), ("p3", 5, False, 8), (7, 6, False, 8), (8, 7, False, 8),
            ("c3", 8, True, 4), (9, 8, False, 4), (10, 9, False, 4), ("c2", 10, True, 2), (11, 10, False, 2),
            (12, 11, False, 2), ("c1", 12, True, 1), (13, 12, False, 1), (14, 13, False, 1))

    def _table(self):
        """The library's layer table, rebuilt when a layer's tensors have moved."""
        key = [(_p(l.wb), _p(l.wbt), _p(l.b)) for l in self.layers]
        if getattr(self, "_tab_key", None) != key:
            self._tab = (NopLayer * len(self.layers))(*[NopLayer(*k, l.cin, l.cout, l.taps, int(l.relu))
                                                        for k, l in zip(key, self.layers)])
            self._tab_key = key
        return self._tab

    def _run(self, x, n, h, w):
        """The forward pass by one library call: (output, buffer of all activations, their offsets)."""
        t, lib, tab = self.torch, _lib(), self._table()
        off = (ctypes.c_int64 * len(self.ACTS))()
        size = lib.clb_nop_net_acts(tab, n, h, w, off)
        if size <= 0:
            raise RuntimeError(f"the network does not take {n} images of {h} x {w}")
        buf = t.empty(size // 2, dtype=t.bfloat16, device="cuda")
        out = t.empty((n, h, w, self.layers[-1].cout), dtype=t.float32, device="cuda")
        _ok(lib.clb_nop_net_forward(tab, _p(x), self.n_in, _p(buf), _p(out), n, h, w, None), "net_forward")
        return out, buf, off

    def forward(self, x, n, h, w):
        """x: (n, h, w, 8) BF16 device tensor -> (n, h, w, 4) FP32, plus the
        activations the backward pass needs (channels padded to multiples of 32)."""
        out, buf, off = self._run(x, n, h, w)
        A = {}
        for (name, l, is_in, d), o in zip(self.ACTS, off):
            c = self.layers[l].cin if is_in else self.layers[l].cout
            shape = (n, h // d, w // d, c)
            A[name] = buf[o // 2:o // 2 + math.prod(shape)].view(shape)
        return out, A

    # ---- backward
    def backward(self, dout, A, n, h, w):
        """Accumulates every layer's weight and bias gradient (cleared first)
        from the gradient of the output and the activations of forward()."""
        t, lib, tab = self.torch, _lib(), self._table()
        if getattr(self, "_ws", None) is None:
            self._ws = t.cuda.Stream()      # the weight gradients run beside the input-gradient chain
        _ok(lib.clb_nop_zero(_p(self.grads), self.grads.numel() * 4, None), "zero")
        nl = len(self.layers)
        gw, gb = (_VP * nl)(*[_p(l.gw) for l in self.layers]), (_VP * nl)(*[_p(l.gb) for l in self.layers])
        acts = (_VP * len(self.ACTS))(*[_p(A[name]) for name, *_ in self.ACTS])
        scratch = t.empty(lib.clb_nop_net_scratch(tab, n, h, w) // 2, dtype=t.bfloat16, device="cuda")
        _ok(lib.clb_nop_net_backward(tab, gw, gb, acts, _p(dout), _p(scratch), n, h, w, None,
                                     _VP(self._ws.cuda_stream)), "net_backward")

    def adam(self, step, lr, b1=0.9, b2=0.999, eps=1e-8):
        # one launch: every layer's weights (BF16 copy and its transpose refreshed) and biases
        _ok(_lib().clb_nop_adam_multi(self._segs, len(self._segs), lr, b1, b2, eps, step, None), "adam")

    def loss_and_grad(self, out, target, weights=None):
        """Channel-weighted MSE and its gradient (weights: device FP32, one per
        output channel, or None)."""
        t = self.torch
        loss = t.zeros(1, dtype=t.float32, device="cuda")
        g = t.empty(out.shape, dtype=t.bfloat16, device="cuda")
        _ok(_lib().clb_nop_mse(_p(out), _p(target), _p(weights), out.shape[-1], _p(g), _p(loss), out.numel(), None),
            "mse")
        return loss, g

    def state(self):
        """Real weights [taps * cin][cout] and biases of every layer (FP32)."""
        return [(l.real(l.w).cpu().numpy(), l.b[:l.cout_real].cpu().numpy()) for l in self.layers]

    def save(self, path):
        """Real weights as BF16 bit patterns (what inference uses) and FP32 biases."""
        arrs = {"scale_coef": np.asarray(self.scale_coef if self.scale_coef is not None else [], dtype=np.float64)}
        for i, l in enumerate(self.layers):
            arrs[f"w{i}"] = l.real(l.wb).contiguous().view(self.torch.int16).cpu().numpy()
            arrs[f"b{i}"] = l.b[:l.cout_real].cpu().numpy()
        np.savez_compressed(path, **arrs)

    def load(self, path):
        z = np.load(path)
        t = self.torch
        self.scale_coef = z["scale_coef"] if len(z["scale_coef"]) else None
        for i, l in enumerate(self.layers):
            real = (l.taps * l.cin_real, l.cout_real)
            if z[f"w{i}"].shape != real:
                raise ValueError(f"layer {i}: stored shape {z[f'w{i}'].shape} != {real}")
            wr = t.from_numpy(z[f"w{i}"]).view(t.bfloat16).float().numpy()
            l.w.copy_(t.from_numpy(l.embed(wr)).to("cuda"))     # BF16 values, exact in FP32
            _ok(_lib().clb_nop_cast_bf16(_p(l.w), _p(l.wb), l.w.numel(), None), "cast")
            l.b.zero_()
            l.b[:l.cout_real].copy_(t.from_numpy(z[f"b{i}"]).to("cuda"))
            l.refresh_t()
        return self


def to_bf16(torch, arr: np.ndarray):
    """Host FP32 array -> device BF16 tensor, converted by the library."""
    x = torch.from_numpy(np.ascontiguousarray(arr, dtype=np.float32)).to("cuda")
    y = torch.empty(x.shape, dtype=torch.bfloat16, device="cuda")
    _ok(_lib().clb_nop_cast_bf16(_p(x), _p(y), x.numel(), None), "cast")
    return y


def train(net: Net, X: np.ndarray, Y: np.ndarray, epochs: int, batch: int = 16, lr: float = 2e-3,
          Xval=None, Yval=None, log=None, weights=None):
    """Adam on the channel-weighted mean squared error (cosine learning-rate
    decay); X: (N, H, W, 8), Y: (N, H, W, 4).  Returns the per-epoch
    (train, validation) losses."""
    torch = net.torch
    n, h, w, _ = X.shape
    wd = None if weights is None else torch.tensor(weights, dtype=torch.float32, device="cuda")
    Xd = to_bf16(torch, X)
    Yd = torch.from_numpy(np.ascontiguousarray(Y, dtype=np.float32)).to("cuda")
    hist = []
    step = 0
    rng = np.random.default_rng(1)
    nb = max(1, n // batch)
    total = epochs * nb
    for ep in range(epochs):
        perm = torch.from_numpy(rng.permutation(n)).to("cuda")
        tot = 0.0
        for b in range(nb):
            idx = perm[b * batch:(b + 1) * batch]
            xb, yb = Xd.index_select(0, idx).contiguous(), Yd.index_select(0, idx).contiguous()
            out, A = net.forward(xb, xb.shape[0], h, w)
            loss, g = net.loss_and_grad(out, yb, wd)
            net.backward(g, A, xb.shape[0], h, w)
            step += 1
            cur = lr * 0.5 * (1.0 + math.cos(math.pi * step / total))
            net.adam(step, cur)
            tot += float(loss.item())
        val = evaluate(net, Xval, Yval, weights) if Xval is not None else None
        hist.append((tot / nb, val))
        if log:
            log(f"epoch {ep + 1}/{epochs}: train {tot / nb:.4e}" + (f"  val {val:.4e}" if val is not None else ""))
    return hist


def predict(net: Net, X: np.ndarray, batch: int = 16) -> np.ndarray:
    torch = net.torch
    n, h, w, _ = X.shape
    outs = []
    for b in range(0, n, batch):
        xb = to_bf16(torch, X[b:b + batch])
        outs.append(net._run(xb, xb.shape[0], h, w)[0].cpu().numpy())
    return np.concatenate(outs, axis=0) if len(outs) != 1 else outs[0]


def warm_fields(net: Net, phi: np.ndarray, Ra: float, Da: float, Pr: float, sigma: float):
    """The network's steady (rho, ux, uy, T) for one cavity, in lattice
    units, ready for clb_set_fields."""
    X = features(phi, Ra, Da, Pr, sigma)[None]
    vs = velocity_scale(net.scale_coef, Ra, Da, Pr, sigma, float(np.mean(phi)))
    return fields_from(predict(net, X)[0], vs)


def evaluate(net: Net, X: np.ndarray, Y: np.ndarray, weights=None) -> float:
    """Channel-weighted mean squared error of the predictions."""
    P = predict(net, X)
    w = np.ones(Y.shape[-1]) if weights is None else np.asarray(weights, dtype=np.float64)
    return float(np.mean(np.mean((P - Y) ** 2, axis=(0, 1, 2)) * w))
