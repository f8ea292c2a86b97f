"""The work that users of this framework have it do, as cases that can be timed and compared.

Three kinds:

* ``lattice``  one lattice from its initial fields through some hundred time steps to the ten
  output fields: ``Lattice.init``, ``Lattice.step``, ``Lattice.moments`` (periodic or Dirichlet,
  with or without a body load, wall data and displacement tracking, every storage format);
* ``batch``    many lattices of uneven size and material advanced together (``lbm_batch_*``);
  ``solver``   is its regular form, the k-step map that trajectory generation and the surrogate's
  check evaluate (``surrogate.relift_and_step``);
* ``unet``     the surrogate network's forward pass on packed moment fields, and ``layer``, the
  backward pass of one of its convolutions.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2408_01081_gb300 import lbm as L
from paper_2408_01081_gb300 import nn as K
from paper_2408_01081_gb300 import surrogate as S

DEV = "cuda"
F64 = dict(dtype=torch.float64, device=DEV)

# U-Net layers by name: level, input channels (first and second tensor), output channels, whether
# the first input is stored at half size
LAYERS = {
    "enc0b": (0, 32, 0, 32, False), "enc1a": (1, 32, 0, 64, False), "enc1b": (1, 64, 0, 64, False),
    "enc2a": (2, 64, 0, 128, False), "enc2b": (2, 128, 0, 128, False), "enc3a": (3, 128, 0, 256, False),
    "enc3b": (3, 256, 0, 256, False), "dec2a": (2, 256, 128, 128, True), "dec2b": (2, 128, 0, 128, False),
    "dec1a": (1, 128, 64, 64, True), "dec1b": (1, 64, 0, 64, False), "dec0a": (0, 64, 32, 32, True),
    "dec0b": (0, 32, 0, 32, False),
}


def _lattice(name, nx, ny, storage, steps, bc="periodic", load=False, track=False):
    c = {"kind": "lattice", "nx": nx, "ny": ny, "storage": storage, "steps": steps, "bc": bc, "load": load,
         "track": track}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest run in earnest: the 64 x 64 periodic manufactured solution (1000 steps with a
        # body load and displacement tracking); every step is a launch of 4096 nodes
        _lattice("periodic_mms_64_f64", 64, 64, "f64", 1000, load=True, track=True),
        # the manufactured solution on the Dirichlet rectangle with wall data, as the convergence
        # sweep runs it on its middle lattices
        _lattice("dirichlet_mms_2048x1024_f64", 2048, 1024, "f64", 100, "dirichlet", True, True),
        # the same in FP32, on a lattice whose rows and columns fill no tile
        _lattice("dirichlet_mms_1021x515_f32", 1021, 515, "f32", 200, "dirichlet", True, True),
        # the long-run stability box (homogeneous Dirichlet, no body load), a state that fits the L2
        _lattice("dirichlet_box_512x256_f64", 512, 256, "f64", 1000, "dirichlet"),
        # the headline lattice in FP64, and in FP32, 16-bit populations and the moment-space format
        # that keeps FP32's error
        _lattice("periodic_8192_f64", 8192, 8192, "f64", 100),
        _lattice("periodic_8192_f32", 8192, 8192, "f32", 300),
        _lattice("periodic_8192_bf16", 8192, 8192, "bf16", 300),
        _lattice("periodic_4095x4001_msbfp", 4095, 4001, "ms_bfp", 300),
        # the ragged batch: half periodic, half Dirichlet, sides 64..1024 with aspect ratios up to 4
        {"name": "batch_128_f32", "kind": "batch", "count": 128, "smin": 64, "smax": 1024, "storage": "f32",
         "steps": 300},
        # the surrogate's solver check and training-data map: 16 periodic lattices of 256^2, 32 steps
        {"name": "solver_16x256_f64", "kind": "solver", "n": 16, "side": 256, "k": 32, "storage": "f64"},
        # the surrogate's inference on the same 16 lattices
        {"name": "unet_16x256", "kind": "unet", "B": 16, "side": 256, "act_bf16": False},
        # training: the backward pass of the network's 32-channel layer at full resolution
        {"name": "layer_backward_enc0b", "kind": "layer", "layer": "enc0b", "B": 8, "side": 256},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice"] * 6 + ["batch", "solver", "unet", "layer"])
    if kind == "lattice":
        storage = rng.choice(["f64", "f64", "f64", "f32", "f32", "bf16", "f16", "ms_bfp", "ms_f16"])
        small = 64 if storage == "f64" else 256
        nx, ny = _log(rng, small, 8192), _log(rng, small, 8192)
        if rng.random() < 0.5:
            nx -= nx % 64
        bc = rng.choice(["periodic", "dirichlet"])
        load = rng.random() < 0.4 and storage in ("f64", "f32")
        most = 2.5e9 if load else 6e9                    # nodes x steps, below the largest listed case
        steps = max(20, min(_log(rng, 50, 1000), int(most / (nx * ny))))
        return _lattice(None, nx, ny, storage, steps, bc, load, load)
    if kind == "batch":
        storage = rng.choice(["f32", "f32", "f64"])
        return {"kind": "batch", "count": _log(rng, 8, 128), "smin": 64, "smax": rng.choice([256, 512, 1024]),
                "storage": storage, "steps": rng.choice([32, 50, 64] if storage == "f64" else [50, 100, 128])}
    if kind == "solver":
        return {"kind": "solver", "n": rng.randint(1, 32), "side": rng.choice([64, 128, 256]),
                "k": rng.choice([16, 31, 32, 64]), "storage": rng.choice(["f64", "f64", "f32"])}
    if kind == "unet":
        return {"kind": "unet", "B": rng.randint(1, 16), "side": rng.choice([128, 256]),
                "act_bf16": rng.random() < 0.25}
    return {"kind": "layer", "layer": rng.choice(sorted(LAYERS)), "B": rng.randint(1, 16),
            "side": rng.choice([128, 256])}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _speeds(nu):
    """(cK, cmu) of a plane-strain Poisson ratio with cK^2 + cmu^2 = 2."""
    ratio = 1.0 / (1.0 - 2.0 * nu)
    cmu2 = 2.0 / (1.0 + ratio)
    return math.sqrt(2.0 - cmu2), math.sqrt(cmu2)


def _geometry(nx, ny, nu):
    """Spacing, time step (0.9 of the CFL-like bound) and wave speeds; the longer side has length 1."""
    cK, cmu = _speeds(nu)
    dx = 1.0 / max(nx, ny)
    return dx, dx * 0.9 / (2.0 * math.sqrt(2.0)), cK, cmu


def _random_field(nx, ny, ell, dx, gen, std=1e-3):
    """Periodic Gaussian random field of correlation length ell cells and its derivatives."""
    kx = 2.0 * math.pi * torch.fft.rfftfreq(nx, **F64)[None, :]
    ky = 2.0 * math.pi * torch.fft.fftfreq(ny, **F64)[:, None]
    W = torch.fft.rfft2(torch.randn((ny, nx), generator=gen, **F64))
    W *= torch.exp(-(kx * kx + ky * ky) * (ell * ell / 4.0))
    W[0, 0] = 0.0
    f = torch.fft.irfft2(W, s=(ny, nx))
    s = std / torch.sqrt((f * f).mean())
    kx[0, -1] = 0.0 if nx % 2 == 0 else kx[0, -1]
    ky[ny // 2] = 0.0 if ny % 2 == 0 else ky[ny // 2]
    fx = torch.fft.irfft2(W * (1j * kx), s=(ny, nx))
    fy = torch.fft.irfft2(W * (1j * ky), s=(ny, nx))
    return f * s, fx * (s / dx), fy * (s / dx)


def _rest_fields(nx, ny, dx, dirichlet, ell, gen):
    """U0, dU0/dx, dU0/dy of a lattice at rest with a random initial velocity that vanishes on the
    walls of a Dirichlet lattice."""
    U = torch.zeros((3, 5, ny, nx), **F64)
    for c in range(2):
        f, fx, fy = _random_field(nx, ny, ell, dx, gen)
        if dirichlet:
            xs, ys = (torch.arange(nx, **F64) + 0.5) / nx, (torch.arange(ny, **F64) + 0.5) / ny
            wx, wy = torch.sin(math.pi * xs)[None, :], torch.sin(math.pi * ys)[:, None]
            dwx = (math.pi / (nx * dx)) * torch.cos(math.pi * xs)[None, :]
            dwy = (math.pi / (ny * dx)) * torch.cos(math.pi * ys)[:, None]
            fx, fy = fx * (wx * wy) + f * (wy * dwx), fy * (wx * wy) + f * (dwy * wx)
            f = f * (wx * wy)
        U[0, c], U[1, c], U[2, c] = f, fx, fy
    return U


def _loaded_fields(case, dx, dt, rng):
    """A manufactured-type run with body load: smooth initial fields and displacement (products of
    sines and cosines of one wavelength per unit length, amplitude 1e-2), the body load and the
    wall velocity as separable tables of four terms with an oscillation in time."""
    nx, ny, steps = case["nx"], case["ny"], case["steps"]
    k, w, amp = 2.0 * math.pi, 4.0 * math.pi, 1e-2
    xs, ys = (np.arange(nx) + 0.5) * dx, (np.arange(ny) + 0.5) * dx
    xw, yw = np.array([0.0, nx * dx]), np.array([0.0, ny * dx])

    def basis(s, first):
        return np.stack([np.sin(k * s), np.sin(k * s), np.cos(k * s), np.cos(k * s)] if first else
                        [np.sin(k * s), np.cos(k * s), np.sin(k * s), np.cos(k * s)])

    def slope(s, first):
        c, m = k * np.cos(k * s), -k * np.sin(k * s)
        return np.stack([c, c, m, m] if first else [c, m, c, m])

    def times(t, scale):
        ph = rng.uniform(0.0, 2.0 * math.pi, (2, 4))
        am = scale * rng.uniform(0.5, 1.0, (2, 4)) * rng.choice([-1.0, 1.0], (2, 4))
        return am * np.cos(w * t[:, None, None] + ph)

    def dense(C, X, Y):
        X, Y, C = (torch.as_tensor(v, **F64) for v in (X, Y, C))
        return torch.einsum("rx,ry,cr->cyx", X, Y, C).contiguous()

    C = rng.uniform(-1.0, 1.0, (5, 4)) * amp * np.array([w, w, k, k, k])[:, None]
    X, Y = basis(xs, True), basis(ys, False)
    T = times(np.arange(steps + 1) * dt, amp * w * w)
    return {
        "U0": dense(C, X, Y), "Ux": dense(C, slope(xs, True), Y), "Uy": dense(C, X, slope(ys, False)),
        "u0": dense(rng.uniform(-amp, amp, (2, 4)), X, Y), "B0": dense(T[0], X, Y), "load": (X, Y, T),
        "wall": (X, basis(xw, True), Y, basis(yw, False), times((np.arange(steps) + 0.5) * dt, amp * w)),
    }


def _lattice_inputs(case, seed):
    nx, ny = case["nx"], case["ny"]
    rng = np.random.default_rng(seed)
    dx, dt, cK, cmu = _geometry(nx, ny, float(rng.uniform(0.0, 0.4)))
    g = {"dx": dx, "dt": dt, "cK": cK, "cmu": cmu}
    if case["load"]:
        return dict(g, **_loaded_fields(case, dx, dt, rng))
    gen = torch.Generator(device=DEV).manual_seed(seed)
    U = _rest_fields(nx, ny, dx, case["bc"] == "dirichlet", min(64.0, min(nx, ny) / 8.0), gen)
    return dict(g, U0=U[0], Ux=U[1], Uy=U[2], u0=None, B0=None, load=None, wall=None)


def _batch_inputs(case, seed):
    """Descriptors and initial fields: the short side log-uniform, the aspect ratio uniform in
    [1, 4], random orientation and Poisson ratio, every second lattice Dirichlet."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    shapes = np.random.default_rng(3)         # sizes as in the benchmark's batch; the fields follow the seed
    descs, fields = [], []
    for i in range(case["count"]):
        s = int(round(math.exp(shapes.uniform(math.log(case["smin"]), math.log(case["smax"])))))
        long = int(round(shapes.uniform(1.0, 4.0) * s))
        nx, ny = (long, s) if shapes.integers(0, 2) else (s, long)
        dx, dt, cK, cmu = _geometry(nx, ny, float(rng.uniform(0.0, 0.49)))
        descs.append((nx, ny, i % 2, dx, dt, cK, cmu))
        fields.append(_rest_fields(nx, ny, dx, i % 2 == 1, s / 16.0, gen))
    return descs, fields


def _solver_inputs(case, seed):
    n, side = case["n"], case["side"]
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    U = torch.zeros((n, 10, side, side), **F64)
    for i in range(n):
        for c in range(5):
            U[i, c] = _random_field(side, side, float(rng.uniform(0.0625, 0.25)) * side, 1.0, gen)[0]
    return U, rng.uniform(0.0, 0.49, n)


def _unet_weights(seed):
    """Weights of a network as training leaves them: every layer active, the output layer too."""
    rng = np.random.default_rng(seed)
    c0, c1, c2, c3 = 32, 64, 128, 256
    shapes = [(32, c0), (c0, c0), (c0, c1), (c1, c1), (c1, c2), (c2, c2), (c2, c3), (c3, c3), (c3 + c2, c2), (c2, c2),
              (c2 + c1, c1), (c1, c1), (c1 + c0, c0), (c0, c0), (c0, 32)]
    sd = {}
    for i, (ci, co) in enumerate(shapes):
        ks = 1 if i == 14 else 3
        sd[f"w{i}"] = (rng.standard_normal((co, ks, ks, ci)) * math.sqrt(2.0 / (ci * ks * ks))).astype(np.float32)
        sd[f"b{i}"] = (0.1 * rng.standard_normal(co)).astype(np.float32)
    return sd


def _unet_inputs(case, seed):
    side, B = case["side"], case["B"]
    U, nu = _solver_inputs({"n": B, "side": side}, seed)
    scale = np.full(5, 1e-3)
    return U, torch.tensor((nu - S.NU_MEAN) / S.NU_STD, dtype=torch.float32, device=DEV), scale


def _layer_inputs(case, seed):
    """One layer's saved tensors in a training step: inputs and output after ReLU, the gradient of
    its output, its weights."""
    lv, C1, C2, Co, half = LAYERS[case["layer"]]
    gen = torch.Generator(device=DEV).manual_seed(seed)
    B, h = case["B"], case["side"] >> lv
    f32 = dict(dtype=torch.float32, device=DEV, generator=gen)
    h1 = h // 2 if half else h
    x1 = torch.randn((B, h1, h1, C1), **f32).clamp_(min=0.0)
    x2 = torch.randn((B, h, h, C2), **f32).clamp_(min=0.0) if C2 else None
    y = torch.randn((B, h, h, Co), **f32).clamp_(min=0.0)
    dy = torch.randn((B, h, h, Co), **f32) * 1e-3
    w = torch.randn((Co, 3, 3, C1 + C2), **f32) * math.sqrt(2.0 / (9 * (C1 + C2)))
    return x1, x2, y, dy, w


# ---------------------------------------------------------------------------
# what a program holds before the call, and the call
# ---------------------------------------------------------------------------

def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        d = _lattice_inputs(case, seed)
        dirichlet = case["bc"] == "dirichlet"
        lat = L.Lattice(case["nx"], case["ny"], d["dx"], d["dt"], d["cK"], d["cmu"], dirichlet=dirichlet,
                        storage=case["storage"], track_displacement=case["track"], stream=_stream())
        if d["load"] is not None:
            lat.set_forcing(*d["load"])
            if dirichlet:
                lat.set_dirichlet_separable(*d["wall"])
        out = torch.empty((10, case["ny"], case["nx"]), **F64)
        return {"case": case, "lat": lat, "init": (d["U0"], d["Ux"], d["Uy"], d["B0"], d["u0"]), "out": out}
    if kind == "batch":
        descs, fields = _batch_inputs(case, seed)
        flat = torch.empty(sum(10 * d[0] * d[1] for d in descs), **F64)
        outs, at = [], 0
        for d in descs:
            n = 10 * d[0] * d[1]
            outs.append(flat[at:at + n].view(10, d[1], d[0]))
            at += n
        return {"case": case, "batch": _Batch(descs, case["storage"]), "fields": fields, "outs": outs, "flat": flat}
    if kind == "solver":
        U, nu = _solver_inputs(case, seed)
        side = case["side"]
        descs = []
        for v in nu:
            dx, dt, cK, cmu = _geometry(side, side, float(v))
            descs.append((side, side, 0, dx, dt, cK, cmu))
        return {"case": case, "U": U, "nu": nu, "batch": _Batch(descs, case["storage"])}
    if kind == "unet":
        U, nu_norm, scale = _unet_inputs(case, seed)
        net = S.UNet((32, 64, 128, 256), seed=0)
        net.load_state_dict(_unet_weights(seed))
        net._alloc(case["B"], case["side"], case["side"])
        return {"case": case, "sur": S.Surrogate(net, scale, 32), "U": U, "nu_norm": nu_norm}
    x1, x2, y, dy, w = _layer_inputs(case, seed)
    lv, C1, C2, Co, half = LAYERS[case["layer"]]
    conv = S.Conv(C1, C2, Co, 3, True, np.random.default_rng(0), torch.device(DEV), zero=True)
    conv.w.copy_(w)
    K.to_bf16(conv.w, conv.wb)
    B, h = case["B"], case["side"] >> lv
    ws = max(K.wgrad_workspace_bytes(C1 + C2, Co, B, h, h, 3), K.bias_grad_workspace_bytes(B * h * h, Co))
    return {"case": case, "conv": conv, "x1": x1, "x2": x2, "y": y, "dy": dy,
            "dx1": torch.empty((B, h, h, C1), dtype=torch.float32, device=DEV),
            "dx2": torch.empty((B, h, h, C2), dtype=torch.float32, device=DEV) if C2 else None,
            "ws": torch.empty(ws // 4 + 1, dtype=torch.float32, device=DEV)}


class _Batch:
    """A lattice batch in the launch mode the framework's own users set for its storage format."""

    def __init__(self, descs, storage):
        self.h = L.lbm_batch_create(descs, storage=L.STORAGE[storage], stream=_stream())
        L.lbm_batch_set_mode(self.h, 3 if storage == "f64" else 2)

    def __del__(self):
        L.lbm_batch_destroy(self.h)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "lattice":
        s["lat"].init(*s["init"])
        s["lat"].step(case["steps"])
        return s["lat"].moments(s["out"])
    if kind == "batch":
        b = s["batch"].h
        for i, U in enumerate(s["fields"]):
            L.lbm_batch_init(b, i, U[0], U[1], U[2])
        L.lbm_batch_step(b, case["steps"])
        for i, out in enumerate(s["outs"]):
            L.lbm_batch_moments(b, i, out)
        return s["flat"]
    if kind == "solver":
        return S.relift_and_step(s["U"], s["nu"], case["k"], case["storage"], s["batch"].h)
    if kind == "unet":
        sur, B, side = s["sur"], case["B"], case["side"]
        sur.pack(s["U"], 10 * side * side, s["nu_norm"], B, side, side)
        sur.net.forward(B, side, side, act_bf16=case["act_bf16"])
        return sur.net.A["out"]
    lv, C1, C2, Co, half = LAYERS[case["layer"]]
    B, h, conv = case["B"], case["side"] >> lv, s["conv"]
    conv.backward(s["dy"], s["y"], s["x1"], s["x2"], B, h, h, s["dx1"], s["dx2"], s["ws"], x1_half=half)
    out = [conv.gw, conv.gb, s["dx1"]]
    return out + [s["dx2"]] if C2 else out


# ---------------------------------------------------------------------------
# what the path cannot do without
# ---------------------------------------------------------------------------

def _unet_layers(case):
    side = case["side"]
    for lv, C1, C2, Co, _ in [(0, 32, 0, 32, False)] + list(LAYERS.values()):
        yield (side >> lv) ** 2, 9 * (C1 + C2), Co
    yield side * side, 32, 32


def work(case):
    """Inputs and outputs once; 59 operations per node and step (35 additions and 12 fused
    multiply-adds), 2 per multiply-add of a convolution."""
    kind = case["kind"]
    if kind == "lattice":
        n = case["nx"] * case["ny"]
        return {"bytes": 8.0 * n * (15 + 10 + (4 if case["load"] else 0)), "flops": 59.0 * n * case["steps"]}
    if kind == "batch":
        shapes = np.random.default_rng(3)
        n = 0
        for _ in range(case["count"]):
            s = int(round(math.exp(shapes.uniform(math.log(case["smin"]), math.log(case["smax"])))))
            n += s * int(round(shapes.uniform(1.0, 4.0) * s))
            shapes.integers(0, 2)
        return {"bytes": 8.0 * n * 25, "flops": 59.0 * n * case["steps"]}
    if kind == "solver":
        n = case["n"] * case["side"] ** 2
        return {"bytes": 8.0 * n * 15, "flops": 59.0 * n * case["k"]}
    if kind == "unet":
        B, side = case["B"], case["side"]
        return {"bytes": 8.0 * B * 5 * side * side + 4.0 * B * 32 * side * side + 2 * 1.95e6,
                "flops": sum(2.0 * B * p * c * co for p, c, co in _unet_layers(case))}
    lv, C1, C2, Co, half = LAYERS[case["layer"]]
    P = case["B"] * (case["side"] >> lv) ** 2
    return {"bytes": 4.0 * P * (C1 / (4 if half else 1) + C2 + 2 * Co + C1 + C2) + 6.0 * 9 * Co * (C1 + C2),
            "flops": 2 * 2.0 * P * 9 * (C1 + C2) * Co}


# ---------------------------------------------------------------------------
# the same in 64 bits with plain torch
# ---------------------------------------------------------------------------

def _phi(U, cK, cmu):
    px = (cK * U[2] + cmu * U[3], cmu * U[4], cK * U[0], cmu * U[0], cmu * U[1])
    py = (cmu * U[4], cK * U[2] - cmu * U[3], cK * U[1], -cmu * U[1], cmu * U[0])
    return px, py


def _exact_init(U0, Ux, Uy, B0, dx, dt, cK, cmu):
    """Second-order initial populations [4][5][ny][nx] (Eq. ic_second)."""
    c = dx / dt
    px, py = _phi(U0, cK, cmu)
    gx, gy = _phi(Ux, cK, cmu)[0], _phi(Uy, cK, cmu)[1]
    dU = [gx[k] + gy[k] for k in range(5)]
    qx, qy = _phi(dU, cK, cmu)
    bx = by = None
    if B0 is not None:
        z = torch.zeros_like(B0[0])
        bx, by = _phi([B0[0], B0[1], z, z, z], cK, cmu)
    f = torch.empty((4,) + tuple(U0.shape), **F64)
    for d, (i, j) in enumerate(((1, 0), (0, 1), (-1, 0), (0, -1))):
        for k in range(5):
            eq = 0.25 * (U0[k] + (2.0 / c) * (i * px[k] + j * py[k]))
            t = c * (i * Ux[k] + j * Uy[k]) + (2 * i * i - 1) * gx[k] + (2 * j * j - 1) * gy[k] \
                - (2.0 / c) * (i * qx[k] + j * qy[k])
            if B0 is not None:
                t = t + (2.0 / c) * (i * bx[k] + j * by[k]) + (B0[k] if k < 2 else 0.0)
            f[d, k] = eq - (dt / 8.0) * t
    return f


def _exact_run(U0, Ux, Uy, B0, u0, dx, dt, cK, cmu, steps, dirichlet, load, wall):
    """The scheme of Sec. 3.6 with omega = 2: moments, equilibrium, collision, streaming, walls."""
    c = dx / dt
    ny, nx = U0.shape[-2:]
    f = _exact_init(U0, Ux, Uy, B0, dx, dt, cK, cmu)
    if load is not None:
        X, Y, T = (torch.as_tensor(v, **F64) for v in load)
        b = lambda m: torch.einsum("rx,ry,cr->cyx", X, Y, T[m])
    if dirichlet and wall is not None:
        Xn, Xw, Yn, Yw, Tw = (torch.as_tensor(v, **F64) for v in wall)
        g_side = lambda m, e: torch.einsum("r,ry,cr->cy", Xw[:, e], Yn, Tw[m])
        g_end = lambda m, e: torch.einsum("rx,r,cr->cx", Xn, Yw[:, e], Tw[m])

    def moment(m):
        U = f.sum(0)
        if load is not None:
            U[:2] += (0.5 * dt) * b(m)
        return U

    def source(i, j, g):
        gx, gy = g
        return (0.5 * gx, 0.5 * gy, (cK / c) * (i * gx + j * gy), (cmu / c) * (i * gx - j * gy),
                (cmu / c) * (j * gx + i * gy))

    us = None
    sign = (-1.0, -1.0, 1.0, 1.0, 1.0)
    for m in range(steps):
        U = moment(m)
        if u0 is not None:
            us = u0 - (0.5 * dt) * U[:2] if us is None else us
            us = us + dt * U[:2]
        px, py = _phi(U, cK, cmu)
        for k in range(5):
            h, x, y = 0.5 * U[k], px[k] / c, py[k] / c
            a = [h + x - f[0, k], h + y - f[1, k], h - x - f[2, k], h - y - f[3, k]]
            f[0, k, :, 1:], f[0, k, :, 0] = a[0][:, :-1], a[0][:, -1]
            f[2, k, :, :-1], f[2, k, :, -1] = a[2][:, 1:], a[2][:, 0]
            f[1, k, 1:], f[1, k, 0] = a[1][:-1], a[1][-1]
            f[3, k, :-1], f[3, k, -1] = a[3][1:], a[3][0]
            if dirichlet:
                f[0, k, :, 0], f[2, k, :, -1] = sign[k] * a[2][:, 0], sign[k] * a[0][:, -1]
                f[1, k, 0], f[3, k, -1] = sign[k] * a[3][0], sign[k] * a[1][-1]
                if wall is not None:
                    f[0, k, :, 0] += source(1, 0, g_side(m, 0))[k]
                    f[2, k, :, -1] += source(-1, 0, g_side(m, 1))[k]
                    f[1, k, 0] += source(0, 1, g_end(m, 0))[k]
                    f[3, k, -1] += source(0, -1, g_end(m, 1))[k]
    U = moment(steps)
    out = torch.zeros((10, ny, nx), **F64)
    out[:5] = U
    if u0 is not None:
        out[5:7] = us + (0.5 * dt) * U[:2]
    out[7] = -(cK * U[2] + cmu * U[3])
    out[8] = -(cK * U[2] - cmu * U[3])
    out[9] = -(cmu * U[4])
    return out


def _taps(x, ks):
    for dy in range(ks):
        for dx in range(ks):
            yield dy, dx, torch.roll(x, (ks // 2 - dy, ks // 2 - dx), (1, 2)) if ks > 1 else x


def _exact_conv(x, w, bias, relu):
    y = bias.expand(x.shape[:3] + (w.shape[0],)).clone()
    for dy, dx, xs in _taps(x, w.shape[1]):
        y += xs @ w[:, dy, dx].T
    return y.clamp_(min=0.0) if relu else y


def _half(x):
    return x.repeat_interleave(2, 1).repeat_interleave(2, 2)


def _exact_unet(case, seed):
    U, nu_norm, scale = _unet_inputs(case, seed)
    sd = _unet_weights(seed)
    w = [torch.from_numpy(sd[f"w{i}"]).to(DEV).to(torch.bfloat16).double() for i in range(15)]
    b = [torch.from_numpy(sd[f"b{i}"]).to(DEV).double() for i in range(15)]
    outs = []
    for n in range(case["B"]):
        side = case["side"]
        x = torch.zeros((1, side, side, 32), **F64)
        x[0, ..., :5] = (U[n, :5] / torch.as_tensor(scale, **F64)[:, None, None]).permute(1, 2, 0)
        x[0, ..., 5] = nu_norm[n].double()
        e = []
        for lv in range(4):
            if lv:
                x = F.avg_pool2d(x.permute(0, 3, 1, 2), 2).permute(0, 2, 3, 1)
            x = _exact_conv(x, w[2 * lv], b[2 * lv], True)
            x = _exact_conv(x, w[2 * lv + 1], b[2 * lv + 1], True)
            e.append(x)
        for i, lv in enumerate((2, 1, 0)):
            x = _exact_conv(torch.cat([_half(x), e[lv]], 3), w[8 + 2 * i], b[8 + 2 * i], True)
            x = _exact_conv(x, w[9 + 2 * i], b[9 + 2 * i], True)
        outs.append(_exact_conv(x, w[14], b[14], False))
    return torch.cat(outs)


def _exact_layer(case, seed):
    x1, x2, y, dy, w = _layer_inputs(case, seed)
    lv, C1, C2, Co, half = LAYERS[case["layer"]]
    B = case["B"]
    w = w.to(torch.bfloat16).double()
    gw, gb, dx = torch.zeros_like(w), torch.zeros(Co, **F64), []
    for n in range(B):
        x = x1[n:n + 1].double()
        x = _half(x) if half else x
        x = torch.cat([x, x2[n:n + 1].double()], 3) if C2 else x
        d = torch.where(y[n:n + 1] > 0, dy[n:n + 1], torch.zeros_like(dy[n:n + 1])).double()
        gb += d.sum((0, 1, 2))
        g = torch.zeros_like(x)
        for ky, kx, xs in _taps(x, 3):
            gw[:, ky, kx] += torch.einsum("byxo,byxi->oi", d, xs)
            g += torch.roll(d @ w[:, ky, kx], (ky - 1, kx - 1), (1, 2))
        dx.append(g)
    dx = torch.cat(dx)
    out = [gw, gb, dx[..., :C1].contiguous()]
    return out + [dx[..., C1:].contiguous()] if C2 else out


def exact(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        d = _lattice_inputs(case, seed)
        return _exact_run(d["U0"], d["Ux"], d["Uy"], d["B0"], d["u0"] if case["track"] else None, d["dx"], d["dt"],
                          d["cK"], d["cmu"], case["steps"], case["bc"] == "dirichlet", d["load"], d["wall"])
    if kind == "batch":
        descs, fields = _batch_inputs(case, seed)
        if len(descs) * case["steps"] > 12000:      # a step of each lattice is some fifty torch calls
            return None
        return torch.cat([_exact_run(U[0], U[1], U[2], None, None, d[3], d[4], d[5], d[6], case["steps"], d[2] == 1,
                                     None, None).reshape(-1) for d, U in zip(descs, fields)])
    if kind == "solver":
        U, nu = _solver_inputs(case, seed)
        outs = []
        for i, v in enumerate(nu):
            dx, dt, cK, cmu = _geometry(case["side"], case["side"], float(v))
            u = U[i, :5]
            ux = (torch.roll(u, -1, 2) - torch.roll(u, 1, 2)) / (2.0 * dx)
            uy = (torch.roll(u, -1, 1) - torch.roll(u, 1, 1)) / (2.0 * dx)
            outs.append(_exact_run(u, ux, uy, None, None, dx, dt, cK, cmu, case["k"], False, None, None))
        return torch.stack(outs)
    return _exact_unet(case, seed) if kind == "unet" else _exact_layer(case, seed)
