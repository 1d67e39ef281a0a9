"""Timed cases of the spectral FNO block library, as a user's program calls it.

A case names one call pattern (``kind``) and its sizes:

* ``block_train``    one FNO block of a training step: ``FNOBlock4d`` forward and
                     its backward through autograd (z, dx and every parameter
                     gradient).
* ``block_infer``    the same block evaluated under ``torch.no_grad``.
* ``spectral_train`` the bare spectral convolution (``SpectralConv4dFn``)
                     forward and backward.
* ``stack_train``    encoder, blocks, decoder, MSE loss and the whole backward by
                     ``StackRunner.step``.
* ``stack_infer``    the ``FNO4d`` model evaluated under ``torch.no_grad``.

Inputs stand for the paper's data: smooth periodic random fields (white noise
filtered by a squared-exponential spectrum, one correlation length per axis) for
the fields, N(0, 1) for upstream gradients, and the library's own initial
distributions for the parameters.
"""
import math

import torch

from paper_2211_12709_gb300 import ops, stack

DEV = "cuda"


def _case(name, kind, precision, B, width, grid, modes, c_in=0, c_out=0, blocks=1):
    c = {"kind": kind, "precision": precision, "B": B, "width": width}
    c.update(zip(("Nx", "Ny", "Nz", "Nt"), grid))
    c.update(zip(("mx", "my", "mz", "mt"), modes))
    if kind.startswith("stack"):
        c.update(c_in=c_in, c_out=c_out, blocks=blocks)
    if name:
        c["name"] = name
    return c


def listed():
    """The sizes are those of the benchmark's workloads and of the tests."""
    co2, ns = (128, 128, 128, 32), (64, 64, 64, 16)
    return [
        # The smallest call: one layer on a toy grid, as in first experiments and
        # unit tests, in the default precision. Launches and host work count.
        _case("layer_16c_t8_fp32", "block_train", "fp32", 1, 8, (16, 16, 16, 8), (4, 4, 4, 4)),
        # A small surrogate evaluated in somebody's loop (optimisation, control):
        # the latency of a whole 4-block model.
        _case("stack_infer_32c_t16", "stack_infer", "bf16x3", 1, 20, (32, 32, 32, 16), (8, 8, 8, 6), 3, 1, 4),
        # The benchmark's small block, in the three precisions that are trained in.
        _case("ns_block_64c_t16", "block_train", "bf16x3", 2, 20, ns, (8, 8, 8, 6)),
        _case("ns_block_64c_t16_fp32", "block_train", "fp32", 2, 20, ns, (8, 8, 8, 6)),
        _case("ns_block_64c_t16_bf16", "block_train", "bf16", 2, 20, ns, (8, 8, 8, 6)),
        # The benchmark's headline: a training step's block on 2.1 M cells.
        _case("co2_block_128c_t32", "block_train", "bf16x3", 1, 20, co2, (12, 12, 8, 8)),
        # A block of the wider Navier-Stokes model, two samples of its batch.
        _case("ns_block_w32_64c_t32", "block_train", "bf16x3", 2, 32, (64, 64, 64, 32), (12, 12, 12, 8)),
        # The paper's own grids: a training block on the CO2 data's, an
        # evaluation on the Navier-Stokes data's.
        _case("co2_block_262x118x64_t86", "block_train", "bf16x3", 1, 20, (262, 118, 64, 86), (26, 12, 6, 8)),
        _case("ns_infer_130c_t84", "block_infer", "bf16x3", 1, 20, (130, 130, 130, 84), (13, 13, 13, 8)),
        # The spectral layer alone, inside a model of the user's own, on a grid
        # with odd sizes everywhere.
        _case("spectral_odd_45x37x27_t21", "spectral_train", "fp32", 2, 12, (45, 37, 27, 21), (9, 7, 5, 5)),
        # A whole training pass of the CO2 model at its small size.
        _case("co2_stack_64c_t16", "stack_train", "bf16x3", 1, 20, ns, (8, 8, 8, 6), 3, 1, 4),
        # The trained CO2 model in use: one prediction on the benchmark's grid.
        _case("co2_stack_infer_128c_t32", "stack_infer", "bf16x3", 1, 20, co2, (12, 12, 8, 8), 3, 1, 4),
    ]


def draw(rng):
    """Another case of the same ranges: toy grids to the paper's, powers of two or ragged."""
    kind = rng.choice(["block_train"] * 5 + ["block_infer"] * 2 + ["spectral_train", "stack_train", "stack_infer"])
    precision = rng.choice(["bf16x3"] * 11 + ["fp32"] * 5 + ["bf16"] * 2 + ["tf32"])
    B = rng.choice([1, 1, 1, 2, 2, 4])
    width = rng.choice([8, 12, 16, 20, 20, 20, 24, 32])
    most = 30.5 if kind.startswith("block") else 28.5
    points = 2 ** rng.uniform(15, most) / (B * width)  # of one channel, x to t
    if rng.random() < 0.5:  # powers of two, as synthetic data come
        nt = rng.choice([8, 16, 16, 32, 32])
        side = max(3, min(7, round(math.log2(points / nt) / 3)))
        grid = [2 ** min(7, max(3, side + rng.choice([0, 0, -1]))) for _ in range(3)] + [nt]
    else:  # as measured data come
        nt = rng.randint(8, 96)
        if precision != "fp32":
            nt += nt % 2
        side = max(8.0, (points / nt) ** (1 / 3))
        grid = [max(8, min(262, round(side * 2 ** rng.uniform(-0.6, 0.6)))) for _ in range(3)] + [nt]
        grid[2] = min(grid[2], 130)
        if precision != "fp32" and grid[2] * nt % 4:
            grid[2] += 1  # the tensor-core precisions take Nz * Nt in multiples of 4
    modes = [max(1, min(cap, n // 2, round(n * rng.uniform(0.06, 0.25)))) for n, cap in zip(grid, (26, 26, 12))]
    modes.append(rng.randint(3, min(8, nt // 2 + 1)))
    while width * width * 8 * modes[0] * modes[1] * modes[2] * modes[3] > 110_000_000:  # weights of 0.9 GB, as the models'
        k = max(range(3), key=lambda a: modes[a])
        modes[k] -= 1
    c_in, c_out = rng.choice([(3, 1), (4, 4)])
    return _case(None, kind, precision, B, width, grid, modes, c_in, c_out, rng.randint(2, 4))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _grid(c):
    return (c["Nx"], c["Ny"], c["Nz"], c["Nt"])


def _modes(c):
    return (c["mx"], c["my"], c["mz"], c["mt"])


def _wshape(c):
    return (c["width"], c["width"], 2 * c["mx"], 2 * c["my"], 2 * c["mz"], c["mt"], 2)


def _field(g, B, C, grid):
    """Periodic random fields [B, C, *grid], unit variance, correlated over about a tenth of each axis."""
    x = torch.empty((B, C) + grid, device=DEV)
    filt = []
    for a, n in enumerate(grid):
        f = torch.fft.rfftfreq(n, device=DEV) if a == 3 else torch.fft.fftfreq(n, device=DEV)
        filt.append(torch.exp(-((math.pi * 0.1 * n * f) ** 2)).reshape([-1 if q == a else 1 for q in range(4)]))
    for b in range(B):
        for c in range(C):
            s = torch.fft.rfftn(torch.randn(grid, generator=g, device=DEV))
            for f in filt:
                s *= f
            v = torch.fft.irfftn(s, s=grid)
            v -= v.mean()
            x[b, c] = v / v.std()
    return x


def _normal(g, shape):
    return torch.randn(shape, generator=g, device=DEV)


def _uniform(g, shape, s):
    return torch.rand(shape, generator=g, device=DEV).mul_(2 * s).sub_(s)


def _block_params(g, c):
    W = c["width"]
    return (_uniform(g, _wshape(c), 1.0 / (W * W)), _uniform(g, (W, W), W ** -0.5), _uniform(g, (W,), W ** -0.5))


def _stack_params(g, c):
    W, ci, co = c["width"], c["c_in"], c["c_out"]
    return {"enc_w": _uniform(g, (ci, W), ci ** -0.5), "enc_b": _uniform(g, (W,), ci ** -0.5),
            "blocks": [_block_params(g, c) for _ in range(c["blocks"])],
            "dec_w": _uniform(g, (W, co), W ** -0.5), "dec_b": _uniform(g, (co,), W ** -0.5)}


def _inputs(c, seed):
    """The tensors of a case from its seed alone."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    B, W, grid, kind = c["B"], c["width"], _grid(c), c["kind"]
    if kind.startswith("stack"):
        t = {"x": _field(g, B, c["c_in"], grid), "params": _stack_params(g, c)}
        if kind == "stack_train":
            t["target"] = torch.sigmoid(_field(g, B, c["c_out"], grid))
        return t
    t = {"x": _field(g, B, W, grid)}
    t["w"], t["w_lin"], t["bias"] = _block_params(g, c)
    if kind.endswith("train"):
        t["dz"] = _normal(g, (B, W) + grid)
    return t


def prepare(case, seed):
    t = _inputs(case, seed)
    kind, modes = case["kind"], _modes(case)
    state = {"kind": kind, "modes": modes, "precision": case["precision"], "x": t["x"]}
    if kind.startswith("block"):
        block = ops.FNOBlock4d(case["width"], (1, 1, 1, 1), case["precision"], device=DEV, seed=0)
        block.modes = modes
        block.weight, block.w_lin, block.bias = (torch.nn.Parameter(t[k]) for k in ("w", "w_lin", "bias"))
        state["block"] = block
    if kind in ("block_train", "spectral_train"):
        state["x"].requires_grad_(True)
        state["dz"] = t["dz"]
    if kind == "spectral_train":
        state["w"] = t["w"].requires_grad_(True)
    if kind == "stack_infer":
        p = t["params"]
        model = stack.FNO4d(case["c_in"], case["width"], case["c_out"], (1, 1, 1, 1), case["blocks"],
                            case["precision"], device=DEV)
        model.enc_w, model.enc_b, model.dec_w, model.dec_b = (
            torch.nn.Parameter(p[k]) for k in ("enc_w", "enc_b", "dec_w", "dec_b"))
        for block, q in zip(model.blocks, p["blocks"]):
            block.modes = modes
            block.weight, block.w_lin, block.bias = (torch.nn.Parameter(v) for v in q)
        state["model"] = model
    if kind == "stack_train":
        state["target"] = t["target"]
        state["runner"] = stack.StackRunner(case["B"], case["c_in"], _grid(case), t["params"], modes,
                                            precision=case["precision"], device=DEV)
    return state


def run(state):
    kind, x = state["kind"], state["x"]
    if kind == "block_train":
        block = state["block"]
        z = block(x)
        dx, dw, dwl, db = torch.autograd.grad(z, (x, block.weight, block.w_lin, block.bias), state["dz"])
        return {"z": z.detach(), "dx": dx, "dw": dw, "dw_lin": dwl, "db": db}
    if kind == "block_infer":
        with torch.no_grad():
            return {"z": state["block"](x)}
    if kind == "spectral_train":
        y = ops.SpectralConv4dFn.apply(x, state["w"], state["modes"], state["precision"])
        dx, dw = torch.autograd.grad(y, (x, state["w"]), state["dz"])
        return {"y": y.detach(), "dx": dx, "dw": dw}
    if kind == "stack_infer":
        with torch.no_grad():
            return {"y": state["model"](x)}
    r = state["runner"]
    loss = r.step(x, state["target"])
    return {"y": r.y, "loss": loss, "grads": r.grads}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _dft_flops(c):
    """Real operations of one truncated transform of one channel, axis by axis (t, z, y, x)."""
    Nx, Ny, Nz, Nt = _grid(c)
    Jx, Jy, Jz, Jt = 2 * c["mx"], 2 * c["my"], 2 * c["mz"], c["mt"]
    return (4.0 * Nx * Ny * Nz * Nt * Jt + 8.0 * Nx * Ny * Nz * Jz * Jt + 8.0 * Nx * Ny * Jy * Jz * Jt
            + 8.0 * Nx * Jx * Jy * Jz * Jt)


def work(case):
    """Each input read once and each output written once; the transforms, the mixing and the 1x1 layers once."""
    kind, B, W = case["kind"], case["B"], case["width"]
    N = float(math.prod(_grid(case)))
    field, weights = 4.0 * B * W * N, 4.0 * math.prod(_wshape(case))
    dft = B * W * _dft_flops(case)
    mix = 4.0 * B * math.prod(_wshape(case))
    lin = 2.0 * B * W * W * N
    fwd_flops = 2 * dft + mix + (0 if kind == "spectral_train" else lin)
    bwd_flops = 2 * dft + 2 * mix + (0 if kind == "spectral_train" else 2 * lin)
    if not kind.startswith("stack"):
        if kind == "block_infer":
            return {"bytes": 2 * field + weights, "flops": fwd_flops}
        return {"bytes": 4 * field + 2 * weights, "flops": fwd_flops + bwd_flops}
    ci, co, L = case["c_in"], case["c_out"], case["blocks"]
    ends = 2.0 * B * N * W * (ci + co)
    if kind == "stack_infer":
        return {"bytes": 4.0 * B * N * (ci + co) + L * weights, "flops": L * fwd_flops + ends}
    return {"bytes": 4.0 * B * N * (ci + 2 * co) + 2 * L * weights, "flops": L * (fwd_flops + bwd_flops) + 3 * ends}


# ---------------------------------------------------------------------------
# The same results in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _bases(case):
    """Forward DFT bases of the axes x, y, z, t: e^{-2 pi i k n / N}, kept k by row, complex128."""
    out = []
    for a, (n, m) in enumerate(zip(_grid(case), _modes(case))):
        k = torch.arange(m, device=DEV) if a == 3 else torch.cat([torch.arange(m), torch.arange(-m, 0)]).to(DEV)
        r = (k[:, None] * torch.arange(n, device=DEV)[None, :]) % n
        ang = r.double() * (-2 * math.pi / n)
        out.append(torch.complex(torch.cos(ang), torch.sin(ang)))
    return out


def _inverse_scale(case):
    """c(kt) / N: the half spectrum's weights and the inverse transform's scale."""
    Nt = case["Nt"]
    c = torch.full((case["mt"],), 2.0, dtype=torch.float64, device=DEV)
    c[0] = 1.0
    if Nt % 2 == 0 and case["mt"] > Nt // 2:
        c[Nt // 2] = 1.0
    return c / math.prod(_grid(case))


def _spectrum(case, F, v):
    """Kept spectra [B, C, Jx, Jy, Jz, Jt] of real fields, one channel at a time."""
    Fx, Fy, Fz, Ft = F
    out = torch.empty(v.shape[:2] + (Fx.shape[0], Fy.shape[0], Fz.shape[0], Ft.shape[0]),
                      dtype=torch.complex128, device=DEV)
    for b in range(v.shape[0]):
        for c in range(v.shape[1]):
            u = v[b, c].double()
            s = torch.complex(u @ Ft.real.T.contiguous(), u @ Ft.imag.T.contiguous())
            s = torch.einsum("kz,xyzt->xykt", Fz, s)
            s = torch.einsum("ky,xyzt->xkzt", Fy, s)
            out[b, c] = torch.einsum("kx,xyzt->kyzt", Fx, s)
    return out


def _synthesis(case, F, s):
    """Real fields sum_j Re(s_j e^{+i theta_j}) of kept spectra, one channel at a time."""
    Ix, Iy, Iz, It = (f.conj() for f in F)
    out = torch.empty(s.shape[:2] + _grid(case), dtype=torch.float64, device=DEV)
    for b in range(s.shape[0]):
        for c in range(s.shape[1]):
            u = torch.einsum("kx,kyzt->xyzt", Ix, s[b, c])
            u = torch.einsum("ky,xkzt->xyzt", Iy, u)
            u = torch.einsum("kz,xykt->xyzt", Iz, u)
            out[b, c] = u.real @ It.real - u.imag @ It.imag
    return out


def _add_linear(out, x, w, bias=None):
    """out[b, o] += sum_i w[i, o] x[b, i] (+ bias[o]), in place, in runs of points."""
    P = math.prod(x.shape[2:])
    for b in range(x.shape[0]):
        xb, ob = x[b].reshape(x.shape[1], P), out[b].reshape(out.shape[1], P)
        for p in range(0, P, 1 << 24):
            ob[:, p:p + (1 << 24)] += w.double().T @ xb[:, p:p + (1 << 24)].double()
    if bias is not None:
        out += bias.double().reshape(1, -1, 1, 1, 1, 1)
    return out


def _contract(x, d):
    """sum over batch and points of x[b, i, p] d[b, o, p]: the gradient of a 1x1 weight."""
    P = math.prod(x.shape[2:])
    r = torch.zeros((x.shape[1], d.shape[1]), dtype=torch.float64, device=DEV)
    for b in range(x.shape[0]):
        xb, gb = x[b].reshape(x.shape[1], P), d[b].reshape(d.shape[1], P)
        for p in range(0, P, 1 << 24):
            r += xb[:, p:p + (1 << 24)].double() @ gb[:, p:p + (1 << 24)].double().T
    return r


def _gelu_(a):
    for v in a.reshape(-1).split(1 << 27):
        v.copy_(torch.nn.functional.gelu(v))
    return a


def _gelu_grad_(a, dz):
    """a <- dz GELU'(a), in place."""
    for v, d in zip(a.reshape(-1).split(1 << 27), dz.reshape(-1).split(1 << 27)):
        v.copy_(d.double() * (0.5 * torch.erfc(v * -(0.5 ** 0.5)) + v * torch.exp(-0.5 * v * v) / math.sqrt(2 * math.pi)))
    return a


def _complex_weight(w):
    return torch.view_as_complex(w.double())


def _pre_act(case, F, x, w, w_lin=None, bias=None):
    """(spectrum of x, S(x) + 1x1 + bias)."""
    xh = _spectrum(case, F, x)
    yh = torch.einsum("bi...,io...->bo...", xh, _complex_weight(w)) * _inverse_scale(case)
    a = _synthesis(case, F, yh)
    return xh, a if w_lin is None else _add_linear(a, x, w_lin, bias)


def _adjoint(case, F, xh, w, d, w_lin=None):
    """(dx, dw) for the gradient d of S(x) + 1x1."""
    g = _spectrum(case, F, d) * _inverse_scale(case)
    dw = torch.view_as_real(torch.einsum("bi...,bo...->io...", xh.conj(), g))
    dx = _synthesis(case, F, torch.einsum("bo...,io...->bi...", g, _complex_weight(w).conj()))
    return dx if w_lin is None else _add_linear(dx, d, w_lin.T), dw


def _block_grads(case, F, x, p, dz):
    """(dx, dw, dw_lin, db) of a block with parameters p for upstream dz."""
    w, wl, bias = p
    xh, a = _pre_act(case, F, x, w, wl, bias)
    d = _gelu_grad_(a, dz)
    dx, dw = _adjoint(case, F, xh, w, d, wl)
    return dx, dw, _contract(x, d), d.sum(dim=(0, 2, 3, 4, 5))


def _pointwise(x, w, bias):
    return _add_linear(torch.zeros((x.shape[0], w.shape[1]) + x.shape[2:], dtype=torch.float64, device=DEV), x, w, bias)


def exact(case, seed):
    t = _inputs(case, seed)
    F = _bases(case)
    kind, x = case["kind"], t["x"]
    if kind == "spectral_train":
        xh, y = _pre_act(case, F, x, t["w"])
        dx, dw = _adjoint(case, F, xh, t["w"], t["dz"])
        return {"y": y, "dx": dx, "dw": dw}
    if kind.startswith("block"):
        p = (t["w"], t["w_lin"], t["bias"])
        z = _gelu_(_pre_act(case, F, x, *p)[1])
        if kind == "block_infer":
            return {"z": z}
        dx, dw, dwl, db = _block_grads(case, F, x, p, t["dz"])
        return {"z": z, "dx": dx, "dw": dw, "dw_lin": dwl, "db": db}
    p = t["params"]
    h = [_gelu_(_pointwise(x, p["enc_w"], p["enc_b"]))]
    for q in p["blocks"]:
        z = _gelu_(_pre_act(case, F, h[-1], *q)[1])
        h = h + [z] if kind == "stack_train" else [z]
    a = _pointwise(h[-1], p["dec_w"], p["dec_b"])
    y = _gelu_(a.clone())
    if kind == "stack_infer":
        return {"y": y}
    diff = y - t["target"].double()
    grads = {"blocks": []}
    d = _gelu_grad_(a, diff * (2.0 / diff.numel()))
    grads["dec_w"], grads["dec_b"] = _contract(h[-1], d), d.sum(dim=(0, 2, 3, 4, 5))
    up = _add_linear(torch.zeros_like(h[-1]), d, p["dec_w"].T)
    for hk, q in zip(reversed(h[:-1]), reversed(p["blocks"])):
        up, dw, dwl, db = _block_grads(case, F, hk, q, up)
        grads["blocks"].insert(0, (dw, dwl, db))
    d = _gelu_grad_(_pointwise(x, p["enc_w"], p["enc_b"]), up)
    grads["enc_w"], grads["enc_b"] = _contract(x, d), d.sum(dim=(0, 2, 3, 4, 5))
    return {"y": y, "loss": (diff * diff).mean().reshape(1), "grads": grads}
