"""Measured cases: what users of this framework have it do.

A case is one call (or one training step, or one replay of a batch of calls)
through the public entry points of ``paper_1604_04374_gb300``: the plan is made
once, as a program that applies one operator many times keeps it, and the call
gets new right-hand sides.  The operators are the space-varying blurs of the
framework's benchmark: hat windows on a node grid and Gaussian impulse
responses whose width (and in 2D orientation) varies over the grid.

Fields of a case
  kind    "apply"  one operator: forward ("fwd"), adjoint ("adj") or one of each ("both"),
                   as the two products of an iterative solver
          "train"  one step of the differentiable operator: forward and the gradients of
                   u, w and hhat (the operator changes from step to step)
          "mix"    an uneven set of operators and directions, replayed as one graph
  shape   "N" or "NyxNx" (powers of two)
  m       terms;  grid  "gyxgx" node grid of the 2D windows (gy gx = m)
  batch   right-hand sides
  form    "dense" (w given as arrays) or "sep" (w_k = wy_k (x) wx_k)
  flags   "", "lowp", "product" or "sectioned"
  tuned   the program called plan.autotune(batch) once
"""
from __future__ import annotations

import math
import random

import torch

from paper_1604_04374_gb300 import Batch, Plan, pce
from paper_1604_04374_gb300.autograd import convolution_product

FLAGS = {"": 0, "lowp": pce.PCE_FLAG_LOWP_STORAGE, "product": pce.PCE_FLAG_PRODUCT_CONVOLUTION,
         "sectioned": pce.PCE_FLAG_SECTIONED}
MIX_SHAPES = ((4096,), (16384,), (65536,), (256, 256), (512, 512), (1024, 1024))
MIX_M = (4, 8, 16, 32)


def _case(kind, shape, m=1, batch=1, *, name=None, dir="fwd", grid="", form="dense", flags="", tuned=False):
    c = {"kind": kind, "shape": shape, "m": m, "batch": batch, "dir": dir, "grid": grid, "form": form,
         "flags": flags, "tuned": tuned}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a short signal, one right-hand side: the smallest call, launch latency and one chain of work
        _case("apply", "1024", 8, 1, name="1d_1024_m8_b1_fwd"),
        # a long signal of one block in many terms, a ragged handful of right-hand sides, backwards
        _case("apply", "8192", 32, 3, name="1d_8192_m32_b3_adj", dir="adj"),
        # a record too long for one block (four-step transforms), one at a time
        _case("apply", "65536", 16, 1, name="1d_65536_m16_b1_fwd"),
        # many short signals at once (a sensor array), an odd number of terms
        _case("apply", "2048", 11, 300, name="1d_2048_m11_b300_adj", dir="adj"),
        # one small image with windows given as arrays
        _case("apply", "256x256", 16, 1, name="2d_256_m16_b1_fwd", grid="4x4"),
        # a stack of wide strips, windows on the output side, a node grid that is no power of two
        _case("apply", "128x512", 6, 24, name="2d_128x512_m6_b24_product", grid="2x3", flags="product"),
        # one image, tensor-product windows, the plan as it comes: one product of each for a solver step
        _case("apply", "1024x1024", 16, 1, name="2d_1024_m16_b1_sep_both", grid="4x4", form="sep", dir="both"),
        # the framework's headline workload: eight images, both products, the plan tuned once
        _case("apply", "1024x1024", 16, 8, name="2d_1024_m16_b8_sep_both", grid="4x4", form="sep", dir="both",
              tuned=True),
        # learning the operator: sixteen 512 x 512 images, gradients of u, w and hhat
        _case("train", "512x512", 16, 16, name="2d_512_m16_b16_train", grid="4x4"),
        # large images, windows and spectra in reduced storage
        _case("apply", "2048x2048", 64, 4, name="2d_2048_m64_b4_lowp_fwd", grid="8x8", flags="lowp"),
        # the same images in full precision with sectioned transforms, backwards
        _case("apply", "2048x2048", 64, 4, name="2d_2048_m64_b4_sectioned_adj", grid="8x8", flags="sectioned",
              dir="adj"),
        # a service's queue: uneven operators, sizes and directions, one graph replay
        _case("mix", "", 0, 256, name="mix_256"),
    ]


def _pow2(rng, lo, hi):
    return 1 << rng.randint(lo, hi)


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    limit = max((work(c) for c in listed()), key=lambda x: x["flops"])
    while True:
        pick = rng.random()
        if pick < 0.3:
            n = _pow2(rng, 8, 18)
            c = _case("apply", str(n), _logint(rng, 1, 48), _logint(rng, 1, 512), dir=rng.choice(("fwd", "adj", "both")),
                      flags=rng.choice(("", "", "product", "lowp" if n <= 8192 else "")))
        elif pick < 0.75:
            ny, nx = _pow2(rng, 6, 11), _pow2(rng, 6, 11)
            gy, gx = rng.randint(1, 8), rng.randint(1, 8)
            form = rng.choice(("dense", "sep"))
            flags = rng.choice(("", "", "", "product", "lowp", "sectioned"))
            if flags == "sectioned":
                if ny < 1024:
                    flags = ""
                else:   # a section holds 1024 rows: box and impulse response together
                    gy = max(gy, ny // 256)
            c = _case("apply", f"{ny}x{nx}", gy * gx, _logint(rng, 1, 24), grid=f"{gy}x{gx}", form=form, flags=flags,
                      dir=rng.choice(("fwd", "adj", "both")), tuned=flags != "sectioned" and rng.random() < 0.2)
        elif pick < 0.92:
            if rng.random() < 0.3:
                c = _case("train", str(_pow2(rng, 8, 13)), _logint(rng, 1, 32), _logint(rng, 1, 64))
            else:
                gy, gx = rng.randint(1, 5), rng.randint(1, 5)
                c = _case("train", f"{_pow2(rng, 6, 10)}x{_pow2(rng, 6, 10)}", gy * gx, _logint(rng, 1, 16),
                          grid=f"{gy}x{gx}")
        else:
            c = _case("mix", "", 0, _logint(rng, 8, 200))
        # no more than the largest listed case
        x = work(c)
        if x["flops"] <= limit["flops"] and x["bytes"] <= limit["bytes"]:
            return c


# ------------------------------------------------------------------ operators

def _shape(case):
    return tuple(int(s) for s in case["shape"].split("x"))


def _grid(case):
    return tuple(int(s) for s in case["grid"].split("x"))


def _hats(n, m, dev):
    """[m][n] periodic hats max(0, 1 - m |t|) at the nodes k / m, in 64 bits."""
    x = torch.arange(n, dtype=torch.float64, device=dev) / n
    t = x[None, :] - torch.arange(m, dtype=torch.float64, device=dev)[:, None] / m
    t = t - torch.round(t)
    return torch.clamp(1.0 - m * t.abs(), min=0.0)


def _psf_1d(n, m, dev, jit):
    """[m][n] periodised Gaussians of width 0.01 + 0.005 sin(2 pi k / m), times 1 / n."""
    x = torch.arange(n, dtype=torch.float64, device=dev) / n
    d = x - torch.floor(x + 0.5)
    sig = (0.01 + 0.005 * torch.sin(2 * math.pi * torch.arange(m, dtype=torch.float64, device=dev) / m)) * jit
    g = sum(torch.exp(-((d[None, :] + j) ** 2) / (2 * sig[:, None] ** 2)) for j in (-1.0, 0.0, 1.0))
    return (g / (math.sqrt(2 * math.pi) * sig[:, None]) / n).float()


def _psf_2d(ny, nx, gy, gx, dev, jit):
    """[gy gx][ny][nx] rotated anisotropic Gaussians of unit sum, origin at [0, 0]."""
    out = torch.empty((gy * gx, ny, nx), dtype=torch.float32, device=dev)
    dx = torch.arange(nx, dtype=torch.float64, device=dev)
    dx = dx - nx * (dx >= nx // 2)
    dy = torch.arange(ny, dtype=torch.float64, device=dev)
    dy = dy - ny * (dy >= ny // 2)
    for a in range(gy):
        for c in range(gx):
            y1, y2 = c / gx, a / gy
            sx, sy, th = (1.5 + y1) * jit, (1.5 + y2) * jit, math.pi * y1 * y2
            co, si = math.cos(th), math.sin(th)
            a11 = co * co / sx ** 2 + si * si / sy ** 2
            a22 = si * si / sx ** 2 + co * co / sy ** 2
            a12 = co * si * (1 / sx ** 2 - 1 / sy ** 2)
            q = a11 * dx[None, :] ** 2 + 2 * a12 * dx[None, :] * dy[:, None] + a22 * dy[:, None] ** 2
            g = torch.exp(-0.5 * q)
            out[a * gx + c] = (g / g.sum()).float()
    return out


def _operator(shape, m, grid, dev, jit):
    """(wy, wx, h) in 2D, (w, None, h) in 1D; float32."""
    if len(shape) == 1:
        return _hats(shape[0], m, dev).float(), None, _psf_1d(shape[0], m, dev, jit)
    gy, gx = grid
    wy = _hats(shape[0], gy, dev).float().repeat_interleave(gx, 0).contiguous()
    wx = _hats(shape[1], gx, dev).float().repeat(gy, 1).contiguous()
    return wy, wx, _psf_2d(shape[0], shape[1], gy, gx, dev, jit)


def _dense(wy, wx):
    return wy if wx is None else (wy[:, :, None] * wx[:, None, :]).contiguous()


def _inputs(case, seed):
    """The arrays of a case on the GPU, from the seed alone."""
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(1604_04374 + seed)
    jit = 1.0 + 0.02 * (2 * torch.rand((), generator=gen, device=dev).item() - 1)
    if case["kind"] == "mix":
        rng = random.Random(1604_04374 + 7 * case["batch"])   # the queue's make-up; its contents follow the seed
        picks = [(rng.randrange(len(MIX_SHAPES)), rng.randrange(len(MIX_M)), rng.randrange(2) == 1)
                 for _ in range(case["batch"])]
        ops = {}
        for s, k, _ in picks:
            if (s, k) not in ops:
                m = MIX_M[k]
                gy = 1 << math.ceil(math.log2(m) / 2)
                ops[(s, k)] = _operator(MIX_SHAPES[s], m, (gy, m // gy), dev, jit)
        ins = []
        for s, _, _ in picks:
            size = (1,) + MIX_SHAPES[s]
            ins.append(torch.randn(size, generator=gen, device=dev) if len(size) == 2
                       else torch.rand(size, generator=gen, device=dev))
        return picks, ops, ins
    shape = _shape(case)
    op = _operator(shape, case["m"], _grid(case) if len(shape) == 2 else None, dev, jit)
    size = (case["batch"],) + shape
    if len(shape) == 1:
        u = torch.randn(size, generator=gen, device=dev)
        v = torch.randn(size, generator=gen, device=dev)
    else:
        u = torch.rand(size, generator=gen, device=dev)
        v = torch.rand(size, generator=gen, device=dev)
    return op, u, v


def _mix_outputs(picks, ins, dtype=torch.float32):
    """One result buffer a shape, [tasks of that shape, *shape], and every task's slice of it."""
    outs, of_task, used = {}, [], {}
    for s in sorted({s for s, _, _ in picks}):
        outs[s] = torch.empty((sum(p[0] == s for p in picks),) + MIX_SHAPES[s], dtype=dtype, device=ins[0].device)
    for s, _, _ in picks:
        i = used.get(s, 0)
        of_task.append(outs[s][i:i + 1])
        used[s] = i + 1
    return list(outs.values()), of_task


def prepare(case, seed):
    if case["kind"] == "mix":
        picks, ops, ins = _inputs(case, seed)
        plans = {k: (Plan(wy, h=h) if wx is None else Plan(wy=wy, wx=wx, h=h)) for k, (wy, wx, h) in ops.items()}
        outs, of_task = _mix_outputs(picks, ins)
        batch = Batch([(plans[(s, k)], x, y, adj) for (s, k, adj), x, y in zip(picks, ins, of_task)])
        return {"case": case, "batch": batch, "outs": outs, "plans": plans}
    (wy, wx, h), u, v = _inputs(case, seed)
    if case["kind"] == "train":
        w = _dense(wy, wx)
        hhat = torch.fft.rfftn(h, dim=tuple(range(1, h.dim())))
        return {"case": case, "u": u.requires_grad_(), "w": w.requires_grad_(), "hhat": hhat.requires_grad_(), "r": v}
    flags = FLAGS[case["flags"]]
    if case["form"] == "sep" and wx is not None:
        plan = Plan(wy=wy, wx=wx, h=h, flags=flags)
    else:
        plan = Plan(_dense(wy, wx), h=h, flags=flags)
    if case["tuned"]:
        plan.autotune(case["batch"])
    return {"case": case, "plan": plan, "u": u, "v": v}


def run(state):
    case = state["case"]
    if case["kind"] == "mix":
        state["batch"].launch()
        return state["outs"]
    if case["kind"] == "train":
        y = convolution_product(state["u"], state["w"], state["hhat"])
        grads = torch.autograd.grad(y, (state["u"], state["w"], state["hhat"]), state["r"])
        return (y.detach(),) + grads
    plan = state["plan"]
    out = []
    if case["dir"] in ("fwd", "both"):
        out.append(plan.apply(state["u"]))
    if case["dir"] in ("adj", "both"):
        out.append(plan.apply_adjoint(state["v"]))
    return tuple(out)


# ------------------------------------------------------------------ what a pass needs

def _apply_work(shape, m, grid, form="dense", lowp=False):
    """(bytes of the operator, bytes and flops of one right-hand side's product).  Operator:
    windows on their supports (or their factors) and half spectra.  Flops: 5 n log2 n a complex
    transform of n samples, half of that a real one, on the window's rows (2D; one set a column
    factor where the windows are products) and the half spectrum's columns, with one inverse for
    the sum; 8 a spectral product and accumulation; one multiply a window sample."""
    n = math.prod(shape)
    half = n // shape[-1] * (shape[-1] // 2 + 1)
    spectra = m * half * (4 if lowp else 8)
    if len(shape) == 1:
        win = min(2 * n // m, n) * m
        flops = (m + 1) * 2.5 * n * math.log2(n) + 8 * m * half + win
        return win * (2 if lowp else 4) + spectra, 8 * n, flops
    ny, nx = shape
    nr, nc = min(2 * ny // grid[0], ny), min(2 * nx // grid[1], nx)
    rows = grid[1] * ny if form == "sep" else m * nr
    win = rows * nc
    flops = ((rows + ny) * 2.5 * nx * math.log2(nx) + (m + 1) * (nx // 2 + 1) * 5 * ny * math.log2(ny)
             + 8 * m * half + win)
    return (4 * m * (ny + nx) if form == "sep" else win * (2 if lowp else 4)) + spectra, 8 * n, flops


def work(case):
    """Bytes and flops of one pass: every input and operator array read once, every output written once."""
    if case["kind"] == "mix":
        rng = random.Random(1604_04374 + 7 * case["batch"])
        nbytes, flops, seen = 0, 0.0, set()
        for _ in range(case["batch"]):
            s, k, _ = rng.randrange(len(MIX_SHAPES)), rng.randrange(len(MIX_M)), rng.randrange(2)
            m = MIX_M[k]
            gy = 1 << math.ceil(math.log2(m) / 2)
            op, io, f = _apply_work(MIX_SHAPES[s], m, (gy, m // gy), "sep")
            nbytes += io + (0 if (s, k) in seen else op)
            flops += f
            seen.add((s, k))
        return {"bytes": int(nbytes), "flops": int(flops)}
    shape = _shape(case)
    grid = _grid(case) if len(shape) == 2 else None
    op, io, f = _apply_work(shape, case["m"], grid, case["form"], case["flags"] == "lowp")
    if case["kind"] == "train":
        # u, r read, y, du written; w and hhat read, their (dense) gradients written.  The forward
        # product, the adjoint one, and for dw and dhhat one transform each a term
        n = math.prod(shape)
        half = n // shape[-1] * (shape[-1] // 2 + 1)
        return {"bytes": case["batch"] * 2 * io + 2 * case["m"] * (4 * n + 8 * half),
                "flops": int(4 * case["batch"] * f)}
    k = (2 if case["dir"] == "both" else 1) * case["batch"]
    return {"bytes": int(op + k * io), "flops": int(k * f)}


# ------------------------------------------------------------------ 64-bit values

def _exact_apply(u, wy, wx, h, adjoint, product=False):
    """sum_k h_k * (w_k . u), or sum_k w_k . (conj-reversed h_k * u); the product form swaps them."""
    dims = tuple(range(1, u.dim()))
    size = u.shape[1:]
    u = u.double()
    acc = None
    windowed_out = adjoint != product
    spec = torch.fft.rfftn(u, dim=dims) if windowed_out else None
    for k in range(h.shape[0]):
        # the window the framework is given: a product of two float32 factors is rounded to float32
        w = (wy[k] if wx is None else wy[k][:, None] * wx[k][None, :]).double()
        hh = torch.fft.rfftn(h[k].double())
        if adjoint:
            hh = hh.conj()
        if windowed_out:
            t = w * torch.fft.irfftn(spec * hh, s=size, dim=dims)
        else:
            t = torch.fft.rfftn(w * u, dim=dims) * hh
        acc = t if acc is None else acc.add_(t)
    return acc if windowed_out else torch.fft.irfftn(acc, s=size, dim=dims)


def exact(case, seed):
    if case["kind"] == "mix":
        picks, ops, ins = _inputs(case, seed)
        outs, of_task = _mix_outputs(picks, ins, torch.float64)
        for (s, k, adj), x, y in zip(picks, ins, of_task):
            y.copy_(_exact_apply(x, *ops[(s, k)], adj))
        return outs
    (wy, wx, h), u, v = _inputs(case, seed)
    if case["kind"] == "train":
        dims = tuple(range(1, u.dim()))
        size = u.shape[1:]
        n = math.prod(size)
        hhat = torch.fft.rfftn(h, dim=dims).to(torch.complex128)   # the values the call is given
        ud = u.double()
        rs = torch.fft.rfftn(v.double(), dim=dims)
        c = torch.full((size[-1] // 2 + 1,), 2.0, dtype=torch.float64, device=u.device)
        c[0] = c[-1] = 1.0
        ys = None
        du = torch.zeros_like(ud)
        dw = torch.empty((h.shape[0],) + tuple(size), dtype=torch.float64, device=u.device)
        dh = torch.empty_like(hhat)
        for k in range(h.shape[0]):
            w = (wy[k] if wx is None else wy[k][:, None] * wx[k][None, :]).double()
            x = torch.fft.rfftn(w * ud, dim=dims)
            ys = x * hhat[k] if ys is None else ys.add_(x * hhat[k])
            q = torch.fft.irfftn(rs * hhat[k].conj(), s=size, dim=dims)
            du += w * q
            dw[k] = (ud * q).sum(0)
            dh[k] = (rs * x.conj()).sum(0) * (c / n)
        return torch.fft.irfftn(ys, s=size, dim=dims), du, dw, dh
    out = []
    product = case["flags"] == "product"
    if case["dir"] in ("fwd", "both"):
        out.append(_exact_apply(u, wy, wx, h, False, product))
    if case["dir"] in ("adj", "both"):
        out.append(_exact_apply(v, wy, wx, h, True, product))
    return tuple(out)
