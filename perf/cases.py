"""The workloads that the library's speed is judged by.

Each case is one call that a program makes through the public entry points: a single evaluation of
S_ph (device or host buffers), a batch of snapshots, the direct sums, the judged surrogate, and the
surrogate's network forward and backward.  Inputs are synthetic streamers (a Gaussian head, a
channel behind it, |E| of a charged head in a background field) drawn from the seed on the GPU.

``exact`` restates each result in FP64 with plain torch: S_ph is a discrete convolution of the
selected sources with G on a uniform grid, summed by FFT; the network is 27 shifted products per
layer, differentiated by autograd.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2112_10059_gb300 as sph
from paper_2112_10059_gb300 import surrogate as sur

I0 = 1.0e20                       # emission peak, cm^-3 s^-1
CHI_MIN, CHI_MAX = 0.035, 2.0     # cm^-1 Torr^-1
FACTOR = 4                        # fine cells per coarse cell of the surrogate, along one axis
LR_EPS, LR_LAMBDA = 1e-4, 0.01    # the network's loss: see include/sph_nn.h

# ------------------------------------------------------------------------------------- the cases


def _eval(name, nx, ny, nz, h, p, i_frac, targets, leaf=64, m2l="bf16x3", radius=0.02, e_frac=0.1, kind="eval"):
    return dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, h=h, p=p, i_frac=i_frac, targets=targets, e_frac=e_frac,
                leaf=leaf, m2l=m2l, radius=radius)


def listed():
    return [
        # the smallest evaluation: a 2 mm cube of 24^3 cells, every cell a source and a target
        # (the plain-quadrature configuration through the FMM); latency and launches count
        _eval("plain_24", 24, 24, 24, 0.2 / 24, 760.0, 0.0, "all"),
        # a demand-oriented evaluation on a ragged box: random target mask, small leaves, low
        # pressure (long range), FP32 translations
        _eval("ragged_mask_f32", 90, 61, 117, 1.0 / 117, 76.0, 1e-3, "mask", leaf=32, m2l="f32"),
        # the headline: one time step's evaluation of a 256^3 adaptive streamer
        _eval("adaptive_256", 256, 256, 256, 1.0 / 256, 760.0, 1e-4, "emag"),
        # no adaptivity: every cell of 128^3 a source and a target; near field and dense M2L
        _eval("full_128", 128, 128, 128, 1.0 / 128, 760.0, 0.0, "all"),
        # a wide channel (radius 1 mm, threshold 1e-5): about a million sources on 192^3
        _eval("wide_192", 192, 192, 192, 1.0 / 192, 380.0, 1e-5, "emag", radius=0.1, e_frac=0.15),
        # eight independent snapshots in one call, grids 64^3 .. 256^3, three pressures
        dict(name="batch_8", kind="batch", count=8, n_lo=64, n_hi=256, shape_seed=1003, leaf=64, m2l="bf16x3"),
        # the same evaluation for a program whose fields live in host memory
        _eval("host_128", 128, 128, 128, 1.0 / 128, 760.0, 1e-4, "emag", kind="host"),
        # the FP64 direct sum of the plain-quadrature configuration (the in-library reference)
        _eval("direct_f64_24", 24, 24, 24, 0.2 / 24, 760.0, 0.0, "all", kind="direct_f64"),
        # the FP32 direct sum over a streamer's selected sources (what the FMM is compared with)
        _eval("direct_f32_160", 160, 160, 160, 1.0 / 160, 760.0, 1e-3, "emag", kind="direct_f32"),
        # the judged surrogate on a 256^3 fine grid (64^3 coarse), gate 1e-3, two samples a block
        dict(name="judged_64", kind="judged", edge=64, p=760.0, i_frac=1e-4, tol=1e-3, samples=2, leaf=64),
        # the network: inference and the gradient of one training batch, at the trainer's sizes
        dict(name="net_forward_64", kind="forward", edge=64, batch=4),
        dict(name="net_backward_64", kind="backward", edge=64, batch=4),
    ]


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def edges(lo, hi, most):
        n = log(lo, hi)
        while True:
            e = [max(lo, min(hi, int(round(n * rng.uniform(0.6, 1.0))))) for _ in range(3)]
            if e[0] * e[1] * e[2] <= most:
                return e
            n *= 0.95

    kind = rng.choice(["eval", "eval", "eval", "full", "host", "batch", "direct_f64", "direct_f32", "judged", "forward",
                       "forward", "backward", "backward"])
    p = rng.choice([76.0, 380.0, 760.0])
    if kind == "full":
        e = edges(16, 128, 128 ** 3)
        c = _eval("", *e, 1.0 / max(e) if max(e) > 48 else 0.2 / max(e), p, 0.0, "all", m2l=rng.choice(["bf16x3", "f32"]))
        if c["m2l"] == "f32" and max(e) > 96:
            c["m2l"] = "bf16x3"
    elif kind in ("eval", "host"):
        e = edges(32, 256 if kind == "eval" else 160, 1 << 24)
        c = _eval("", *e, 1.0 / max(e), p, log(1e-5, 1e-3), rng.choice(["emag", "emag", "mask", "all"]),
                  leaf=rng.choice([32, 64, 64, 128]), radius=log(0.015, 0.06), e_frac=rng.uniform(0.05, 0.2), kind=kind)
    elif kind == "batch":
        c = dict(kind="batch", count=rng.randrange(2, 9), n_lo=48, n_hi=rng.randrange(64, 225), shape_seed=rng.randrange(1 << 20),
                 leaf=64, m2l="bf16x3")
    elif kind == "direct_f64":
        e = edges(8, 26, 24 ** 3)
        c = _eval("", *e, 0.2 / max(e), p, 0.0, "all", kind=kind)
    elif kind == "direct_f32":
        e = edges(32, 160, 160 ** 3)
        c = _eval("", *e, 1.0 / max(e), p, log(1e-3, 1e-2), rng.choice(["emag", "mask"]), radius=0.02, kind=kind)
    elif kind == "judged":
        c = dict(kind="judged", edge=rng.choice([16, 32, 64]), p=p, i_frac=log(1e-5, 1e-3), tol=1e-3, samples=rng.randrange(1, 4), leaf=64)
    else:
        edge = rng.choice([8, 16, 32, 64])
        most = min(64, 4 * 64 ** 3 // edge ** 3)
        c = dict(kind=kind, edge=edge, batch=int(round(log(1, most))))
    c.pop("name", None)
    return c


# ------------------------------------------------------------------------------------- inputs


def _pO2(p):
    return p * 150.0 / 760.0


def _scale(p):
    return 0.06 * 30.0 / (p + 30.0)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _axes(nx, ny, nz, h):
    a = [(torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * h for n in (nx, ny, nz)]
    return a[0].view(1, 1, -1), a[1].view(1, -1, 1), a[2].view(-1, 1, 1)


def _streamer(nx, ny, nz, h, radius, r, cloud=False):
    """Emission (peak about I0) and |E| (kV/cm) of a streamer whose head position, channel length
    and head width come from the random stream ``r``; float32, x fastest."""
    X, Y, Z = _axes(nx, ny, nz, h)
    lx, ly, lz = nx * h, ny * h, nz * h
    hx, hy = lx * (0.5 + 0.1 * (r.random() - 0.5)), ly * (0.5 + 0.1 * (r.random() - 0.5))
    length = lz * (0.45 + 0.1 * r.random())
    hz = 0.5 * (lz - length)
    sig = 0.015 * (0.95 + 0.1 * r.random()) * max(lx, ly, lz)
    rho2 = (X - hx) ** 2 + (Y - hy) ** 2
    r2 = rho2 + (Z - hz) ** 2
    q = torch.exp(-r2 / sig ** 2) + 1e-2 * torch.exp(-rho2 / radius ** 2) * ((Z >= hz) & (Z <= hz + length))
    if cloud:
        q = q + 1e-3 * torch.exp(-(rho2 + (Z - 0.5 * hz) ** 2) / 0.1 ** 2)
    d = torch.sqrt(r2).clamp(min=1e-12)
    ball = torch.where(d < sig, 150.0 * d / sig, 150.0 * (sig / d) ** 2) / d
    e = torch.sqrt((ball * (X - hx)) ** 2 + (ball * (Y - hy)) ** 2 + (ball * (Z - hz) - 30.0) ** 2)
    return (q * I0).float().reshape(-1).contiguous(), e.float().reshape(-1).contiguous()


def _fields(case, seed):
    """q, |E| or None, mask or None of an evaluation."""
    nx, ny, nz, h = case["nx"], case["ny"], case["nz"], case["h"]
    r = random.Random(seed)
    if case["i_frac"] == 0.0:          # every cell a source: a Gaussian with noise
        X, Y, Z = _axes(nx, ny, nz, h)
        c = [0.5 * n * h * (0.95 + 0.1 * r.random()) for n in (nx, ny, nz)]
        q = torch.exp(-((X - c[0]) ** 2 + (Y - c[1]) ** 2 + (Z - c[2]) ** 2) / (0.1 * nz * h) ** 2)
        q = q + 1e-3 * torch.rand(q.shape, dtype=torch.float64, device="cuda", generator=_gen(seed))
        q, e = (q * I0).float().reshape(-1).contiguous(), None
    else:
        q, e = _streamer(nx, ny, nz, h, case["radius"], r)
    if case["targets"] == "emag":
        return q, e, None
    if case["targets"] == "mask":
        m = torch.rand(nx * ny * nz, device="cuda", generator=_gen(seed + 1)) < 0.3
        return q, None, m.to(torch.uint8)
    return q, None, None


def _snapshots(case, seed):
    """Per snapshot of a batch: n, pressure, thresholds (from the case) and fields (from the seed)."""
    s = random.Random(case["shape_seed"])
    for k in range(case["count"]):
        n = int(round(math.exp(s.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        if k == 0:
            n = case["n_hi"]
        p, i_frac, e_frac = s.choice([76.0, 380.0, 760.0]), 10.0 ** s.uniform(-5.0, -3.0), s.uniform(0.05, 0.2)
        yield dict(nx=n, ny=n, nz=n, h=1.0 / n, p=p, i_frac=i_frac, targets="emag", e_frac=e_frac, radius=0.02), 64 * seed + k


# layer name, input and output channels, level; the flat parameter order of include/sph_nn.h
LAYERS = [("c00", 16, 16, 0), ("c01", 16, 16, 0), ("c10", 16, 32, 1), ("c11", 32, 32, 1), ("c20", 32, 32, 2), ("c21", 32, 32, 2),
          ("c30", 32, 32, 3), ("c31", 32, 32, 3), ("c22", 32, 32, 2), ("c12", 32, 32, 1), ("c02", 32, 16, 0), ("c03", 16, 16, 0)]


def _params(seed):
    """He-normal weights with small biases, flat float32, as a trained network's are sized."""
    g = np.random.default_rng(seed)
    parts = []
    for name, ci, co, _ in LAYERS:
        w = g.standard_normal((co, 27, ci)) * math.sqrt(2.0 / (27 * ci))
        if name == "c00":
            w[:, :, 4:] = 0.0      # only four input channels carry fields
        parts += [w.ravel(), 0.02 * g.standard_normal(co)]
    parts += [0.05 * g.standard_normal(32), np.array([0.0, -4.6])]
    return np.concatenate(parts).astype(np.float32)


def _net_batch(edge, batch, seed):
    """Network inputs as sph_nn_make_inputs lays them out (four channels of normalised fields) and
    log-ratio targets."""
    n, g, r = edge, _gen(seed), random.Random(seed)
    x = torch.zeros((batch, n ** 3, 16), dtype=torch.bfloat16, device="cuda")
    for b in range(batch):
        q, e = _streamer(n, n, n, 1.5 / n, 0.03, r, cloud=True)
        q = q / q.max()
        x[b, :, 0] = (torch.log10(q + 1e-8) / 8 + 1).clamp(min=0)
        x[b, :, 1] = e / e.max()
        s = q.view(n, n, n).double()
        for ax in range(3):        # a wide blur stands for the coarse estimate
            k = torch.exp(-((torch.arange(n, device="cuda").double().view(-1, 1) - torch.arange(n, device="cuda").view(1, -1)).abs()) * 8.0 / n)
            s = torch.movedim(torch.tensordot(k, s, dims=([1], [ax])), 0, ax)
        s = (s / s.max()).reshape(-1).float()
        x[b, :, 2] = (torch.log(s + 1e-12) / 27.631021 + 1).clamp(min=0)
        x[b, :, 3] = (torch.log10(1.5 * q + 1e-8) / 8 + 1).clamp(min=0, max=1)
    t = 0.05 * torch.randn(batch * n ** 3, device="cuda", generator=g) + 0.1 * x[:, :, 0].float().reshape(-1)
    return x.reshape(-1).contiguous(), t.contiguous()


# ------------------------------------------------------------------------------------- the calls


def _criteria(ctx, case):
    sph.set_criteria(ctx, case["i_frac"], case.get("e_frac", 0.0), 0.0, 1, case["leaf"],
                     sph.M2L_F32 if case.get("m2l") == "f32" else sph.M2L_BF16X3)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind, case=case)
    if kind in ("forward", "backward"):
        s["net"] = sur.Net(edge=case["edge"], max_batch=case["batch"])
        s["net"].set_params(_params(seed))
        s["x"], s["t"] = _net_batch(case["edge"], case["batch"], seed)
        s["y"] = torch.empty(case["batch"] * case["edge"] ** 3 * 2, device="cuda")
        return s
    ctx = s["ctx"] = sph.Context(0)
    if kind == "batch":
        _criteria(ctx, dict(case, i_frac=0.0))
        s["problems"] = []
        for c, sd in _snapshots(case, seed):
            q, e, _ = _fields(c, sd)
            s["problems"].append(sph.BatchProblem(c["nx"], c["ny"], c["nz"], c["h"], _pO2(c["p"]), q, _scale(c["p"]), emag=e,
                                                  i_frac=c["i_frac"], e_frac=c["e_frac"]))
        return s
    if kind == "judged":
        n = case["edge"] * FACTOR
        q, e = _streamer(n, n, n, 1.5 / n, 0.03, random.Random(seed), cloud=True)
        sph.set_grid(ctx, n, n, n, 1.5 / n, _pO2(case["p"]))
        sph.set_sources(ctx, q, _scale(case["p"]))
        sph.set_targets(ctx, emag=e)
        _criteria(ctx, case)
        s["net"] = sur.Net(edge=case["edge"], max_batch=1)
        s["net"].set_params(_params(seed))
        s["out"] = torch.empty(case["edge"] ** 3, device="cuda")
        return s
    q, e, m = _fields(case, seed)
    n = q.numel()
    sph.set_grid(ctx, case["nx"], case["ny"], case["nz"], case["h"], _pO2(case["p"]))
    sph.set_sources(ctx, q, _scale(case["p"]))
    sph.set_targets(ctx, emag=e, mask=m)
    _criteria(ctx, case)
    if kind == "host":
        s["q"], s["e"], s["m"] = (None if a is None else a.cpu().numpy() for a in (q, e, m))
        s["out"] = np.empty(n, np.float32)
    else:
        s["out"] = torch.empty(n, dtype=torch.float64 if kind == "direct_f64" else torch.float32, device="cuda")
    return s


def run(s):
    kind = s["kind"]
    if kind == "eval":
        return sph.eval_sph(s["ctx"], s["out"])[0]
    if kind == "host":
        return sph.eval_sph_host(s["ctx"], s["q"], s["e"], s["m"], s["out"])[0]
    if kind == "batch":
        return sph.eval_sph_batch(s["ctx"], s["problems"])[0]
    if kind in ("direct_f64", "direct_f32"):
        return sph.eval_direct(s["ctx"], fp64=kind == "direct_f64", out=s["out"])
    if kind == "judged":
        c = s["case"]
        return sur.evaluate(s["ctx"], s["net"], FACTOR, tol=c["tol"], samples=c["samples"], seed=7, out=s["out"])[0]
    if kind == "forward":
        return s["net"].forward(s["x"], s["case"]["batch"], s["y"])
    loss = s["net"].backward(s["x"], s["t"], s["case"]["batch"])
    return {"loss": loss, "grads": s["net"].get_grads()}


def _cells(case):
    """Cells, and a mean count of sources (a streamer's channel and head above the threshold)."""
    n = case["nx"] * case["ny"] * case["nz"]
    if case["i_frac"] == 0.0:
        return n, n
    rho2 = case["radius"] ** 2 * math.log(max(1e-2 / case["i_frac"], 1.0))
    return n, math.pi * rho2 * 0.5 * case["nz"] * case["h"] / case["h"] ** 3


def work(case):
    kind = case["kind"]
    if kind in ("forward", "backward"):
        v = case["batch"] * case["edge"] ** 3
        conv = sum(2 * 27 * ci * co * case["batch"] * (case["edge"] >> lv) ** 3 for _, ci, co, lv in LAYERS)
        npar = sum(27 * ci * co + co for _, ci, co, _ in LAYERS) + 34
        if kind == "forward":
            return {"bytes": v * (32 + 8) + 4 * npar, "flops": conv}
        return {"bytes": v * (32 + 4) + 8 * npar, "flops": 3 * conv - 2 * 27 * 256 * v}
    if kind == "judged":   # the fine fields once, the coarse result
        return {"bytes": 8 * (FACTOR * case["edge"]) ** 3 + 4 * case["edge"] ** 3, "flops": 0}
    if kind == "batch":
        return {"bytes": sum(12 * c["nx"] ** 3 for c, _ in _snapshots(case, 0)), "flops": 0}
    n, ns = _cells(case)
    b = n * (4 + {"emag": 4, "mask": 1, "all": 0}[case["targets"]] + (8 if kind == "direct_f64" else 4))
    if kind in ("direct_f64", "direct_f32"):
        nt = 0.3 * n if case["targets"] == "mask" else n
        return {"bytes": b, "flops": 12 * nt * ns}
    # every cell a source: the 27 leaves of 4^3 cells around a target, 12 operations a pair
    return {"bytes": b, "flops": 12 * 27 * 64 * n if ns == n else 0}


# ------------------------------------------------------------------------------------- in 64 bits


def _s_ph(q, nx, ny, nz, h, p, i_frac, targets):
    """S_ph (float64) at the cells where ``targets`` is set: sources q >= i_frac max q convolved
    with G, plus the integral of G over a ball of one cell's volume at the cell itself."""
    al, be, L = CHI_MIN * _pO2(p), CHI_MAX * _pO2(p), math.log(CHI_MAX / CHI_MIN)
    q = q.double().view(nz, ny, nx)
    I = torch.where(q >= i_frac * q.max(), q, torch.zeros_like(q)) * _scale(p)
    m = [2 * k for k in (nz, ny, nx)]

    def off(k):
        a = torch.arange(2 * k, device="cuda", dtype=torch.float64)
        return torch.where(a < k, a, a - 2 * k) * h

    R = torch.sqrt(off(nz).view(-1, 1, 1) ** 2 + off(ny).view(1, -1, 1) ** 2 + off(nx).view(1, 1, -1) ** 2)
    R[0, 0, 0] = 1.0
    G = torch.exp(-al * R) * -torch.expm1((al - be) * R) / (4 * math.pi * L * R ** 3) * h ** 3
    # 1 - (E1(al a) - E1(be a)) / L with E1(al a) - E1(be a) = int exp(-a e^u) du, u from ln al to ln be
    a = h * (3 / (4 * math.pi)) ** (1 / 3)
    z, w = np.polynomial.legendre.leggauss(96)
    u = 0.5 * L * (z + 1) + math.log(al)
    G[0, 0, 0] = 1 - 0.5 * float(np.sum(w * np.exp(-a * np.exp(u))))
    Gf = torch.fft.rfftn(G)
    del G, R
    S = torch.fft.irfftn(Gf * torch.fft.rfftn(I, s=m), s=m)[:nz, :ny, :nx]
    return torch.where(targets.view(nz, ny, nx), S, torch.zeros_like(S)).reshape(-1)


def _s_ph_of(case, q, e, m):
    if e is not None:
        t = e.double() >= case["e_frac"] * e.double().max()
    else:
        t = m != 0 if m is not None else torch.ones_like(q, dtype=torch.bool)
    return _s_ph(q, case["nx"], case["ny"], case["nz"], case["h"], case["p"], case["i_frac"], t)


def _net64(flat, x, batch, n):
    """The network in float64: flat parameters and x [batch, n^3, 16] to y [batch, n^3, 2]."""
    P, at = {}, 0
    for name, ci, co, _ in LAYERS:
        P[name] = flat[at:at + co * 27 * ci].view(co, 27, ci), flat[at + co * 27 * ci:at + co * 27 * ci + co]
        at += co * 27 * ci + co

    def conv(name, v):            # v [batch, z, y, x, c]
        w, b = P[name]
        d = v.shape[1]
        pad = torch.nn.functional.pad(v, (0, 0, 1, 1, 1, 1, 1, 1))
        out = b
        for tap in range(27):
            k, j, i = tap // 9, tap // 3 % 3, tap % 3
            out = out + pad[:, k:k + d, j:j + d, i:i + d] @ w[:, tap].T
        return torch.relu(out)

    def pool(v):
        b, d, c = v.shape[0], v.shape[1] // 2, v.shape[4]
        return v.view(b, d, 2, d, 2, d, 2, c).mean(dim=(2, 4, 6))

    def up(v):
        for ax in (1, 2, 3):
            v = v.repeat_interleave(2, dim=ax)
        return v

    s0 = conv("c01", conv("c00", x.view(batch, n, n, n, 16)))
    s1 = conv("c11", conv("c10", pool(s0)))
    s2 = conv("c21", conv("c20", pool(s1)))
    d2 = conv("c22", up(conv("c31", conv("c30", pool(s2)))) + s2)
    d1 = conv("c12", up(d2) + s1)
    f = conv("c03", conv("c02", up(d1)) + s0)
    return f @ flat[at:at + 32].view(2, 16).T + flat[at + 32:]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("forward", "backward"):
        n, b = case["edge"], case["batch"]
        x, t = _net_batch(n, b, seed)
        flat = torch.from_numpy(_params(seed)).cuda().double().requires_grad_(kind == "backward")
        if kind == "forward":
            with torch.no_grad():
                return torch.cat([_net64(flat, x[i * n ** 3 * 16:(i + 1) * n ** 3 * 16].double(), 1, n).reshape(-1) for i in range(b)])
        loss = 0.0
        for i in range(b):         # one sample at a time: the graph of one fits easily
            y = _net64(flat, x[i * n ** 3 * 16:(i + 1) * n ** 3 * 16].double(), 1, n).reshape(-1, 2)
            d = y[:, 0] - t[i * n ** 3:(i + 1) * n ** 3].double()
            part = (d ** 2 + LR_LAMBDA * (y[:, 1] - torch.log(d.abs() + LR_EPS).detach()) ** 2).sum() / (b * n ** 3)
            part.backward()
            loss += float(part.detach())
        return {"loss": loss, "grads": flat.grad}
    if kind == "batch":
        return [_s_ph_of(c, *_fields(c, sd)) for c, sd in _snapshots(case, seed)]
    if kind == "judged":           # every block that passes the gate is within it of this
        n, m = case["edge"] * FACTOR, case["edge"]
        q, _ = _streamer(n, n, n, 1.5 / n, 0.03, random.Random(seed), cloud=True)
        S = _s_ph(q, n, n, n, 1.5 / n, case["p"], case["i_frac"], torch.ones_like(q, dtype=torch.bool))
        return S.view(m, FACTOR, m, FACTOR, m, FACTOR).mean(dim=(1, 3, 5)).reshape(-1)
    return _s_ph_of(case, *_fields(case, seed))
